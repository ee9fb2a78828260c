"""viper_sync and viper_get_state report their own scene's errors, not what an earlier
failed call has left behind; viper_sync launches nothing."""
import ctypes as C

import numpy as np
import pytest

from paper_1906_05260_gb300 import scenes as S

pytestmark = pytest.mark.gpu
KEYS = ("x4", "v4", "q4", "w4")


def _scenes(n):
    from paper_1906_05260_gb300 import viper as V
    out = [V.Scene(S.plain_small()) for _ in range(n)]
    for g in out:
        g.frame()
        assert g.sync() == 0
    return V, out


def _failed_sync(V, g):
    """A sync that fails on the host: its stream is being captured (nothing is launched)."""
    cu = C.CDLL("libcuda.so.1")
    stream, graph = C.c_void_p(g.stream.cuda_stream), C.c_void_p()
    assert cu.cuStreamBeginCapture_v2(stream, 1) == 0  # thread-local mode
    rc = g.sync()
    assert cu.cuStreamEndCapture(stream, C.byref(graph)) != 0 and not graph.value  # a sync ends the capture
    assert rc == V.ECUDA


@pytest.mark.parametrize("call", ["sync", "step", "get_state_host", "get_state_device"])
def test_an_earlier_failure_is_not_reported_again(call):
    import torch
    V, (g, other) = _scenes(2)
    ref = other.get_state()
    _failed_sync(V, g)
    if call == "sync":
        assert other.sync() == 0
    elif call == "step":
        assert other.step() == 0
    elif call == "get_state_host":
        s = other.get_state()
        assert s["rc"] == 0
        for k in KEYS:
            np.testing.assert_array_equal(s[k], ref[k], err_msg=k)
    else:
        buf = [torch.zeros(ref[k].shape, device="cuda") for k in KEYS]
        torch.cuda.synchronize()
        rc = V.lib().viper_get_state(other.handle, *[C.c_void_p(a.data_ptr()) for a in buf])
        assert rc == 0
        for k, a in zip(KEYS, buf):
            np.testing.assert_array_equal(a.cpu().numpy(), ref[k], err_msg=k)
    assert g.sync() == 0 and other.sync() == 0


def test_sync_launches_no_kernel():
    """So it does not need the scene's device to be the current one."""
    _, (g,) = _scenes(1)
    before = g.launch_count()
    assert g.sync() == 0
    assert g.launch_count() == before
