"""State set and get through every kind of array, and the one-scene graph of a
scene of more than 20,000 pills against the multi-scene step."""
import ctypes as C

import numpy as np
import pytest

from paper_1906_05260_gb300 import scenes as S

pytestmark = pytest.mark.gpu
KEYS = ("x4", "v4", "q4", "w4")


def _scene():
    from paper_1906_05260_gb300 import viper as V
    g = V.Scene(S.plain_small())
    for _ in range(3):
        g.frame()
    return V, g


def _call(V, name, g, arrays):
    rc = getattr(V.lib(), name)(g.handle, *[C.c_void_p(a.data_ptr() if a is not None else 0) for a in arrays])
    assert rc == 0, (name, rc)


@pytest.mark.parametrize("offset", [0, 1, 4], ids=["aligned", "four-bytes-off", "sixteen-bytes-off"])
@pytest.mark.parametrize("device", ["cuda", "cpu", "mixed"])
def test_state_round_trip(device, offset):
    import torch
    V, g = _scene()
    ref = g.get_state()
    n = [ref[k].size for k in KEYS]
    where = [("cuda" if (device == "cuda" or (device == "mixed" and k % 2)) else "cpu") for k in range(4)]
    buf = [torch.full((m + 8,), 7.0, device=w)[offset:offset + m] for m, w in zip(n, where)]
    _call(V, "viper_get_state", g, buf)
    for k, b in zip(KEYS, buf):
        np.testing.assert_array_equal(b.cpu().numpy(), ref[k].reshape(-1), err_msg=k)
    g.frame()
    _call(V, "viper_set_state", g, buf)
    back = g.get_state()
    # frames are normalised and radii divided by their rest radius on the way in
    for k, tol in zip(KEYS, (1e-7, 1e-7, 3e-7, 0.0)):
        np.testing.assert_allclose(back[k], ref[k], rtol=tol, atol=tol, err_msg=k)


def test_get_state_leaves_out_and_overlaps():
    import torch
    V, g = _scene()
    ref = g.get_state()
    one = torch.zeros(ref["v4"].size, device="cuda")
    _call(V, "viper_get_state", g, [None, one, None, None])
    np.testing.assert_array_equal(one.cpu().numpy(), ref["v4"].reshape(-1))
    _call(V, "viper_get_state", g, [None, one, None, one])  # the later array holds where they overlap
    m = ref["w4"].size
    np.testing.assert_array_equal(one[:m].cpu().numpy(), ref["w4"].reshape(-1))
    np.testing.assert_array_equal(one[m:].cpu().numpy(), ref["v4"].reshape(-1)[m:])


def test_large_scene_alone_equals_multi_scene_step():
    from paper_1906_05260_gb300 import viper as V
    sc = S.hair(n_rods=1500)
    assert sc.ns > 20_000
    a, b = V.Scene(sc), V.Scene(sc)
    batch = V.Batch()
    for _ in range(3):
        a.step()
        batch.step([b], [None], None, sc.dt, sc.substeps, sc.iterations)
    batch.synchronize()
    assert a.sync() == 0 and b.sync() == 0
    sa, sb = a.get_state(), b.get_state()
    for k in KEYS:
        np.testing.assert_array_equal(sa[k], sb[k], err_msg=k)
    np.testing.assert_array_equal(a.pairs(), b.pairs())
