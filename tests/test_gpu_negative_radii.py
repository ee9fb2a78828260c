"""Pills squeezed past zero (negative bounding radii, some larger in size than every
positive one) in scenes, on each path of the broadphase, and a multi-scene call in
which one scene is past the cluster's grid and the other is not."""
import numpy as np
import pytest

import oracle
from test_gpu_grid_cluster import _scene

pytestmark = pytest.mark.gpu


def _squeeze(g, sc, seed):
    """Every tenth rod's radii to -0.02 .. -0.06 (a pill's half length is 0.005)."""
    x4 = g.get_state()["x4"].reshape(sc.n_rods, -1, 4)
    rng = np.random.default_rng(seed)
    x4[::10, :, 3] = -rng.uniform(0.02, 0.06, x4[::10, :, 3].shape)
    g.set_state(x4=x4.reshape(-1, 4))


def _check_pairs(g, sc):
    x4, rb = g.predicted()
    ref = oracle.broadphase_f32(sc.rod_offsets, sc.group, x4, rb, brute=True)
    assert len(ref) > 100
    np.testing.assert_array_equal(g.pairs(), ref)


# the cluster's grid with the cull and without it, the multi-kernel path, past the cluster's grid
@pytest.mark.parametrize("kw", [
    dict(seed=0, rods=120, verts=12, spread=0.15), dict(seed=1, rods=700, verts=3, spread=0.2),
    dict(seed=2, rods=700, verts=31, spread=0.5), dict(seed=3, rods=513, verts=82, spread=0.6),
], ids=lambda k: f"{k['rods']}x{k['verts']}")
@pytest.mark.parametrize("iterations", [0, 1])
def test_pairs_of_squeezed_pills(kw, iterations):
    from paper_1906_05260_gb300 import viper as V
    sc = _scene(**kw)
    for path in ("alone", "batch", "frame"):
        g = V.Scene(sc, solver=V.SOLVER_FRAME if path == "frame" else V.SOLVER_BATCHED, max_pairs=200 * sc.ns)
        _squeeze(g, sc, kw["seed"])
        if path == "batch":
            batch = V.Batch()
            batch.step([g], [None], None, sc.dt, 1, iterations)
            batch.synchronize()
        else:
            g.step(substeps=1, iterations=iterations)
        _check_pairs(g, sc)


def test_large_and_small_scene_in_one_call():
    from paper_1906_05260_gb300 import viper as V
    scs = [_scene(4, 513, 82, 0.6), _scene(5, 90, 9, 0.1), _scene(6, 600, 4, 0.2)]
    assert scs[0].ns > 40_960 > scs[1].ns
    mixed, alone = [V.Scene(sc) for sc in scs], [V.Scene(sc) for sc in scs]
    batch = V.Batch()
    for _ in range(2):
        batch.step(mixed, [None] * 3, None, scs[0].dt, 3, 2)
        for g in alone:
            g.step(substeps=3, iterations=2)
    batch.synchronize()
    for a, b, sc in zip(mixed, alone, scs):
        assert a.sync() == 0 and b.sync() == 0
        _check_pairs(a, sc)
        sa, sb = a.get_state(), b.get_state()
        for k in sa:
            np.testing.assert_array_equal(sa[k], sb[k], err_msg=k)
