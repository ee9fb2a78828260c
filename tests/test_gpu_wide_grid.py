"""The pair search where the grid is far wider than the pills: pairs near tangency
across cell borders, with a stray pill 2 to 100 km away along each axis."""
import numpy as np
import pytest

import oracle
from paper_1906_05260_gb300 import scenes as S

pytestmark = pytest.mark.gpu
F = np.float32
HALF, THIN, THICK = F(2.0 ** -8), F(0.001), F(0.02)  # half length of a pill, radii


def _pills(n_pairs, rows, axis, far):
    """Vertices (n, 2, 3) and radii (n,) of 2 n_pairs + 2 pills.  Pairs along `axis` at
    cell borders (`rows` per border) near the origin: the second pill within half a unit
    in the last place of the border, as measured from the grid's corner, the first just
    less than the sum of the bounding radii before it; one pair in 32 is thick
    (oversized for the grid).  Two stray pills at -far (the corner) and far / 4 make the
    cells the grid's extent / 4096 wide."""
    radius = np.full(2 * n_pairs + 2, THIN, F)
    radius[0:-2:64] = radius[1:-2:64] = THICK
    bound = (HALF + radius).astype(np.float64)
    reach = bound[:-2:2] + bound[1:-2:2]
    rng = np.random.default_rng(0)
    corner, end = F(-far), F(0.25 * far)
    ext = F(end - corner)
    inv = F(1.0) / F(ext * F(1.0 / 4096.0))
    k = int(far * inv) - 1 - np.arange(n_pairs) // rows
    d = (k / np.float64(inv)).astype(F)  # to the smallest offset of cell k
    for _ in range(8):
        d = np.where(np.floor(d * inv) < k, np.nextafter(d, F(np.inf)), d)
    for _ in range(8):
        low = np.nextafter(d, F(0.0))
        d = np.where(np.floor(low * inv) >= k, low, d)
    b = (d + rng.uniform(-0.5, 0.5, n_pairs) * np.spacing(d) + np.float64(corner)).astype(F)
    a = (b - reach * (1.0 - 10.0 ** rng.uniform(-5.0, -3.0, n_pairs))).astype(F)
    c = np.zeros((2 * n_pairs + 2, 3), F)
    thick = radius[:-2:2] == THICK  # searched from the higher id: there the one before the border
    c[:-2:2, axis], c[1:-2:2, axis] = np.where(thick, b, a), np.where(thick, a, b)
    c[:-2, (axis + 1) % 3] = np.repeat(F(0.125) * (np.arange(n_pairs) % rows), 2)
    c[-2, axis], c[-1, axis] = corner, end
    x = np.repeat(c[:, None, :], 2, axis=1)  # along the third axis, where every centre is zero
    x[:, 0, (axis + 2) % 3], x[:, 1, (axis + 2) % 3] = -HALF, HALF
    return x, radius


def _scene(x, radius, axis):
    n = len(x)
    d = np.zeros((n, 3))
    d[:, (axis + 2) % 3] = 1.0
    cs, none = np.full(n, 1e-7), np.zeros(0, np.int32)
    return S.Scene(
        name="wide", rod_offsets=(2 * np.arange(n + 1)).astype(np.int32), rest_pos=x.reshape(-1, 3).astype(np.float64),
        rest_quat=S.quat_from_z(d), radius=np.repeat(radius, 2).astype(np.float64), density=np.full(n, 1000.0), c_stretch=cs,
        c_bend=cs, c_volume=cs, group=np.arange(n, dtype=np.int32), gravity=np.zeros(3), pin_vertex=none, pin_bone=none,
        pin_offset=np.zeros((0, 3)), bones=None, planes=np.zeros((0, 4)), contact_compliance=1e-9, contacts=True,
        volume=True, dt=1.0 / 60.0, substeps=1, iterations=1, frames=1)


def _reference(off, group, x4, rbar, n_pairs):
    ref = oracle.broadphase_f32(off, group, x4, rbar, brute=True)
    assert len(ref) > 0.5 * n_pairs  # most are within reach once their coordinates are rounded
    return ref


@pytest.mark.parametrize("far", [2e3, 1e4, 1e5])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_query_on_a_wide_grid(axis, far):
    import torch
    from paper_1906_05260_gb300 import viper as V
    n = 4000
    x, radius = _pills(n, 8, axis, far)
    x4 = np.concatenate([x.reshape(-1, 3), np.ones((2 * len(x), 1), F)], axis=1)
    off, group = (2 * np.arange(len(x) + 1)).astype(np.int32), np.arange(len(x), dtype=np.int32)
    rbar = np.repeat(radius, 2)
    ref = _reference(off, group, x4, rbar, n)
    t = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    got, total = V.broadphase(t(off), t(group), t(x4), t(rbar), max_pairs=len(ref) + 16)
    assert total == len(ref)
    np.testing.assert_array_equal(got, ref)


# the grid by a cluster of CTAs; the multi-kernel path of one scene; scenes past the cluster's grid
@pytest.mark.parametrize("n,rows", [(4000, 8), (10_100, 16), (20_500, 32)])
@pytest.mark.parametrize("axis,far", [(0, 2e3), (0, 1e4), (0, 1e5), (1, 1e4), (2, 1e4)])
def test_scene_pairs_on_a_wide_grid(n, rows, axis, far):
    from paper_1906_05260_gb300 import viper as V
    sc = _scene(*_pills(n, rows, axis, far), axis)
    alone, mixed = V.Scene(sc), V.Scene(sc)
    alone.frame()
    batch = V.Batch()
    batch.step([mixed], [None], None, sc.dt, 1, 1)
    batch.synchronize()
    ref = None
    for g in (alone, mixed):  # the one-scene graph and the multi-scene step
        x4, rb = g.predicted()
        ref = _reference(sc.rod_offsets, sc.group, x4, rb, n) if ref is None else ref
        np.testing.assert_array_equal(g.pairs(), ref)
