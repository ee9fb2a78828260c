"""The pair search of large scenes at its edges: warps that are not full, rows
of hits that are flushed early, equal oversized radii, radii below zero."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _pills(seed, n, spread, long=0, length=0.02, negative=0):
    """n two-vertex rods in a cube; `long` of them ten times as long (all of one length), `negative` with scales below zero."""
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(n, 3))
    d *= length / np.linalg.norm(d, axis=1, keepdims=True)
    d[:long] *= 10.0
    a = rng.uniform(-spread, spread, (n, 3))
    x4 = np.ones((n, 2, 4), np.float32)
    x4[:, 0, :3], x4[:, 1, :3] = a, a + d
    if long:  # axis-aligned and of one scale: their bounding radii are equal to the bit
        x4[:long, 0, :3] = np.round(x4[:long, 0, :3] * 64) / 64
        x4[:long, 1, :3] = x4[:long, 0, :3] + np.array([0.25, 0, 0], np.float32)
    x4[long:long + negative, :, 3] = -0.5
    x4[long + negative:, :, 3] = rng.uniform(0.5, 1.5, (n - long - negative, 2))
    return ((2 * np.arange(n + 1)).astype(np.int32), np.arange(n, dtype=np.int32), x4.reshape(-1, 4),
            np.full(2 * n, 0.004, np.float32))


@pytest.mark.parametrize("kw", [
    dict(seed=0, n=1, spread=0.01), dict(seed=1, n=2, spread=0.005), dict(seed=2, n=31, spread=0.02),
    dict(seed=3, n=32, spread=0.02), dict(seed=4, n=33, spread=0.02), dict(seed=5, n=257, spread=0.05),
    dict(seed=6, n=700, spread=0.006),                    # everything overlaps: rows flushed again and again
    dict(seed=7, n=9000, spread=0.3, long=40),            # oversized pills of equal radius, on equal corners
    dict(seed=8, n=9000, spread=0.2, negative=300),       # squeezed past zero
    dict(seed=9, n=9000, spread=0.2, long=300, negative=700),  # more than the cut leaves out
], ids=lambda k: "-".join(f"{a}{b}" for a, b in k.items() if a != "seed"))
def test_pair_search_edges_match_brute_force(kw):
    import torch
    from paper_1906_05260_gb300 import viper as V
    off, group, x4, rbar = _pills(**kw)
    ref = oracle.broadphase_f32(off, group, x4, rbar, brute=True)
    t = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    got, total = V.broadphase(t(off), t(group), t(x4), t(rbar), max_pairs=len(ref) + 16)
    assert total == len(ref)
    np.testing.assert_array_equal(got, ref)
