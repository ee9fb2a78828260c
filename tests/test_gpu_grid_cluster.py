"""The grid build by a cluster of CTAs and its cull of pills that can touch no
other group, at their edges: slices and warps that are not full, one group or
none meeting, the largest number of groups that is culled and one more, pills of
very different sizes, scenes far from the origin."""
import numpy as np
import pytest

import oracle
from paper_1906_05260_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _scene(seed, rods, verts, spread, groups=None, seg=0.01, far=0.0, thick=1.0):
    """Straight rods of `verts` vertices in a box, radii between 0.003 and 0.003 thick."""
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(rods, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    pos = rng.uniform(-spread, spread, (rods, 1, 3)) + far + seg * np.arange(verts)[None, :, None] * d[:, None, :]
    nv = rods * verts
    cs = np.full(rods, 1e-7)
    none = np.zeros(0, np.int32)
    group = np.arange(rods) if groups is None else rng.integers(0, groups, rods)
    return S.Scene(
        name="rods", rod_offsets=(np.arange(rods + 1) * verts).astype(np.int32), rest_pos=pos.reshape(nv, 3),
        rest_quat=np.repeat(S.quat_from_z(d), verts - 1, axis=0),
        radius=np.repeat(0.003 * np.exp(rng.uniform(0.0, np.log(thick), rods)), verts), density=np.full(rods, 1000.0),
        c_stretch=cs, c_bend=cs, c_volume=cs, group=(7 * group - 1000).astype(np.int32), gravity=S.GRAVITY.copy(),
        pin_vertex=none, pin_bone=none, pin_offset=np.zeros((0, 3)), bones=None, planes=np.zeros((0, 4)),
        contact_compliance=1e-9, contacts=True, volume=True, dt=1.0 / 60.0, substeps=1, iterations=1, frames=1)


@pytest.mark.parametrize("kw", [
    dict(seed=0, rods=1, verts=2, spread=0.01), dict(seed=1, rods=2, verts=2, spread=0.002),
    dict(seed=2, rods=33, verts=2, spread=0.03), dict(seed=3, rods=64, verts=9, spread=0.05, groups=1),
    dict(seed=4, rods=40, verts=17, spread=0.1, thick=8.0), dict(seed=5, rods=40, verts=17, spread=10.0),
    dict(seed=6, rods=512, verts=3, spread=0.15), dict(seed=7, rods=513, verts=3, spread=0.15),
    dict(seed=8, rods=700, verts=12, spread=0.3, groups=25, thick=9.0), dict(seed=9, rods=300, verts=20, spread=0.2, far=50.0),
    dict(seed=10, rods=1100, verts=16, spread=0.4, thick=3.0),
    dict(seed=11, rods=512, verts=81, spread=0.5), dict(seed=12, rods=513, verts=81, spread=0.5),  # 40,960 pills, and more
], ids=lambda k: "-".join(f"{a}{b}" for a, b in k.items() if a != "seed"))
def test_scene_pairs_match_brute_force(kw):
    from paper_1906_05260_gb300 import viper as V
    sc = _scene(**kw)
    alone, mixed, other = V.Scene(sc), V.Scene(sc), V.Scene(_scene(99, 90, 5, 0.1))
    alone.frame()
    batch = V.Batch()
    batch.step([other, mixed], [None, None], None, sc.dt, 1, 1)
    batch.synchronize()
    for g in (alone, mixed):  # the one-scene graph and the multi-scene step
        x4, rb = g.predicted()
        ref = oracle.broadphase_f32(sc.rod_offsets, sc.group, x4, rb, brute=True)
        np.testing.assert_array_equal(g.pairs(), ref)
    print(len(ref), "pairs")
