"""Performance cases of the VIPER rod solver: what a program has it compute.

Every case goes through the public interface (the binding in
paper_1906_05260_gb300/viper.py and the C ABI behind it) and covers one use:

  rods    independent rods without contacts, a clip of frames from a saved state
  rig     bone-driven muscles with contacts and a skinned surface, a clip
  bundle  muscles of bundled fibres (shape matching), contacts, a clip
  hair    contact-heavy strands in a box of half-planes, a clip
  scenes  one multi-scene frame of many skinned rigs (the serving step)
  skin    linear blend skinning of a large mesh
  query   the scene-free broadphase on device-resident state

A clip starts from a state the program keeps on the device (a checkpoint, a
take that is simulated again) and ends with the new state on the device.

listed() are the measured cases, draw() gives further ones of the same ranges,
prepare() builds what a program holds before the call, run() is one call,
work() its unavoidable bytes and operations, exact() its results in 64 bits.
"""
import ctypes as C
import dataclasses
import math

import numpy as np
import torch

from paper_1906_05260_gb300 import scenes as S
from paper_1906_05260_gb300 import viper as V

DT = float(np.float32(1.0 / 60.0))
PAIRS_PER_PILL = 64  # pair capacity of the strand scenes (peak use is about 36 per pill)


def listed():
    return [
        # the smallest simulation: 16 hanging rods of 32 vertices, every launch and copy counts
        {"name": "rods_small", "kind": "rods", "rods": 16, "nmin": 32, "nmax": 32, "solver": "graph",
         "substeps": 10, "iterations": 4, "surface": False, "frames": 2},
        # thousands of rods of uneven length (4 to 256 vertices): throughput of the rod solve
        {"name": "rods_ragged", "kind": "rods", "rods": 4096, "nmin": 4, "nmax": 256, "solver": "graph",
         "substeps": 20, "iterations": 8, "surface": False, "frames": 1},
        # an odd number of rods with the surface-bending term, on the persistent frame solver
        {"name": "rods_surface_frame", "kind": "rods", "rods": 1021, "nmin": 4, "nmax": 256, "solver": "frame",
         "substeps": 10, "iterations": 4, "surface": True, "frames": 1},
        # an animated character: 200 muscles between 20 bones, contacts, a 200k-vertex skin each frame
        {"name": "rig", "kind": "rig", "rods": 200, "mesh": 200_000, "frames": 2},
        # anatomical muscles: 96 bundles of 7 fibres with shape matching and contacts
        {"name": "bundles", "kind": "bundle", "muscles": 96, "fibers": 7, "verts": 16, "frames": 2},
        # a partial groom: 3,000 strands settled in their box (45,000 pills)
        {"name": "hair_mid", "kind": "hair", "rods": 3000, "verts": 16, "settled": True, "frames": 1},
        # the full groom in its first frames: contacts are searched for, few are active
        {"name": "hair_falling", "kind": "hair", "rods": 20_000, "verts": 16, "settled": False, "frames": 1},
        # the full groom piled up: contacts everywhere, the heaviest single scene
        {"name": "hair_settled", "kind": "hair", "rods": 20_000, "verts": 16, "settled": True, "frames": 1},
        # a serving step at its usual load: 6 rigs of different sizes with their meshes
        {"name": "scenes_6", "kind": "scenes", "scenes": 6, "rods_lo": 50, "rods_hi": 500, "mesh_lo": 10_000,
         "mesh_hi": 300_000},
        # a serving step at full load: 64 rigs
        {"name": "scenes_64", "kind": "scenes", "scenes": 64, "rods_lo": 50, "rods_hi": 500, "mesh_lo": 10_000,
         "mesh_hi": 300_000},
        # a film-resolution mesh skinned by a 200-rod rig
        {"name": "skin_8m", "kind": "skin", "rods": 200, "mesh": 8_000_000},
        # candidate pairs for rods whose state another program holds
        {"name": "query", "kind": "query", "rods": 20_000, "verts": 16},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rods", "rods", "rig", "bundle", "hair", "hair", "scenes", "skin", "query"])
    if kind == "rods":
        nmin = rng.choice([2, 4, 7, 16])
        sub, it = rng.choice([(10, 4), (20, 8), (7, 3)])
        return {"kind": kind, "rods": _log_int(rng, 16, 4096), "nmin": nmin,
                "nmax": nmin + _log_int(rng, 1, 257 - nmin) - 1, "solver": rng.choice(["graph", "frame"]),
                "substeps": sub, "iterations": it, "surface": rng.random() < 0.3, "frames": 1}
    if kind == "rig":
        return {"kind": kind, "rods": _log_int(rng, 24, 500), "mesh": _log_int(rng, 2000, 300_000),
                "frames": rng.choice([2, 4])}
    if kind == "bundle":
        return {"kind": kind, "muscles": _log_int(rng, 8, 128), "fibers": rng.randint(3, 7),
                "verts": rng.randint(8, 24), "frames": 2}
    if kind == "hair":
        return {"kind": kind, "rods": _log_int(rng, 400, 20_000), "verts": rng.randint(9, 16),
                "settled": rng.random() < 0.5, "frames": 1}
    if kind == "scenes":
        return {"kind": kind, "scenes": _log_int(rng, 2, 60), "rods_lo": _log_int(rng, 40, 100),
                "rods_hi": _log_int(rng, 250, 500), "mesh_lo": 10_000, "mesh_hi": _log_int(rng, 100_000, 300_000)}
    if kind == "skin":
        return {"kind": kind, "rods": _log_int(rng, 50, 500), "mesh": _log_int(rng, 100_000, 8_000_000)}
    return {"kind": kind, "rods": _log_int(rng, 400, 20_000), "verts": rng.randint(9, 16)}


# ---------------------------------------------------------------- inputs
def _rods_scene(case, seed):
    """Straight rods along +x pinned at vertex 0, of log-uniform length, bent by
    up to 45 degrees per segment at the start (rods of one length hang straight
    at first): the batching workload.  The lengths are the case's, all else the seed's."""
    rng = np.random.default_rng(seed)
    n, nmin, nmax, seg = case["rods"], case["nmin"], case["nmax"], 0.01
    count = np.exp(np.random.default_rng(n).uniform(math.log(nmin), math.log(nmax), n)) if nmax > nmin else np.full(n, nmin)
    count = np.clip(np.rint(count), nmin, nmax).astype(np.int64)
    off = np.concatenate([[0], np.cumsum(count)]).astype(np.int32)
    nv, side = int(off[-1]), int(math.ceil(math.sqrt(n)))
    rod = np.repeat(np.arange(n), count)
    loc = np.arange(nv) - off[rod]
    pos = np.stack([seg * loc, 0.1 * (rod // side), 0.1 * (rod % side)], axis=1)
    first = np.nonzero(loc < count[rod] - 1)[0]  # the first vertex of every segment
    straight = np.tile(S.quat_from_z(np.array([1.0, 0.0, 0.0])), (first.size, 1))
    cs, cb = np.exp(rng.uniform(math.log(1e-8), math.log(1e-5), (2, n)))
    sc = S.Scene(
        name="rods", rod_offsets=off, rest_pos=pos, rest_quat=straight, radius=rng.uniform(0.005, 0.02, n)[rod],
        density=np.full(n, 1000.0), c_stretch=cs, c_bend=cb, c_volume=cs.copy(), group=np.arange(n, dtype=np.int32),
        gravity=S.GRAVITY.copy(), pin_vertex=off[:-1], pin_bone=np.full(n, -1, np.int32),
        pin_offset=pos[off[:-1]], bones=None, planes=np.zeros((0, 4)), contact_compliance=1e-9, contacts=False,
        volume=True, dt=1.0 / 60.0, substeps=case["substeps"], iterations=case["iterations"], frames=300,
        surface_bending=case["surface"])
    if nmax == nmin:
        return sc
    phi = rng.uniform(0.0, 2.0 * math.pi, first.size)
    axis = np.stack([np.zeros_like(phi), np.cos(phi), np.sin(phi)], axis=1)
    quat = S.quat_mul(S.axis_angle_quat(axis * np.radians(rng.uniform(-45.0, 45.0, (first.size, 1)))), straight)
    step = np.zeros((nv, 3))
    step[first + 1] = seg * S.quat_rotate(quat, np.tile(np.array([0.0, 0.0, 1.0]), (first.size, 1)))
    run = np.cumsum(step, axis=0)
    return dataclasses.replace(sc, init_pos=pos[off[rod]] + run - run[off[rod]], init_quat=quat)


def _rig_scene(sc, seed):
    """A rig whose bones move, and whose rods are as thick and as stiff, as the seed says."""
    rng = np.random.default_rng(seed)
    n, bones = sc.n_rods, sc.bones
    cs, cb = np.exp(rng.uniform(math.log(1e-8), math.log(1e-5), (2, n)))
    if sc.bundle_offsets is not None:  # the fibres of a muscle are alike
        cs, cb = cs[sc.bundle_offsets[sc.group]], cb[sc.bundle_offsets[sc.group]]
    bones = dataclasses.replace(bones, amp=bones.amp * rng.uniform(0.7, 1.0, bones.amp.shape),
                                phase=rng.uniform(0.0, 2.0 * math.pi, bones.phase.shape))
    thick = rng.uniform(0.9, 1.1, sc.group.max() + 1)[np.repeat(sc.group, sc.rod_lengths())]
    return dataclasses.replace(sc, bones=bones, c_stretch=cs, c_bend=cb, c_volume=cs.copy(), radius=sc.radius * thick)


def _sphere_points(rng, n, radius):
    """n points spread evenly over a sphere (a jittered spiral, turned at random)."""
    k = np.arange(n) + 0.5
    z = 1.0 - 2.0 * k / n
    phi = math.pi * (1.0 + math.sqrt(5.0)) * k + rng.uniform(0.0, 2.0 * math.pi)
    rho = np.sqrt(1.0 - z * z)
    p = np.stack([rho * np.cos(phi), rho * np.sin(phi), z], axis=1)
    p += rng.normal(scale=0.15 * math.sqrt(4.0 * math.pi / n), size=p.shape)
    q = rng.normal(size=4)
    return radius * S.quat_rotate(q / np.linalg.norm(q), p / np.linalg.norm(p, axis=1, keepdims=True))


def _strands(case, seed):
    """Radial strands on a sphere in a box of six half-planes: the sizes and
    materials of the hair workload, the sphere and the box scaled so that any
    number of strands is as dense as 20,000 on a 0.2 m sphere.  Returns the
    scene and its state (positions, scales, velocities, frames, spins)."""
    rng = np.random.default_rng(seed)
    n, m = case["rods"], case["verts"]
    f = math.sqrt(n / 20_000.0)
    radius, seg, box = 0.002, 0.005, 0.3 * f
    roots = _sphere_points(rng, n, 0.2 * f)
    normals = roots / np.linalg.norm(roots, axis=1, keepdims=True)
    step = seg * np.arange(m)
    pos = (roots[:, None] + step[None, :, None] * normals[:, None]).reshape(-1, 3)
    box = max(box, float(np.abs(pos).max()) + 0.02)
    planes = np.array([[1, 0, 0, -box], [-1, 0, 0, -box], [0, 1, 0, -box], [0, -1, 0, -box],
                       [0, 0, 1, -box], [0, 0, -1, -box]], dtype=np.float64)
    quat = np.repeat(S.quat_from_z(normals), m - 1, axis=0)
    cs = np.full(n, 1e-8)
    none = np.zeros(0, np.int32)
    sc = S.Scene(
        name="strands", rod_offsets=(np.arange(n + 1) * m).astype(np.int32), rest_pos=pos, rest_quat=quat,
        radius=np.full(n * m, radius), density=np.full(n, 1000.0), c_stretch=cs,
        c_bend=np.exp(rng.uniform(math.log(1e-7), math.log(1e-5), n)), c_volume=cs.copy(),
        group=np.arange(n, dtype=np.int32), gravity=S.GRAVITY.copy(), pin_vertex=none, pin_bone=none,
        pin_offset=np.zeros((0, 3)), bones=None, planes=planes, contact_compliance=1e-9, contacts=True, volume=True,
        dt=1.0 / 60.0, substeps=10, iterations=4, frames=200)
    if case.get("settled"):
        state = _settled(rng, n, m, seg, radius, box)
    else:  # a few frames into the fall
        p = pos.reshape(n, m, 3) + rng.normal(scale=1e-4, size=(n, 1, 3))
        v = np.zeros_like(p)
        v[..., 1] = -0.8
        state = _state_of(p, np.full((n, m), radius), v)
    return sc, state


def _settled(rng, n, m, seg, radius, box):
    """Strands lying over each other on the floor of the box, as the hair
    workload's do around its frame 55: mostly level and bent, overlapping as
    deeply (about 35 candidate pairs a pill, a third of them touching), their
    radii squeezed by the contacts (a few to nothing), a few segments stretched."""
    depth = 0.0145 * (n / 20_000) * (0.3 / box) ** 2
    start = rng.uniform(-box, box, size=(n, 3))
    start[:, 1] = -box + depth * rng.gamma(1.5, size=n) / 1.5
    az = rng.uniform(0.0, 2.0 * math.pi, n)[:, None] + np.cumsum(rng.normal(scale=0.3, size=(n, m - 1)), axis=1)
    el = rng.normal(scale=0.06, size=(n, 1)) + rng.normal(scale=0.12, size=(n, m - 1))
    d = np.stack([np.cos(el) * np.cos(az), np.sin(el), np.cos(el) * np.sin(az)], axis=2)
    length = seg * np.exp(np.abs(rng.normal(scale=0.03, size=(n, m - 1))))
    length *= np.where(rng.random((n, m - 1)) < 0.015, rng.uniform(1.2, 2.0, (n, m - 1)), 1.0)
    p = np.concatenate([np.zeros((n, 1, 3)), np.cumsum(d * length[..., None], axis=1)], axis=1)
    p += (start - p.mean(axis=1))[:, None]
    p = np.where(np.abs(p) > box, 2.0 * np.sign(p) * box - p, p)  # folded back at the walls and the floor
    r = radius * np.clip(rng.normal(0.88, 0.075, size=(n, m)), 0.3, 1.0)
    r = np.where(rng.random((n, m)) < 0.015, radius * rng.uniform(-0.05, 0.3, (n, m)), r)
    v = rng.normal(scale=0.08, size=(n, 1, 3)) + rng.normal(scale=0.05, size=(n, m, 3))
    return _state_of(p, r, v, rng.normal(scale=80.0, size=(n * (m - 1), 1)))


def _state_of(p, r, v, twist=0.0):
    """State arrays of strands at positions p [n, m, 3] with radii r and
    velocities v; frames follow the segments, spins are those of the segments
    and `twist` about their axes."""
    n, m = r.shape
    e = np.diff(p, axis=1)
    l = np.maximum(np.linalg.norm(e, axis=2, keepdims=True), 1e-9)
    t = (e / l).reshape(-1, 3)
    w = np.cross(t, (np.diff(v, axis=1) / l).reshape(-1, 3)) + twist * t
    x4 = np.concatenate([p, r[..., None]], axis=2).reshape(-1, 4)
    v4 = np.concatenate([v, np.zeros((n, m, 1))], axis=2).reshape(-1, 4)
    w4 = np.concatenate([w, np.zeros((w.shape[0], 1))], axis=1)
    return [np.ascontiguousarray(a, np.float32) for a in (x4, v4, S.quat_from_z(t), w4)]


def _surface(sc, n, seed):
    """A mesh of n points on the rest pills (frames j-1 .. j+2 of a rod, Dirichlet weights), made on the device."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    off = torch.from_numpy(sc.rod_offsets.astype(np.int64)).cuda()
    pos = torch.from_numpy(sc.rest_pos).cuda()
    rad = torch.from_numpy(sc.radius).cuda()
    rod = torch.randint(0, sc.n_rods, (n,), generator=g, device="cuda")
    nseg = off[rod + 1] - off[rod] - 1
    j = (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * nseg).long()
    t = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    a, b = pos[off[rod] + j], pos[off[rod] + j + 1]
    d = (b - a) / (b - a).norm(dim=1, keepdim=True)
    u = torch.linalg.cross(d, torch.tensor([[0.0, 1.0, 0.0]], dtype=torch.float64, device="cuda").expand(n, 3))
    u = u / u.norm(dim=1, keepdim=True)
    w = torch.linalg.cross(d, u)
    phi = 2.0 * math.pi * torch.rand(n, 1, generator=g, device="cuda", dtype=torch.float64)
    r = ((1 - t) * rad[off[rod] + j] + t * rad[off[rod] + j + 1])[:, None]
    rest = torch.zeros(n, 4, device="cuda")
    rest[:, :3] = (a + t[:, None] * (b - a) + r * (torch.cos(phi) * u + torch.sin(phi) * w)).float()
    loc = j[:, None] + torch.arange(-1, 3, device="cuda")[None]
    loc = torch.minimum(loc.clamp(min=0), nseg[:, None] - 1)
    idx = (off[rod][:, None] - rod[:, None] + loc).int().contiguous()
    e = torch.empty(n, 4, device="cuda").exponential_(generator=g)
    mesh = V.Mesh.__new__(V.Mesh)
    mesh.n, mesh.rest, mesh.idx, mesh.w = n, rest, idx, (e / e.sum(dim=1, keepdim=True)).contiguous()
    mesh.out = torch.empty(n, 4, device="cuda")
    return mesh


def _poses(sc, frames):
    """Bone poses of the given frames of the scene's animation."""
    return [tuple(np.ascontiguousarray(a, np.float32) for a in sc.bone_pose(k * sc.dt)) for k in frames]


def _clip(n):
    """Frame numbers of a clip of n frames that ends where it began, so that it can be played again."""
    return [min(k, n - k) for k in range(1, n + 1)]


def _scene(case, seed):
    """The scene of a clip and its state (None: the rest or initial pose at rest)."""
    if case["kind"] == "rods":
        return _rods_scene(case, seed), None
    if case["kind"] in ("rig", "skin"):
        return _rig_scene(S.muscle_rig(seed=1, n_rods=case["rods"], mesh_verts=0), seed), None
    if case["kind"] == "bundle":
        return _rig_scene(S.bundled_muscles(n_muscles=case["muscles"], fibers=case["fibers"],
                                            n_verts=case["verts"]), seed), None
    return _strands(case, seed)


def _start_state(sc, state):
    """x4, v4, q4, w4 of a clip's first frame."""
    if state is not None:
        return state
    x4 = np.zeros((sc.nv, 4), np.float32)
    x4[:, :3] = sc.rest_pos if sc.init_pos is None else sc.init_pos
    x4[:, 3] = sc.radius
    q4 = np.ascontiguousarray(sc.rest_quat if sc.init_quat is None else sc.init_quat, np.float32)
    return [x4, np.zeros((sc.nv, 4), np.float32), q4, np.zeros((sc.ns, 4), np.float32)]


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    kind = case["kind"]
    if kind == "query":
        sc, state = _strands(case, seed)
        cap = 9 * sc.ns  # falling strands have about 7 candidate pairs a pill
        x4 = torch.from_numpy(state[0]).cuda()
        x4[:, 3] /= torch.from_numpy(sc.radius).float().cuda()
        return {"kind": kind, "nv": sc.nv, "rods": sc.n_rods, "off": torch.from_numpy(sc.rod_offsets).cuda(),
                "group": torch.from_numpy(sc.group).cuda(), "x4": x4,
                "rbar": torch.from_numpy(sc.radius.astype(np.float32)).cuda(), "cap": cap,
                "pairs": torch.empty(cap, 2, dtype=torch.int32, device="cuda"),
                "n": torch.zeros(1, dtype=torch.int32, device="cuda"), "slot": torch.arange(cap, device="cuda")}
    if kind == "scenes":
        rng = np.random.default_rng(seed)
        n = case["scenes"]
        size = lambda lo, hi: [int(round(math.exp(math.log(lo) + (i + 0.5) / n * math.log(hi / lo)))) for i in range(n)]  # noqa: E731
        rods, verts = size(case["rods_lo"], case["rods_hi"]), size(case["mesh_lo"], case["mesh_hi"])
        verts = [verts[7 * i % n] if n % 7 else verts[i - 1] for i in range(n)]  # large meshes on small rigs too
        out = torch.empty(sum(verts), 4, device="cuda")  # the skins of all scenes, one after the other
        scenes, meshes, poses, at = [], [], [], 0
        for i in range(n):
            sc = _rig_scene(S.muscle_rig(seed=40_000 + i, n_rods=rods[i], mesh_verts=0), int(rng.integers(1 << 31)))
            scenes.append(V.Scene(sc))
            mesh = _surface(sc, verts[i], int(rng.integers(1 << 31)))
            mesh.out = out[at:at + verts[i]]
            at += verts[i]
            meshes.append(mesh)
            track = _poses(sc, range(25))  # the animation, played to its end and back
            poses.append(track + track[-2:0:-1])
        return {"kind": kind, "batch": V.Batch(), "scenes": scenes, "meshes": meshes, "poses": poses, "frame": 0,
                "out": out}
    sc, state = _scene(case, seed)
    frame = case.get("solver") == "frame"
    g = V.Scene(sc, solver=V.SOLVER_FRAME if frame else V.SOLVER_AUTO,
                max_pairs=PAIRS_PER_PILL * sc.ns if kind == "hair" else 0)
    start = [torch.from_numpy(a).cuda() for a in _start_state(sc, state)]
    st = {"kind": kind, "scene": g, "start": start, "end": [torch.empty_like(a) for a in start],
          "frames": case.get("frames", 1), "poses": _poses(sc, _clip(case.get("frames", 1))) if sc.bones else None}
    if "mesh" in case:
        st["mesh"] = _surface(sc, case["mesh"], seed)
    if kind == "skin":  # a posed rig: its rods bent away from rest
        g.set_bones(*_poses(sc, [6])[0])
        V._check(V.lib().viper_set_state(g.handle, *_pointers(_posed(sc, seed))), "viper_set_state")
    elif not frame:
        V._check(V.lib().viper_prepare(g.handle, sc.dt, sc.substeps, sc.iterations), "viper_prepare")
    return st


def _pointers(tensors):
    return [C.c_void_p(t.data_ptr()) for t in tensors]


def _posed(sc, seed):
    """A rig's state away from rest: positions moved, radii changed, frames turned."""
    rng = np.random.default_rng(seed + 77)
    x4, v4, q4, w4 = [a.copy() for a in _start_state(sc, None)]
    x4[:, :3] += rng.normal(scale=0.01, size=(sc.nv, 3)).astype(np.float32)
    x4[:, 3] *= rng.uniform(0.8, 1.2, sc.nv).astype(np.float32)
    q4 = S.quat_mul(S.axis_angle_quat(rng.normal(scale=0.3, size=(sc.ns, 3))), q4.astype(np.float64))
    return [torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda() for a in (x4, v4, q4, w4)]


def run(st):
    kind = st["kind"]
    if kind == "skin":
        return st["scene"].skin(st["mesh"])
    if kind == "scenes":
        k = st["frame"] = st["frame"] + 1
        st["batch"].step(st["scenes"], [p[k % len(p)] for p in st["poses"]], st["meshes"], DT, 10, 4)
        torch.cuda.current_stream().wait_stream(st["batch"].stream)
        return st["out"]
    if kind == "query":
        V._check(V.lib().viper_broadphase(st["rods"], st["nv"], *_pointers([st["off"], st["group"], st["x4"], st["rbar"],
                                                                         st["pairs"]]), st["cap"],
                                          *_pointers([st["n"]]), C.c_void_p(torch.cuda.current_stream().cuda_stream)),
                 "viper_broadphase")
        # the list has no order of its own: sorted by its ids (the unused slots last), as a program keeps it
        ids = st["pairs"].view(torch.int64).view(-1)
        return torch.where(st["slot"] < st["n"], (ids << 32) | (ids >> 32), 1 << 62).sort().values
    g = st["scene"]
    V._check(V.lib().viper_set_state(g.handle, *_pointers(st["start"])), "viper_set_state")
    for f in range(st["frames"]):
        if st["poses"] is not None:
            g.set_bones(*st["poses"][f])
        g.step()
        if "mesh" in st:
            g.skin(st["mesh"])
    V._check(V.lib().viper_get_state(g.handle, *_pointers(st["end"])), "viper_get_state")
    return st["end"] + ([st["mesh"].out] if "mesh" in st else [])


def work(case):
    """Unavoidable bytes (each input read once, each output written once) and FP32 operations of run()."""
    kind = case["kind"]
    mean = lambda lo, hi: (hi - lo) / math.log(hi / lo) if hi > lo else float(lo)  # noqa: E731  (of a log-uniform value)
    mesh = 64.0 * case.get("mesh", 0)  # rest, frame ids, weights in, position out
    sweep = 1030.0  # operations of a vertex's constraints in one sweep
    if kind == "skin":
        return {"bytes": mesh, "flops": 4 * 40.0 * case["mesh"]}
    if kind == "query":
        ns = case["rods"] * (case["verts"] - 1)
        return {"bytes": 20.0 * case["rods"] * case["verts"] + 8.0 * 7 * ns, "flops": 9.0 * 7 * ns}
    per_vertex = 128.0 + 104.0  # the state in and out, the rest tables in
    if kind == "scenes":
        nv = case["scenes"] * 36 * mean(case["rods_lo"], case["rods_hi"])
        m = case["scenes"] * mean(case["mesh_lo"], case["mesh_hi"])
        return {"bytes": per_vertex * nv + 64.0 * m, "flops": 40 * sweep * nv + 160.0 * m}
    if kind == "rods":
        nv = case["rods"] * mean(case["nmin"], case["nmax"])
        return {"bytes": per_vertex * nv,
                "flops": case["frames"] * case["substeps"] * case["iterations"] * sweep * nv}
    if kind == "hair":
        nv = case["rods"] * case["verts"]
        ns = nv - case["rods"]
        pairs, touching = (33.0, 11.0) if case["settled"] else (7.0, 0.0)  # per pill and contact pass
        return {"bytes": per_vertex * nv + 80.0 * pairs * ns,
                "flops": 40 * (sweep * nv + (77.5 * pairs + 892.5 * touching) * ns)}
    nv = case["rods"] * 36 if kind == "rig" else case["muscles"] * case["fibers"] * case["verts"]
    frames = case["frames"]
    return {"bytes": per_vertex * nv + frames * mesh, "flops": frames * (40 * sweep * nv + 2.5 * mesh)}


# ---------------------------------------------------------------- 64-bit results
# The method in plain torch: FP64 tensors over all rods, one colour at a time.
def _qmul(a, b):
    ax, ay, az, aw = a.unbind(-1)
    bx, by, bz, bw = b.unbind(-1)
    return torch.stack([aw * bx + bw * ax + ay * bz - az * by, aw * by + bw * ay + az * bx - ax * bz,
                        aw * bz + bw * az + ax * by - ay * bx, aw * bw - ax * bx - ay * by - az * bz], -1)


def _conj(q):
    return q * q.new_tensor([-1.0, -1.0, -1.0, 1.0])


def _unit(q):
    return q / q.norm(dim=-1, keepdim=True)


def _turn(q, v):
    u = q[..., :3]
    t = 2.0 * torch.linalg.cross(u, v)
    return v + q[..., 3:] * t + torch.linalg.cross(u, t)


def _rotate_by(q, d):
    return _unit(q + 0.5 * _qmul(torch.cat([d, torch.zeros_like(d[..., :1])], -1), q))


def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


class _Solver64:
    """One scene's substeps in 64 bits: even / odd colours, contacts by averaging, shape matching."""

    def __init__(self, sc, state):
        t = lambda a: torch.as_tensor(np.asarray(a), device="cuda")  # noqa: E731
        d = lambda a: t(np.asarray(a, np.float64))  # noqa: E731
        n = np.diff(sc.rod_offsets)
        off = sc.rod_offsets[:-1].astype(np.int64)
        rod_v = np.repeat(np.arange(sc.n_rods), n)
        loc = np.arange(sc.nv) - off[rod_v]
        first = np.nonzero(loc < n[rod_v] - 1)[0]
        inner = np.nonzero((loc > 0) & (loc < n[rod_v] - 1))[0]
        rod_s = rod_v[first]
        self.sc, self.v0, self.rbar = sc, t(first), d(sc.radius)
        l = np.linalg.norm(sc.rest_pos[first + 1] - sc.rest_pos[first], axis=1)
        rm = 0.5 * (sc.radius[first] + sc.radius[first + 1])
        mass = math.pi * rm * rm * sc.density[rod_s] * l
        mv, jv = np.zeros(sc.nv), np.zeros(sc.nv)
        for e in (first, first + 1):
            np.add.at(mv, e, 0.5 * mass)
            np.add.at(jv, e, 0.25 * mass * rm * rm)
        w = 1.0 / mv
        w[sc.pin_vertex] = 0.0
        area = math.pi * rm * rm * l
        self.l, self.imr2, self.w, self.ws = d(l)[:, None], d(1.0 / (mass * rm * rm))[:, None], d(w)[:, None], d(1.0 / jv)[:, None]
        self.aS, self.aV = d(sc.c_stretch[rod_s] / area)[:, None], d(sc.c_volume[rod_s] / area)[:, None]
        self.aX, self.aG = 0.5 * self.aS, d(sc.c_stretch[rod_s] / (0.5 * area * rm * rm))[:, None]
        self.segs = [t(np.nonzero(loc[first] % 2 == c)[0]) for c in (0, 1)]
        sid = -np.ones(sc.nv, np.int64)
        sid[first] = np.arange(first.size)
        qr = _unit(d(sc.rest_quat))
        p = _qmul(_conj(qr[t(sid[inner - 1])]), qr[t(sid[inner])])
        p = torch.where(p[:, 3:] < 0, -p, p)
        la, lb = l[sid[inner - 1]], l[sid[inner]]
        r4l = math.pi * sc.radius[inner] ** 4 * 0.5 * (la + lb)
        self.inner, self.ga, self.gb = t(inner), t(sid[inner - 1]), t(sid[inner])
        self.kappa = d(4.0 / (la + lb))[:, None]
        self.rest_om = self.kappa * p[:, :3]
        self.aB, self.aVb = d(sc.c_bend[rod_v[inner]] / r4l)[:, None], d(4.0 * sc.c_volume[rod_v[inner]] / r4l)[:, None]
        self.jp, self.jn = d(2.0 / (la * (la + lb)))[:, None], d(2.0 / (lb * (la + lb)))[:, None]
        self.aL = 2.0 * self.aB
        self.vtx = [t(np.nonzero(loc[inner] % 2 == c)[0]) for c in (0, 1)]
        self.lap = [t(np.nonzero(loc[inner] % 3 == c)[0]) for c in (0, 1, 2)]
        self.group = t(sc.group[rod_s])
        self.pin_v, self.pin_b, self.pin_o = t(sc.pin_vertex.astype(np.int64)), t(sc.pin_bone.astype(np.int64)), d(sc.pin_offset)
        self.planes, self.grav = d(sc.planes), d(sc.gravity)
        x4, v4, q4, w4 = [d(a) for a in state]
        self.x, self.s = x4[:, :3].clone(), x4[:, 3:] / self.rbar[:, None]
        self.v, self.sv, self.q, self.om = v4[:, :3].clone(), v4[:, 3:] / self.rbar[:, None], _unit(q4), w4[:, :3].clone()
        if sc.bundle_offsets is not None:
            self._bundles(sc, off, n, qr)

    def _bundles(self, sc, off, n, qr):
        """Cross-sections (vertex, segment, rest offset) without pins; every bundle has the same shape."""
        t = lambda a: torch.as_tensor(np.asarray(a), device="cuda")  # noqa: E731
        rods = np.asarray(sc.bundle_rods).reshape(len(sc.bundle_offsets) - 1, -1)
        m = int(n[rods[0, 0]])
        pinned = np.zeros(sc.nv, bool)
        pinned[sc.pin_vertex] = True
        verts = (off[rods][:, None, :] + np.arange(m)[None, :, None]).reshape(-1, rods.shape[1])
        segs = verts - np.repeat(rods, m, axis=0)
        framed = np.tile(np.arange(m) < m - 1, rods.shape[0])
        keep = ~pinned[verts].any(axis=1)
        self.xv, self.xs, self.xf = t(verts[keep]), t(np.where(framed, segs.T, 0).T[keep]), t(framed[keep])
        c = torch.as_tensor(sc.rest_pos, device="cuda")[self.xv]
        self.xrel = c - c.mean(dim=1, keepdim=True)
        self.xq = qr[self.xs]
        self.xden = (self.xrel ** 2).sum(dim=(1, 2)) + 3.0 * self.xf * rods.shape[1]

    # -- constraints
    def _segments(self, c, ih2):
        g = self.segs[c]
        a, b = self.v0[g], self.v0[g] + 1
        xa, xb, sa, sb, q = self.x[a], self.x[b], self.s[a], self.s[b], self.q[g]
        wa, wb, wsa, wsb, il = self.w[a], self.w[b], self.ws[a], self.ws[b], 1.0 / self.l[g]
        d3 = _turn(q, torch.zeros_like(xa) + xa.new_tensor([0.0, 0.0, 1.0]))
        k = 4.0 * self.imr2[g] / (0.5 * (sa + sb)) ** 2
        wp, at = (wa + wb) * il * il, self.aS[g] * ih2
        rhs = d3 - (xb - xa) * il - at * self.lS[g]
        dn = _dot(rhs, d3)
        dl = (rhs - dn * d3) / (wp + k + at) + d3 * dn / (wp + at)
        self.lS[g] += dl
        xa, xb = xa - wa * il * dl, xb + wb * il * dl
        q = _rotate_by(q, k * torch.linalg.cross(dl, d3))
        if self.sc.volume:
            d3 = _turn(q, torch.zeros_like(xa) + xa.new_tensor([0.0, 0.0, 1.0]))
            dx, sm = xb - xa, 0.5 * (sa + sb)
            e, jx = _dot(d3, dx), sm * sm * il
            js, jt = sm * e * il, jx * torch.linalg.cross(d3, dx)
            k, at = 4.0 * self.imr2[g] / sm ** 2, self.aV[g] * ih2
            dl = (1.0 - jx * e - at * self.lV[g]) / ((wa + wb) * jx * jx + (wsa + wsb) * js * js + k * _dot(jt, jt) + at)
            self.lV[g] += dl
            xa, xb = xa - wa * jx * dl * d3, xb + wb * jx * dl * d3
            sa, sb = sa + wsa * js * dl, sb + wsb * js * dl
            q = _rotate_by(q, k * dl * jt)
        at = self.aX[g] * ih2
        dl = (1.0 - 0.5 * (sa + sb) - at * self.lX[g]) / (0.25 * (wsa + wsb) + at)
        self.lX[g] += dl
        sa, sb = sa + 0.5 * wsa * dl, sb + 0.5 * wsb * dl
        at = self.aG[g] * ih2
        dl = ((sa - sb) * il - at * self.lG[g]) / ((wsa + wsb) * il * il + at)
        self.lG[g] += dl
        self.x[a], self.x[b], self.q[g] = xa, xb, q
        self.s[a], self.s[b] = sa - wsa * il * dl, sb + wsb * il * dl

    def _vertices(self, c, ih2):
        i = self.vtx[c]
        v, ga, gb = self.inner[i], self.ga[i], self.gb[i]
        qa, qb, s, sp, sn, ws = self.q[ga], self.q[gb], self.s[v], self.s[v - 1], self.s[v + 1], self.ws[v]
        eye = torch.eye(3, dtype=qa.dtype, device=qa.device)
        zero = torch.zeros_like(s)

        def skew(u):
            x, y, z = u.unbind(-1)
            o = torch.zeros_like(x)
            return torch.stack([o, -z, y, z, o, -x, -y, x, o], -1).reshape(-1, 3, 3)

        def matrix(q):
            return torch.stack([_turn(q, eye[k].expand(q.shape[0], 3)) for k in range(3)], -1)

        for volume in ([False, True] if self.sc.volume else [False]):
            p = _qmul(_conj(qa), qb)
            p = torch.where(p[:, 3:] < 0, -p, p)
            om = self.kappa[i] * p[:, :3]
            da, db = 4.0 * self.imr2[ga] / (0.5 * (sp + s)) ** 2, 4.0 * self.imr2[gb] / (0.5 * (s + sn)) ** 2
            body = qa.new_tensor([1.0, 1.0, 0.5])
            ra, rb = matrix(qa), matrix(qb)
            ia = (ra * (da * body)[:, None, :]) @ ra.transpose(1, 2)
            ib = (rb * (db * body)[:, None, :]) @ rb.transpose(1, 2)
            jb = 0.5 * self.kappa[i][..., None] * (p[:, 3, None, None] * eye - skew(p[:, :3])) @ ra.transpose(1, 2)
            rows = 2 if volume else 3
            f, df = (s ** 3, 3.0 * s ** 2) if volume else (s, zero + 1.0)
            J, js = (f[..., None] * jb)[:, :rows], (df * om)[:, :rows]
            lam = (self.lVb if volume else self.lB)[i]
            at = (self.aVb[i] * qa.new_tensor([1.0, 1.0]) if volume else self.aB[i] * qa.new_tensor([4.0, 4.0, 2.0])) * ih2
            A = J @ (ia + ib) @ J.transpose(1, 2) + ws[..., None] * js[:, :, None] * js[:, None, :] + torch.diag_embed(at)
            dl = torch.linalg.solve(A, (self.rest_om[i] - f * om)[:, :rows] - at * lam)
            (self.lVb if volume else self.lB)[i] += dl
            jl = (J.transpose(1, 2) @ dl[..., None])
            qa, qb = _rotate_by(qa, -(ia @ jl)[..., 0]), _rotate_by(qb, (ib @ jl)[..., 0])
            s = s + ws * (js * dl).sum(-1, keepdim=True)
        self.q[ga], self.q[gb], self.s[v] = qa, qb, s

    def _laplacians(self, c, ih2):
        i = self.lap[c]
        v, jp, jn, at = self.inner[i], self.jp[i], self.jn[i], self.aL[i] * ih2
        wp, w, wn = self.ws[v - 1], self.ws[v], self.ws[v + 1]
        C_ = jn * (self.s[v + 1] - self.s[v]) - jp * (self.s[v] - self.s[v - 1])
        dl = (-C_ - at * self.lL[i]) / (wp * jp * jp + w * (jp + jn) ** 2 + wn * jn * jn + at)
        self.lL[i] += dl
        self.s[v - 1] += wp * jp * dl
        self.s[v] -= w * (jp + jn) * dl
        self.s[v + 1] += wn * jn * dl

    # -- contacts
    def _pairs(self):
        """Pills of different groups whose bounding spheres overlap, lower segment first."""
        a, b = self.v0, self.v0 + 1
        c = 0.5 * (self.x[a] + self.x[b])
        r = self.s[:, 0] * self.rbar
        R = 0.5 * (self.x[a] - self.x[b]).norm(dim=1) + torch.maximum(r[a], r[b])
        got = []
        for k in range(0, c.shape[0], 2048):
            near = torch.cdist(c[k:k + 2048], c, compute_mode="donot_use_mm_for_euclid_dist") <= R[k:k + 2048, None] + R[None]
            i, j = near.nonzero(as_tuple=True)
            i = i + k
            ok = (i < j) & (self.group[i] != self.group[j])
            got.append(torch.stack([i[ok], j[ok]]))
        return torch.cat(got, 1)

    def _contacts(self, ih2):
        at = self.sc.contact_compliance * ih2
        dx, ds, cnt = torch.zeros_like(self.x), torch.zeros_like(self.s), torch.zeros_like(self.s)
        r = self.s * self.rbar[:, None]
        if self.pairs.shape[1]:
            va, vb = self.v0[self.pairs[0]], self.v0[self.pairs[1]]
            a1, a2, b1, b2 = self.x[va], self.x[va + 1], self.x[vb], self.x[vb + 1]
            ra1, ra2, rb1, rb2 = r[va], r[va + 1], r[vb], r[vb + 1]
            e = b2 - b1
            l = e.norm(dim=1, keepdim=True)
            u, sn = e / l, (rb1 - rb2) / l
            tn = sn / torch.sqrt((1.0 - sn * sn).clamp(min=1e-300))

            def separation(al):
                p = (1 - al) * a1 + al * a2
                ax = _dot(p - b1, u)
                h = (p - b1 - ax * u).norm(dim=1, keepdim=True)
                be = ((ax - h * tn) / l).clamp(0.0, 1.0)
                be = torch.where(sn >= 1, 0.0, torch.where(sn <= -1, 1.0, be))
                d = p - (1 - be) * b1 - be * b2
                return d.norm(dim=1, keepdim=True) - (1 - al) * ra1 - al * ra2 - (1 - be) * rb1 - be * rb2, be, d

            lo, hi = torch.zeros_like(l), torch.ones_like(l)
            for _ in range(10):
                mid, eps = 0.5 * (lo + hi), 1e-3 * (hi - lo)
                left = separation(mid - 0.5 * eps)[0] < separation(mid + 0.5 * eps)[0]
                lo, hi = torch.where(left, lo, mid - 0.5 * eps), torch.where(left, mid + 0.5 * eps, hi)
            al = 0.5 * (lo + hi)
            C_, be, d = separation(al)
            on = (C_ < 0) & (d.norm(dim=1, keepdim=True) >= 1e-12)
            nrm = d / d.norm(dim=1, keepdim=True).clamp(min=1e-300)
            parts = [(va, 1 - al), (va + 1, al), (vb, be - 1), (vb + 1, -be)]
            den = at + sum((self.w[v] + self.ws[v] * self.rbar[v, None] ** 2) * k * k for v, k in parts)
            dl = torch.where(on, (-C_ - at * self.lC) / den, 0.0)
            self.lC += dl
            for v, k in parts:
                dx.index_add_(0, v, self.w[v] * k * dl * nrm)
                ds.index_add_(0, v, -self.ws[v] * k.abs() * self.rbar[v, None] * dl)
                cnt.index_add_(0, v, on.to(cnt.dtype))
        for k in range(self.planes.shape[0]):
            pl = self.planes[k]
            C_ = self.x @ pl[:3, None] - pl[3] - r
            den = self.w + self.ws * self.rbar[:, None] ** 2 + at
            dl = torch.where(C_ < 0, (-C_ - at * self.lP[k]) / den, 0.0)
            self.lP[k] += dl
            dx += self.w * dl * pl[:3]
            ds -= self.ws * self.rbar[:, None] * dl
            cnt += (C_ < 0).to(cnt.dtype)
        self.x += dx / cnt.clamp(min=1)
        self.s += ds / cnt.clamp(min=1)

    def _match(self):
        c, s, q = self.x[self.xv], self.s[self.xv], self.q[self.xs]
        mu = c.mean(dim=1, keepdim=True)
        A = (c - mu).transpose(1, 2) @ self.xrel
        eye = torch.eye(3, dtype=c.dtype, device=c.device)
        rel = _qmul(q, _conj(self.xq))
        R = torch.stack([_turn(rel, eye[k].expand(*rel.shape[:-1], 3)) for k in range(3)], -1)
        A = A + (s[..., None] * R * self.xf[:, None, None, None]).sum(dim=1)
        U, _, Vh = torch.linalg.svd(A)
        U = U * torch.stack([torch.ones_like(U[:, 0, 0]), torch.ones_like(U[:, 0, 0]), torch.det(U @ Vh)], -1)[:, None, :]
        R = U @ Vh
        sc = (R * A).sum(dim=(1, 2)) / self.xden
        # the rotation's quaternion: the eigenvector of the largest eigenvalue
        K = torch.zeros(R.shape[0], 4, 4, dtype=c.dtype, device=c.device)
        K[:, :3, :3] = R + R.transpose(1, 2) - torch.diagonal(R, dim1=1, dim2=2).sum(-1)[:, None, None] * eye
        K[:, :3, 3] = K[:, 3, :3] = torch.stack([R[:, 2, 1] - R[:, 1, 2], R[:, 0, 2] - R[:, 2, 0], R[:, 1, 0] - R[:, 0, 1]], -1)
        K[:, 3, 3] = torch.diagonal(R, dim1=1, dim2=2).sum(-1)
        best = torch.linalg.eigh(K)[1][:, :, -1][:, None, :]
        turned = _unit(_qmul(best.expand_as(self.xq), self.xq))
        turned = torch.where(_dot(turned, q) < 0, -turned, turned)  # of the two signs, the old frame's
        self.x[self.xv] = mu + sc[:, None, None] * (self.xrel @ R.transpose(1, 2))
        self.s[self.xv] = sc[:, None, None].expand_as(s).clone()
        self.q[self.xs[self.xf]] = turned[self.xf]

    # -- one frame
    def frame(self, bones0, bones1):
        sc = self.sc
        h = DT / sc.substeps
        ih2 = 1.0 / (h * h)
        z = lambda n, k: torch.zeros(n, k, dtype=torch.float64, device="cuda")  # noqa: E731
        for k in range(sc.substeps):
            x0, s0, q0 = self.x.clone(), self.s.clone(), self.q.clone()
            self.x = self.x + h * self.v + h * h * self.grav
            if self.pin_v.numel():
                target = self.pin_o
                if bones1 is not None:
                    t = (k + 1) / sc.substeps
                    (qa, ta), (qb, tb) = bones0, bones1
                    qb = torch.where(_dot(qa, qb) < 0, -qb, qb)
                    b = self.pin_b
                    target = _turn(_unit((1 - t) * qa + t * qb)[b], self.pin_o) + ((1 - t) * ta + t * tb)[b]
                self.x[self.pin_v] = target
            self.s = self.s + h * self.sv
            self.q = _rotate_by(self.q, h * self.om)
            ns, ni = self.v0.numel(), self.inner.numel()
            self.lS, self.lV, self.lX, self.lG = z(ns, 3), z(ns, 1), z(ns, 1), z(ns, 1)
            self.lB, self.lVb, self.lL = z(ni, 3), z(ni, 2), z(ni, 1)
            if sc.contacts:
                self.pairs = self._pairs()
                self.lC, self.lP = z(self.pairs.shape[1], 1), [z(sc.nv, 1) for _ in range(self.planes.shape[0])]
            for _ in range(sc.iterations):
                self._segments(0, ih2)
                self._segments(1, ih2)
                self._vertices(0, ih2)
                self._vertices(1, ih2)
                for c in range(3 if sc.surface_bending else 0):
                    self._laplacians(c, ih2)
                if sc.contacts:
                    self._contacts(ih2)
            if sc.bundle_offsets is not None:
                self._match()
            self.v, self.sv = (self.x - x0) / h, (self.s - s0) / h
            d = _qmul(self.q, _conj(q0))
            self.om = torch.where(d[:, 3:] < 0, -2.0, 2.0) * d[:, :3] / h

    def state(self):
        r = self.rbar[:, None]
        return [torch.cat([self.x, self.s * r], 1), torch.cat([self.v, self.sv * r], 1), self.q,
                torch.cat([self.om, torch.zeros_like(self.om[:, :1])], 1)]


def _skin64(sc, state, mesh):
    """Linear blend skinning of a mesh by the segments' similarity frames."""
    x, q = state[0].double(), _unit(state[2].double())
    v = np.delete(np.arange(sc.nv), sc.rod_offsets[1:] - 1)
    v = torch.as_tensor(v, device="cuda")
    s = x[:, 3] / torch.as_tensor(sc.radius, device="cuda")
    rest = torch.as_tensor(sc.rest_pos, device="cuda")
    r = _unit(_qmul(q, _conj(_unit(torch.as_tensor(sc.rest_quat, device="cuda")))))
    sm = 0.5 * (s[v] + s[v + 1])[:, None]
    cb, c = 0.5 * (rest[v] + rest[v + 1]), 0.5 * (x[v, :3] + x[v + 1, :3])
    out = torch.zeros(mesh.n, 4, dtype=torch.float64, device="cuda")
    for k in range(4):
        g = mesh.idx[:, k].long()
        out[:, :3] += mesh.w[:, k:k + 1].double() * (sm[g] * _turn(r[g], mesh.rest[:, :3].double() - cb[g]) + c[g])
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "query":
        return None  # whole numbers
    if kind == "scenes" and case["scenes"] > 1:
        return None  # many rigs one after the other: minutes in 64 bits
    if kind == "hair":
        # hundreds of thousands of pills: too long in 64 bits; and piled-up strands
        # move apart exponentially from differences of one rounding
        return None
    sc, state = _scene(case, seed)
    if kind == "skin":
        return _skin64(sc, _posed(sc, seed), _surface(sc, case["mesh"], seed))
    solver = _Solver64(sc, _start_state(sc, state))
    poses = None
    if sc.bones:
        poses = [[torch.as_tensor(np.asarray(a, np.float32), device="cuda").double() for a in p]
                 for p in _poses(sc, [0] + _clip(case["frames"]))]
        # the pose the scene starts from and every later one as unit quaternions
        poses = [(_unit(q), t) for q, t in poses]
    for f in range(case["frames"]):
        solver.frame(poses[f] if poses else None, poses[f + 1] if poses else None)
    out = solver.state()
    return out + ([_skin64(sc, out, _surface(sc, case["mesh"], seed))] if "mesh" in case else [])
