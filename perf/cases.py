"""Performance cases: the calls that users of the simulator make, over the sizes they make them at.

Every case goes through the public binding (`Context`, `Scene`, `BatchJob`, `SpectraFn`).  Scenes, sensors and
materials are generated from a seed with the shapes of the repository's workloads: the 4 x 3 x 2.5 m room, clutter
(spheres and posts on a ground plane), leaves around a bat, a forest of instanced plants.

Kinds of pass
  simulate  one pose of a prepared scene: spectra (and, with `signal`, the received signals of a call)
  frame     the same for a moving sensor: emitter and receivers set again, then simulated
  train     a differentiable simulate and its backward pass (`SpectraFn`), as in fitting materials and positions
  adjoint   simulate and the reverse pass on device buffers (`Context.backward`)
  poses     many poses over several scenes in one batched call
  move      instances of a forest moved, then simulated
  build     a mesh loaded and pre-processed (hierarchy, curvature, sample counts)
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2602_19652_gb300 as st

F32 = np.float32
SPEED, ALPHA = 343.0, 0.033          # m/s; air absorption in dB / (m kHz), the library's defaults
BANDS = 16

_SIM = dict(kind="simulate", scene="clutter", tris=20_000, materials=4, rays=100_000, bounces=3, mics=32, bins=128,
            lo_khz=20, hi_khz=80, samples=1_000_000, array_m=0.06, per_mic=False, tables=False, diffraction=True,
            signal=0)


def listed():
    return [
        # the smallest call: the empty room, one omnidirectional microphone, 10k rays (latency of a call)
        dict(_SIM, name="room_one_mic", scene="room", tris=12, materials=1, rays=10_000, mics=1, bins=128),
        # one step of fitting wall materials, lobe widths, microphone and emitter positions in the room
        dict(_SIM, name="room_train", kind="train", scene="room", tris=12, rays=10_000, mics=32, bins=128,
             diffraction=False),
        # a frame of the paper's robot: 80k rays, three hits, 32 microphones, 14 bins, the sensor moved each frame
        dict(_SIM, name="robot_frame", kind="frame", tris=50_000, rays=80_000, mics=32, bins=14,
             samples=500_000),
        # the paper's bioacoustic setup: 600k rays, three hits, 64 microphones, 14 bins
        dict(_SIM, name="bio_64_mics", tris=100_000, rays=600_000, mics=64, bins=14, lo_khz=30, hi_khz=90,
             samples=4_000_000),
        # the benchmark workload: 200k triangles, 1M rays x 5 bounces, 32 microphones x 512 bins, 4M samples
        dict(_SIM, name="clutter_large", tris=200_000, rays=1_000_000, bounces=5, bins=512, samples=4_000_000),
        # odd sizes and the received signals of a call: 17 microphones x 331 bins, specular and direct paths
        dict(_SIM, name="echo_odd", tris=3_000, rays=60_011, bounces=4, mics=17, bins=331, hi_khz=95,
             diffraction=False, signal=3001),
        # a bat among leaves: two ears with their directivity, a piston mouth, 1024 bins
        dict(_SIM, name="bat_leaves", scene="leaves", tris=1_000_000, materials=2, rays=1_000_000, bounces=4, mics=2,
             bins=1024, hi_khz=120, samples=1_000_000, tables=True),
        # microphones spread over the scene, each with its own visibility test
        dict(_SIM, name="spread_mics", tris=60_000, rays=77_777, bounces=4, mics=24, bins=257, array_m=5.0,
             per_mic=True, samples=300_000),
        # gradients of a sensor array in a cluttered scene, forward and reverse pass
        dict(_SIM, name="clutter_adjoint", kind="adjoint", tris=200_000, rays=200_000, bounces=5, bins=512,
             samples=1_000_000),
        # a pose sweep: 20 poses over 4 scenes, 2-64 microphones, 256-2048 bins, 1-5 bounces
        dict(_SIM, name="pose_sweep", kind="poses", tris=60_000, rays=32_768, bounces=5, mics=64, bins=2048,
             samples=65_536, poses=20, scenes=4),
        # a dynamic forest: every plant moved (rigidly), then one simulate
        dict(_SIM, name="forest_move", kind="move", scene="forest", tris=0, plants=2_000, rays=100_000, mics=8,
             bins=128, samples=400_000),
        # geometric pre-processing of a mesh that a user loads
        dict(_SIM, name="scene_build", kind="build", tris=200_000, samples=4_000_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["simulate"] * 4 + ["frame", "frame", "train", "adjoint", "poses", "move", "build"])
    c = dict(_SIM, kind=kind, tris=_log(rng, 2_000, 200_000), materials=rng.randint(1, 6), bounces=rng.randint(1, 6),
             mics=_log(rng, 1, 64), bins=_log(rng, 8, 1024), samples=_log(rng, 20_000, 2_000_000),
             lo_khz=rng.choice([20, 25, 30]), hi_khz=rng.choice([70, 80, 96, 120]), array_m=rng.choice([0.03, 0.06, 0.5]))
    c["rays"] = _log(rng, 5_000, 600_000)
    if kind in ("simulate", "frame"):
        c["scene"] = rng.choice(["clutter", "clutter", "room", "leaves"])
        c["diffraction"] = rng.random() < 0.8
        c["per_mic"] = rng.random() < 0.15
        c["signal"] = rng.choice([0, 0, _log(rng, 500, 5000)])
        c["tables"] = c["mics"] <= 8 and rng.random() < 0.5
    elif kind == "train":
        c.update(scene="room", rays=_log(rng, 2_000, 30_000), diffraction=False, mics=_log(rng, 2, 48),
                 bins=_log(rng, 16, 256))
    elif kind == "adjoint":
        c.update(rays=_log(rng, 5_000, 150_000))
    elif kind == "poses":
        c.update(rays=_log(rng, 2_000, 32_768), mics=rng.randint(8, 64), bins=_log(rng, 256, 2048),
                 samples=_log(rng, 4_096, 65_536), poses=rng.randint(4, 20), scenes=rng.randint(1, 4))
    elif kind == "move":
        c.update(scene="forest", tris=0, plants=_log(rng, 50, 3_000), mics=_log(rng, 2, 16), rays=_log(rng, 5_000, 200_000))
    if c["scene"] == "room":
        c.update(tris=12, materials=rng.choice([1, 4]))
    if c["scene"] == "leaves":
        c.update(tris=_log(rng, 8_000, 800_000), materials=2)
    # no dearer than the largest listed case: terms, visibility rays
    per_ray = c["bounces"] * c["mics"] * max(c["bins"], 32) * (4 if kind == "adjoint" else 1) * c.get("poses", 1)
    c["rays"] = max(1_000, min(c["rays"], int(4e10 / per_ray)))
    if c["per_mic"]:
        c["rays"] = max(1_000, min(c["rays"], int(2e7 / (c["bounces"] * c["mics"]))))
    return c


# ------------------------------------------------------------------------------------------------ inputs
def _ico(level):
    t = (1 + math.sqrt(5)) / 2
    v = np.array([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t], [0, 1, -t],
                  [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]]) / math.sqrt(1 + t * t)
    f = np.array([[0, 11, 5], [0, 5, 1], [0, 1, 7], [0, 7, 10], [0, 10, 11], [1, 5, 9], [5, 11, 4], [11, 10, 2],
                  [10, 7, 6], [7, 1, 8], [3, 9, 4], [3, 4, 2], [3, 2, 6], [3, 6, 8], [3, 8, 9], [4, 9, 5], [2, 4, 11],
                  [6, 2, 10], [8, 6, 7], [9, 8, 1]])
    for _ in range(level):
        edges = np.sort(np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]), 1)
        pairs, at = np.unique(edges, axis=0, return_inverse=True)
        mid = v[pairs].sum(1)
        v, (a, b, c) = (np.concatenate([v, mid / np.linalg.norm(mid, axis=1, keepdims=True)]),
                        len(v) + at.reshape(3, -1))
        f = np.concatenate([np.stack(x, 1) for x in ((f[:, 0], a, c), (f[:, 1], b, a), (f[:, 2], c, b), (a, b, c))])
    return v, f


def _post(seg):
    a = np.arange(seg) * (2 * math.pi / seg)
    ring = np.stack([np.cos(a), np.sin(a)], 1)
    v = np.concatenate([np.c_[ring, np.zeros(seg)], np.c_[ring, np.ones(seg)], [[0, 0, 0]], [[0, 0, 1]]])
    i, j = np.arange(seg), (np.arange(seg) + 1) % seg
    return v, np.concatenate([np.stack(x, 1) for x in (
        (i, j, seg + j), (i, seg + j, seg + i), (np.full(seg, 2 * seg), j, i), (np.full(seg, 2 * seg + 1), seg + i, seg + j))])


_GROUND = (np.array([[0, 0, 0], [20, 0, 0], [20, 20, 0], [0, 20, 0]], float), np.array([[0, 1, 2], [0, 2, 3]]))
_SENSOR = np.array([10.0, 10.0, 1.0])
_SHAPES = {}


def _shape(key, make):
    if key not in _SHAPES:
        _SHAPES[key] = make()
    return _SHAPES[key]


def _join(parts, mats):
    base = np.cumsum([0] + [len(v) for v, _ in parts])
    verts = np.concatenate([v for v, _ in parts]).astype(F32)
    tris = np.concatenate([f + b for (_, f), b in zip(parts, base)]).astype(np.int32)
    n = [len(f) for _, f in parts]
    return dict(verts=verts, tris=tris, mat=np.repeat(np.asarray(mats, np.int32), n),
                obj=np.repeat(np.arange(len(parts), dtype=np.int32), n))


def _mesh(c, rng):
    """verts, tris, material and object of each triangle, and the sensor's place."""
    if c["scene"] == "room":
        size = np.array([4.0, 3.0, 2.5])
        v = size * np.array([[0, 0, 0], [1, 0, 0], [1, 1, 0], [0, 1, 0], [0, 0, 1], [1, 0, 1], [1, 1, 1], [0, 1, 1]])
        f = np.array([[0, 1, 2], [0, 2, 3], [4, 7, 6], [4, 6, 5], [0, 3, 7], [0, 7, 4], [1, 5, 6], [1, 6, 2], [0, 4, 5],
                      [0, 5, 1], [3, 2, 6], [3, 6, 7]])
        m = _join([(v, f)], [0])
        m["mat"] = (np.array([0, 0, 1, 1, 2, 2, 2, 2, 3, 3, 3, 3]) % c["materials"]).astype(np.int32)
        return m, rng.uniform(0.8, size - 0.8)
    if c["scene"] == "leaves":
        n = max(1, c["tris"] // 8)
        a = np.arange(8) * (math.pi / 4)
        disc = np.concatenate([[[0, 0]], np.stack([np.cos(a), np.sin(a)], 1)])
        u = rng.normal(size=(n, 3, 3))
        u[:, 0] /= np.linalg.norm(u[:, 0], axis=1, keepdims=True)
        u[:, 1] -= (u[:, 1] * u[:, 0]).sum(1, keepdims=True) * u[:, 0]
        u[:, 1] /= np.linalg.norm(u[:, 1], axis=1, keepdims=True)
        place = u[:, 2] / np.linalg.norm(u[:, 2], axis=1, keepdims=True)
        place *= 6 * np.cbrt(rng.uniform(0.05 ** 3, 1, n))[:, None]
        v = place[:, None] + np.einsum("kj,nji->nki", disc, u[:, :2]) * rng.uniform(0.02, 0.05, n)[:, None, None]
        fan = np.array([[0, 1 + i, 1 + (i + 1) % 8] for i in range(8)])
        return dict(verts=v.reshape(-1, 3).astype(F32),
                    tris=(fan[None] + 9 * np.arange(n)[:, None, None]).reshape(-1, 3).astype(np.int32),
                    mat=np.repeat(rng.integers(0, 2, n), 8).astype(np.int32),
                    obj=np.repeat(np.arange(n) // 256, 8).astype(np.int32)), np.zeros(3)
    parts, mats, count = [_GROUND], [0], 2
    fine = 1 if c["tris"] < 20_000 else 2
    pick = np.random.default_rng(c["tris"])  # which objects: the case's own, so that every seed has as many triangles
    while count < c["tris"]:
        if pick.uniform() < 0.5:
            r = math.exp(pick.uniform(math.log(0.05), math.log(0.5)))
            level = fine + (r > 0.12) + (r > 0.25)
            (v, f), size = _shape(("ico", level), lambda: _ico(level)), np.array([r, r, r])
            low, high, flat = np.array([r, r, r]), np.array([20 - r, 20 - r, 5 - r]), [1, 1, 1]
        else:
            r, seg = pick.uniform(0.02, 0.2), int(pick.integers(16, 33))
            (v, f), size = _shape(("post", seg), lambda: _post(seg)), np.array([r, r, pick.uniform(0.2, 3)])
            low, high, flat = np.array([1, 1, 0.0]), np.array([19, 19, 0.0]), [1, 1, 0]
        at = rng.uniform(low, high)
        while np.linalg.norm((at - _SENSOR) * flat) < r + 0.6:
            at = rng.uniform(low, high)
        parts.append((v * size + at, f))
        mats.append(int(rng.integers(0, c["materials"])))
        count += len(f)
    return _join(parts, mats), _SENSOR


def _curves(rng, n, lo, hi):
    x = np.linspace(0, 1, BANDS)
    s = sum(rng.uniform(0.3, 1, (n, 1)) * np.cos(2 * math.pi * rng.uniform(0.2, 1.5, (n, 1)) * x
                                                 + rng.uniform(0, 2 * math.pi, (n, 1))) for _ in range(3))
    s = (s - s.min(1, keepdims=True)) / np.maximum(np.ptp(s, axis=1)[:, None], 1e-9)
    return (lo + (hi - lo) * s).astype(F32)


def _directions(n):
    i = np.arange(n, dtype=np.float64)
    z = 1 - (2 * i + 1) / n
    phi, rho = i * (math.pi * (3 - math.sqrt(5))), np.sqrt(np.maximum(0, 1 - z * z))
    return np.stack([rho * np.cos(phi), rho * np.sin(phi), z], 1).astype(F32)


def _quat(rng):
    q = rng.normal(size=4)
    return (q / np.linalg.norm(q)).astype(F32)


def _array(rng, n, radius, at, room):
    """n microphones: a disc facing +x around `at`, or with a large radius a spread over the scene."""
    r, a = radius * np.sqrt(rng.uniform(0, 1, n)), rng.uniform(0, 2 * math.pi, n)
    off = np.stack([np.zeros(n), r * np.cos(a), r * np.sin(a)], 1)
    if radius > 1:
        off = np.stack([r * np.cos(a), r * np.sin(a), rng.uniform(-0.5, 0.5, n)], 1)
    return (at + off).astype(F32)


def _ear(rng, n_az=90, n_el=46):
    el, az = np.meshgrid(np.linspace(-math.pi / 2, math.pi / 2, n_el), -math.pi + 2 * math.pi * np.arange(n_az) / n_az,
                         indexing="ij")
    d = np.stack([np.cos(el) * np.cos(az), np.cos(el) * np.sin(az), np.sin(el)], -1)
    axis = np.array([0.8, 0, 0]) + 0.4 * rng.normal(size=3)
    sharp = 1 + 4 * np.arange(BANDS) / (BANDS - 1)
    v = np.exp(sharp * ((d @ (axis / np.linalg.norm(axis)))[..., None] - 1))
    return (0.05 + 0.95 * (v - v.min()) / np.ptp(v)).astype(F32)


def _problem(c, seed):
    """Everything that a user's program has on the host before it touches the library."""
    rng = np.random.default_rng([int(seed), 17])
    mesh, at = _mesh(c, rng) if c["scene"] != "forest" else (None, _SENSOR)
    n, lo, hi = c["materials"], c["lo_khz"] * 1e3, c["hi_khz"] * 1e3
    p = dict(mesh=mesh, at=at, rng=rng, lo=lo, hi=hi, band=np.linspace(lo, hi, BANDS).astype(F32),
             k=_curves(rng, n, 0.3, 0.95), beta=np.deg2rad(_curves(rng, n, 5, 30)).astype(F32),
             diff=_curves(rng, n, 0.02, 0.08), dirs=_directions(c["rays"]),
             emitter=(at + [0.01, 0, 0]).astype(F32), quat=_quat(rng),
             mics=_array(rng, c["mics"], c["array_m"], at, c["scene"] == "room"))
    if c["scene"] == "room":  # anywhere in the room
        p["emitter"] = rng.uniform(0.3, [3.7, 2.7, 2.2]).astype(F32)
    p["fov"] = math.pi / 2 if c["scene"] == "leaves" else math.pi
    if c["tables"]:
        p["ears"] = np.stack([_ear(rng) for _ in range(c["mics"])])
        p["ear_quats"] = np.stack([_quat(rng) for _ in range(c["mics"])])
    return p


def _piston(c, p, radius=0.002, n_theta=1801):
    """Directivity of a circular piston, |2 J1(x) / x| with x = k a sin(theta), on the device."""
    th = torch.linspace(0, math.pi, n_theta, dtype=torch.float64, device="cuda")
    k = 2 * math.pi * torch.linspace(p["lo"], p["hi"], c["bins"], dtype=torch.float64, device="cuda") / SPEED
    x = torch.sin(th)[:, None] * (k * radius)
    return torch.where(x > 1e-12, 2 * torch.special.bessel_j1(x) / x.clamp_min(1e-12), 1.0).abs().float()


# ------------------------------------------------------------------------------------------------ states
def _params(c, **more):
    on = st.ST_COMP_SPECULAR | st.ST_COMP_DIRECT | (st.ST_COMP_DIFFRACTION if c["diffraction"] else 0)
    return st.sim_params(max_bounces=c["bounces"], max_distance=60.0, components=on,
                         los_mode=st.ST_LOS_PER_MIC if c["per_mic"] else st.ST_LOS_REFERENCE, **more)


def _scene(ctx, c, p):
    m = p["mesh"]
    scene = st.Scene(ctx, m["verts"], m["tris"], m["mat"], m["obj"])
    scene.set_materials(p["band"], p["k"], p["beta"], p["diff"])
    scene.precompute(st.curv_params(sample_budget=c["samples"]))
    return scene


def _dev(x):
    return torch.as_tensor(x, device="cuda")


def _sensor(ctx, c, p, s):
    ctx.set_frequencies(c["bins"], p["lo"], p["hi"])
    s["table"] = _piston(c, p) if c["tables"] else None
    s["ears"] = _dev(p["ears"]) if c["tables"] else None
    s["ear_quats"] = _dev(p["ear_quats"]) if c["tables"] else None
    s["dirs"], s["mics"] = _dev(p["dirs"]), _dev(p["mics"])
    s.update(emitter=p["emitter"], quat=p["quat"], fov=p["fov"])
    _set_pose(ctx, s)


def _set_pose(ctx, s):
    ctx.set_emitter(s["emitter"], s["quat"], s["dirs"], s["table"], s["fov"])
    ctx.set_receivers(s["mics"], s["ear_quats"], s["ears"])


def _plants(c, rng):
    """Shared meshes (ground, tree, bush, rock), the plants' meshes and their maps, and the maps after a move."""
    trunk, crown, bush, rock = _post(12), _ico(2), _ico(3), _ico(0)
    tree_v = np.concatenate([trunk[0] * [0.08, 0.08, 2], crown[0] * 0.7 + [0, 0, 2.5]])
    tree_f = np.concatenate([trunk[1], crown[1] + len(trunk[0])])
    tree_m = np.repeat([1, 2], [len(trunk[1]), len(crown[1])])
    n = c["materials"]
    protos = [(_GROUND[0].astype(F32), _GROUND[1].astype(np.int32), np.zeros(2, np.int32)),
              (tree_v.astype(F32), tree_f.astype(np.int32), (tree_m % n).astype(np.int32)),
              ((bush[0] * 0.45 + [0, 0, 0.45]).astype(F32), bush[1].astype(np.int32),
               np.full(len(bush[1]), 2 % n, np.int32)),
              ((rock[0] * 0.25 + [0, 0, 0.2]).astype(F32), rock[1].astype(np.int32), np.full(len(rock[1]), 3 % n, np.int32))]
    count = c["plants"]
    kind = np.concatenate([[0], rng.integers(1, 4, count)]).astype(np.int32)
    ang = rng.uniform(0, 2 * math.pi, count)
    rad = np.sqrt(rng.uniform(1.5 ** 2, 9.5 ** 2, count))
    place = _SENSOR[:2] + rad[:, None] * np.stack([np.cos(ang), np.sin(ang)], 1)

    def maps(turn, size, shift):
        x = np.zeros((count + 1, 3, 4))
        x[0, :, :3] = np.eye(3)
        x[1:, 0, 0] = x[1:, 1, 1] = size * np.cos(turn)
        x[1:, 0, 1], x[1:, 1, 0], x[1:, 2, 2] = -size * np.sin(turn), size * np.sin(turn), size
        x[1:, :2, 3] = place + shift
        return x.astype(F32)

    turn, size = rng.uniform(0, 2 * math.pi, count), rng.uniform(0.6, 1.4, count)
    return protos, kind, maps(turn, size, 0.0), maps(turn + rng.normal(0, 0.2, count), size,
                                                     rng.normal(0, 0.05, (count, 2)))


def prepare(case, seed):
    c, p = case, _problem(case, seed)
    rng, s = p["rng"], dict(case=case)
    if c["kind"] == "build":
        return dict(s, ctx=st.Context(0), problem=p)
    ctx = s["ctx"] = st.Context(0)
    s["params"] = _params(c)
    if c["kind"] == "poses":
        pick, scenes = np.random.default_rng(c["poses"]), []  # the sizes of the jobs are the case's own
        for _ in range(c["scenes"]):
            size = dict(c, tris=int(c["tris"] * pick.uniform(0.3, 1.7)))
            scenes.append(_scene(ctx, c, dict(p, mesh=_mesh(size, rng)[0])))
        dirs, s["jobs"] = _dev(p["dirs"]), []
        for i in range(c["poses"]):
            at = _SENSOR + rng.uniform([-2, -2, -0.5], [2, 2, 0.5])
            mics = _array(rng, int(pick.integers(2, c["mics"] + 1)), c["array_m"], at, False)
            s["jobs"].append(st.BatchJob(scenes[i % len(scenes)], (at + [0.01, 0, 0]).astype(F32), _quat(rng), dirs,
                                         mics, int(pick.integers(c["bins"] // 8, c["bins"] + 1)), p["lo"], p["hi"],
                                         int(pick.integers(1, c["bounces"] + 1)), pose_index=i))
        return s
    if c["kind"] == "move":
        protos, kind, maps, moved = _plants(c, rng)
        scene = st.Scene.from_instances(ctx, protos, kind, maps)
        scene.set_materials(p["band"], p["k"], p["beta"], p["diff"])
        scene.precompute(st.curv_params(sample_budget=c["samples"]))
        s["moved"] = _dev(moved)
    else:
        scene = _scene(ctx, c, p)
    s["scene"] = scene
    _sensor(ctx, c, p, s)
    if c["signal"]:
        s["call"] = _call(seed)
    if c["kind"] in ("adjoint", "train"):
        s["grad"] = _upstream(c, seed)
    if c["kind"] == "train":
        s["leaves"] = [_dev(x).requires_grad_() for x in (p["k"], p["mics"], p["emitter"], p["beta"])]
    return s


SIGNAL_HZ = 250e3


def _call(seed, n=500):
    """A 2 ms falling chirp with a random phase."""
    t = torch.arange(n, device="cuda", dtype=torch.float64) / SIGNAL_HZ
    phase = 2 * math.pi * (80e3 * t - 1.25e7 * t * t) + (seed % 628) / 100
    return (torch.sin(phase) * torch.hann_window(n, periodic=False, device="cuda", dtype=torch.float64)).float()


def _upstream(c, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 5)
    return torch.randn((3, c["mics"], c["bins"]), dtype=torch.complex64, device="cuda", generator=g)


# ------------------------------------------------------------------------------------------------ the passes
def run(state):
    c, ctx = state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "build":
        p = state["problem"]
        scene = _scene(ctx, c, p)
        G, C, n = scene.curvature()
        scene.close()
        return {"curvature": G, "metric": C, "samples": n}
    if kind == "poses":
        return [S.unbind(0) for S in ctx.simulate_batch(state["jobs"], state["params"])]
    scene, params = state["scene"], state["params"]
    if kind == "train":
        k, mics, emitter, beta = state["leaves"]
        S = st.SpectraFn.apply(ctx, scene, params, k, mics, emitter, beta)
        gk, gm, ge, gb = torch.autograd.grad(S, (k, mics, emitter, beta), state["grad"])
        return {"spectra": S.detach().unbind(0), "k": gk, "mics": gm, "emitter": ge, "beta": gb}
    if kind == "frame":
        _set_pose(ctx, state)
    if kind == "move":
        scene.set_instance_transforms(state["moved"], keep_curvature=True)
    S = ctx.simulate(scene, params)
    specular, diffraction, direct = S.unbind(0)
    out = {"specular": specular, "diffraction": diffraction, "direct": direct}
    if kind == "adjoint":
        out["k"], out["mics"], out["emitter"] = ctx.backward(scene, state["grad"], c["materials"], BANDS)
    if c["signal"]:
        out["signal"] = ctx.impulse_response(S, c["lo_khz"] * 1e3, c["hi_khz"] * 1e3, SIGNAL_HZ, c["signal"],
                                             call=state["call"])
    return out


# shares of a scene's records and samples that reach the sensor, and of its rays that find a hit (about)
_SHARE = dict(room=(1.0, 0.5, 1.0), clutter=(0.16, 0.27, 0.38), leaves=(0.1, 0.1, 0.8), forest=(0.25, 0.2, 0.5))
# floating operations that a path tracer cannot do without for one ray (about 20 boxes and 4 triangles), and for one
# (path, microphone, bin) term: a phasor step and a complex sum
_RAY_FLOPS, _TERM_FLOPS = 700, 10


def work(case):
    c = case
    seen, kept, hit = _SHARE[c["scene"]]
    mesh = 12 * 1.5 * c["tris"] + 8 * c["tris"]          # positions and indices, normals or materials
    if c["kind"] == "build":
        return dict(bytes=mesh + 8 * c["tris"], flops=200 * c["tris"])
    if c["kind"] == "move":
        mesh = 700 * c["plants"] * 20 + 48 * c["plants"]
    samples = c["samples"] * 0.5 if c["diffraction"] else 0
    records = c["rays"] * c["bounces"] * hit
    paths = c["rays"] * c["bounces"] * seen + samples * kept
    times = 1.0
    if c["kind"] == "poses":                             # bounces, microphones and bins spread over their ranges
        times, mesh = c["poses"] * 0.5 * 0.56 * 0.6, mesh * c["scenes"]
    terms = paths * c["mics"] * c["bins"] * times * (3.0 if c["kind"] in ("train", "adjoint") else 1.0)
    rays = (records * (1 + (c["mics"] if c["per_mic"] else 1)) + samples) * times
    io = 12 * c["rays"] + 24 * c["mics"] * c["bins"] * (2 if c["kind"] in ("train", "adjoint") else 1) * (
        c["poses"] * 0.56 if c["kind"] == "poses" else 1)
    tables = (1801 * c["bins"] * 4 + c["mics"] * 46 * 90 * BANDS * 4) if c["tables"] else 0
    return dict(bytes=mesh + io + tables + 4 * c["signal"] * c["mics"],
                flops=_RAY_FLOPS * rays + _TERM_FLOPS * terms + 8.0 * c["signal"] * c["mics"] * c["bins"])


# ------------------------------------------------------------------------------------------------ 64-bit values
_TESTS = 2e10  # ray-triangle tests of the plain tracer, about ten seconds


def _d(x):
    return torch.as_tensor(np.asarray(x, np.float64), device="cuda")


def _nearest(V, o, d, skip, far=None):
    """Plain Moeller-Trumbore over all triangles: (t, triangle) of the nearest hit, or whether any lies before `far`."""
    n, (v0, e1, e2) = len(o), V
    t_out = torch.full((n,), math.inf, dtype=torch.float64, device="cuda")
    i_out = torch.full((n,), -1, dtype=torch.long, device="cuda")
    step = max(1, int(2e7) // len(v0))
    normal = torch.linalg.cross(e1, e2)
    for a in range(0, n, step):
        O, D = o[a:a + step], d[a:a + step]
        det = -(D @ normal.T)
        inv = 1 / det
        # o - v0 enters through three triple products that split into per-ray and per-triangle parts
        odn = O @ normal.T - (v0 * normal).sum(1)
        m = torch.linalg.cross(O, D)
        u = (m @ e2.T + D @ torch.linalg.cross(v0, e2).T) * inv
        v = -(m @ e1.T + D @ torch.linalg.cross(v0, e1).T) * inv
        t = odn * inv
        ok = (u >= -1e-12) & (v >= -1e-12) & (u + v <= 1 + 1e-12) & (t > 1e-5) & torch.isfinite(t)
        s = skip[a:a + step]
        ok[torch.nonzero(s >= 0)[:, 0], s[s >= 0]] = False
        if far is not None:
            ok &= t < far[a:a + step, None]
        t = torch.where(ok, t, math.inf)
        t_out[a:a + step], i_out[a:a + step] = t.min(1)
    return t_out, torch.where(torch.isfinite(t_out), i_out, -1)


def _turn(q, v):
    t = 2 * torch.linalg.cross(q[1:].expand_as(v), v)
    return v + q[0] * t + torch.linalg.cross(q[1:].expand_as(v), t)


def _trace(c, p):
    """The specular paths: for each visible record its ray's chain of triangles and directions."""
    m = p["mesh"]
    corner = _d(m["verts"])[torch.as_tensor(m["tris"].astype(np.int64), device="cuda")]
    V = corner[:, 0], corner[:, 1] - corner[:, 0], corner[:, 2] - corner[:, 0]
    normal = torch.nn.functional.normalize(torch.linalg.cross(V[1], V[2]), dim=1)
    mics, source = _d(p["mics"]), _d(p["emitter"])
    d = _turn(_d(p["quat"]), _d(p["dirs"]))
    n = len(d)
    o, r = source.expand(n, 3), torch.zeros(n, dtype=torch.float64, device="cuda")
    prev, chain, heads, paths = torch.full((n,), -1, device="cuda"), [], [d], []
    for j in range(c["bounces"]):
        t, tri = _nearest(V, o, d, prev)
        hit = tri >= 0
        o, d, r, tri, t = o[hit], d[hit], r[hit], tri[hit], t[hit]
        chain, heads = [x[hit] for x in chain] + [tri], [x[hit] for x in heads]
        o = o + t[:, None] * d
        d = d - 2 * (d * normal[tri]).sum(1, keepdim=True) * normal[tri]
        d = torch.nn.functional.normalize(d, dim=1)
        heads, r = heads + [d], r + t
        targets = mics if c["per_mic"] else mics.mean(0, keepdim=True)
        sees = torch.stack([_sees(V, o, x, tri) for x in targets], 1).expand(len(o), len(mics))
        some = sees.any(1)
        paths.append(dict(tri=[x[some] for x in chain], dir=[x[some] for x in heads], sees=sees[some]))
        go = r < 60.0
        o, d, r, prev = o[go], d[go], r[go], tri[go]
        chain, heads = [x[go] for x in chain], [x[go] for x in heads]
    direct = torch.stack([_sees(V, source[None], x, torch.full((1,), -1, device="cuda"))[0] for x in mics])
    return paths, direct, V, normal


def _sees(V, o, target, skip):
    to = target - o
    far = to.norm(dim=1) - 1e-4
    _, tri = _nearest(V, o, to / to.norm(dim=1, keepdim=True), skip, far)
    return tri < 0


def _bands(c, p):
    """Bin frequencies and the bins' weights over the material bands."""
    f = torch.linspace(p["lo"], p["hi"], c["bins"], dtype=torch.float64, device="cuda") if c["bins"] > 1 else _d([p["lo"]])
    band = _d(p["band"])
    at = torch.clamp(torch.searchsorted(band, f, right=True) - 1, 0, BANDS - 2)
    w = torch.clamp((f - band[at]) / (band[at + 1] - band[at]), 0, 1)
    W = torch.zeros((BANDS, c["bins"]), dtype=torch.float64, device="cuda")
    cols = torch.arange(c["bins"], device="cuda")
    W[at, cols] = 1 - w
    W[at + 1, cols] += w
    return f, W


def _wave(r, f):
    """Spreading, air absorption and delay."""
    amp = torch.exp(-2 * torch.log(r)[..., None] - r[..., None] * (ALPHA * f / 1e3 * (math.log(10) / 20)))
    return torch.polar(amp, torch.remainder(r[..., None] * (f / SPEED), 1.0) * (2 * math.pi))


def _specular(c, p, path, geometry, k, beta, mics, source):
    """Summed spectra of one chunk of paths of equal length (differentiable; chain and directions frozen)."""
    V, normal, mat = geometry
    f, W = _bands(c, p)
    P, r, gain = source.expand(len(path["tri"][0]), 3), 0.0, 1.0
    for tri, d in zip(path["tri"], path["dir"]):
        t = ((V[0][tri] - P) * normal[tri]).sum(1) / (d * normal[tri]).sum(1)
        P, r, gain = P + t[:, None] * d, r + t, gain * (k @ W)[mat[tri]]
    to = mics[None] - P[:, None]
    dist = to.norm(dim=2)
    u, d = to / dist[..., None], path["dir"][-1][:, None].expand_as(to)
    gamma = torch.atan2(torch.linalg.cross(d, u).norm(dim=2), (d * u).sum(2))
    lobe = torch.exp(-(gamma ** 2)[..., None] * ((1 / (2 * beta ** 2)) @ W)[mat[path["tri"][-1]]][:, None])
    return (_wave(r[:, None] + dist, f) * (lobe * gain[:, None]) * path["sees"][..., None]).sum(0)


def _chunks(c, paths):
    for path in paths:
        step = max(1, int(4e7) // (c["mics"] * c["bins"]))
        for a in range(0, len(path["sees"]), step):
            yield {k: [x[a:a + step] for x in v] if isinstance(v, list) else v[a:a + step] for k, v in path.items()}


def _curvature(case, p):
    """Meyer's discrete mean curvature at the welded vertices and the triangles' metric (Eq. 1)."""
    m = p["mesh"]
    V, weld = np.unique(m["verts"] + F32(0), axis=0, return_inverse=True)
    weld = torch.as_tensor(weld.reshape(-1), device="cuda")
    T = weld[torch.as_tensor(m["tris"].astype(np.int64), device="cuda")]
    x = _d(V)[T]
    area2 = torch.linalg.cross(x[:, 1] - x[:, 0], x[:, 2] - x[:, 0]).norm(dim=1)
    e = lambda a, b: x[:, b] - x[:, a]  # noqa: E731
    dots = torch.stack([(e(i, (i + 1) % 3) * e(i, (i + 2) % 3)).sum(1) for i in range(3)], 1)
    cot, obtuse = dots / area2[:, None], (dots < 0).any(1)
    K = torch.zeros((len(V), 3), dtype=torch.float64, device="cuda")
    A = torch.zeros(len(V), dtype=torch.float64, device="cuda")
    for i in range(3):
        a, b = (i + 1) % 3, (i + 2) % 3
        K.index_add_(0, T[:, i], -(cot[:, b, None] * e(i, a) + cot[:, a, None] * e(i, b)))
        voronoi = (e(i, b).square().sum(1) * cot[:, a] + e(i, a).square().sum(1) * cot[:, b]) / 8
        A.index_add_(0, T[:, i], torch.where(obtuse, area2 / torch.where(dots[:, i] < 0, 4.0, 8.0), voronoi))
    G = K.norm(dim=1) / (4 * A.clamp_min(1e-300))
    g = G[T]
    C = torch.clamp(area2 / 2 / 1e-4, 0, 1) * (g.amax(1) - g.amin(1))
    return {"curvature": G[weld].cpu().numpy(), "metric": C.cpu().numpy(), "samples": None}


def exact(case, seed):
    c = case
    if c["kind"] == "build":
        return _curvature(c, _problem(c, seed))
    tests = c["rays"] * max(c["tris"], 1) * c["bounces"] * (1 + (c["mics"] if c["per_mic"] else 1))
    if c["kind"] in ("poses", "move", "adjoint") or c["tables"] or tests > _TESTS:
        return None
    p = _problem(c, seed)
    paths, seen, V, normal = _trace(c, p)
    f, _ = _bands(c, p)
    mat = torch.as_tensor(p["mesh"]["mat"].astype(np.int64), device="cuda")
    leaves = [_d(x) for x in (p["k"], p["mics"], p["emitter"], p["beta"])]
    train = c["kind"] == "train"
    grads = [torch.zeros_like(x) for x in leaves]
    if train:
        leaves = [x.requires_grad_() for x in leaves]
    up = _upstream(c, seed).to(torch.complex128) if train else None
    k, mics, source, beta = leaves

    def add(total, part, g):
        if train and part.requires_grad:
            for acc, x in zip(grads, torch.autograd.grad(part, leaves, g, allow_unused=True)):
                if x is not None:
                    acc += x
        total += part.detach()

    specular = torch.zeros((c["mics"], c["bins"]), dtype=torch.complex128, device="cuda")
    direct = torch.zeros_like(specular)
    for path in _chunks(c, paths):
        add(specular, _specular(c, p, path, (V, normal, mat), k, beta, mics, source), up[0] if train else None)
    add(direct, _wave((mics - source).norm(dim=1), f) * seen[:, None], up[2] if train else None)
    if train:
        S = specular, torch.zeros_like(specular), direct
        return {"spectra": S, "k": grads[0], "mics": grads[1], "emitter": grads[2], "beta": grads[3]}
    none = torch.zeros_like(specular)
    out = {"specular": specular, "diffraction": None if c["diffraction"] else none, "direct": direct}
    if c["signal"]:
        out["signal"] = None if c["diffraction"] else _received(c, p, f, specular + direct, seed)
    return out


def _received(c, p, f, S, seed):
    call = _call(seed).double()
    i = torch.arange(len(call), dtype=torch.float64, device="cuda") / SIGNAL_HZ
    E = (torch.exp(2j * math.pi * torch.outer(f, i)) @ call.to(torch.complex128)) / SIGNAL_HZ
    t = torch.arange(c["signal"], dtype=torch.float64, device="cuda") / SIGNAL_HZ
    df = (p["hi"] - p["lo"]) / (c["bins"] - 1) if c["bins"] > 1 else 1.0
    return 2 * df * ((S * E) @ torch.exp(-2j * math.pi * torch.outer(f, t))).real
