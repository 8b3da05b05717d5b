"""What a user of this library has it do, as cases that can be timed.

Every case is one call sequence of the public binding (`gg.Sim`, `gg_bin_sort_noalloc`)
on inputs a user's program would hold: time steps of scenes with the shapes and sizes of
the benchmark and the tests, the host-driven loop over pinned buffers, a taped rollout
with its reverse pass, the two depth cameras, the allocation-free binning.

The scenes are packed beds generated here from the seed alone: a jittered lattice of
spheres (the recipe of `scenes.jittered_lattice`, +-10 or 15 % radii) at the density
where neighbours touch, relaxed geometrically until only small penetrations are left, so
a sphere has about as many contacts (2-4), as deep, as in a bed that has settled.  A pass
puts that state in, takes the steps and reads the new state (an environment that is
reset to, or exchanged at, a given state); bodies go on from where the last pass left
them, as they do in a simulation that is kept.

`exact` gives the same outputs in 64 bits with plain torch: contact decisions are the
documented FP32 ones (Eq. 6-7 tests on float32 positions), everything else is float64.
"""
from __future__ import annotations

import ctypes
import functools
import math

import numpy as np
import torch

from paper_2306_01369_gb300 import gg, scenes

DEV = "cuda"
F32, F64 = torch.float32, torch.float64


# --------------------------------------------------------------------------- #
# the cases
# --------------------------------------------------------------------------- #

def listed():
    return [
        # one step of the benchmark's small settle box: a call whose cost is all launches
        {"name": "settle_4k", "kind": "step", "scene": "box", "n": 4096, "steps": 1, "tune_table": False},
        # a 16k-sphere column (a size of the table and loop experiments), several steps a call
        {"name": "column_16k", "kind": "step", "scene": "column", "n": 16384, "steps": 8, "tune_table": False},
        # the headline: 262,144 spheres mid-collapse, a packed foot under spheres still falling
        {"name": "collapse_262k", "kind": "step", "scene": "collapse", "n": 262144, "steps": 4, "tune_table": True},
        # the same spheres come to rest: every one of them in contact
        {"name": "pile_262k", "kind": "step", "scene": "column", "n": 262144, "steps": 4, "tune_table": True},
        # a stirred bed: an odd count, ids in no spatial order, as after pouring or mixing
        {"name": "stirred_100k", "kind": "step", "scene": "stirred", "n": 100003, "steps": 3, "tune_table": False},
        # gears as sampled SDFs in a tube with the cyclic vertical boundary
        {"name": "tower_65k", "kind": "step", "scene": "tower", "n": 65536, "steps": 4, "tune_table": False},
        # the largest scene: 1M-sphere excavation, scoop and two free cubes, 30 sweeps,
        # the wrench on every body of every step read back
        {"name": "excavation_1m", "kind": "step", "scene": "excavation", "n": 1048576, "steps": 2, "tune_table": True},
        # 64 environments of 8k-64k spheres stepped together, each with its own scoop
        {"name": "batch_64", "kind": "batch", "envs": 64, "n_min": 8192, "n_max": 65536, "steps": 2},
        # the host-driven loop at the paper's 50,000-particle excavation: state in from
        # pinned host memory, one step, state out
        {"name": "host_loop_50k", "kind": "io", "n": 50000},
        # a taped rollout and the gradient w.r.t. the tool's path and mu
        {"name": "gradient_32k", "kind": "grad", "n": 32768, "steps": 20, "every": 20},
        # one observation: the sky (height) camera and the ego (depth) camera
        {"name": "cameras_262k", "kind": "views", "n": 262144, "sky_w": 72, "sky_h": 36, "ego_w": 36, "ego_h": 36},
        # the allocation-free binning of an odd number of spheres
        {"name": "binning_300k", "kind": "bin", "n": 300007, "factor": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "batch", "io", "grad", "views", "bin"])
    if kind == "step":
        scene = rng.choice(["box", "column", "collapse", "stirred", "tower", "excavation"])
        hi = {"box": 65536, "column": 300000, "collapse": 400000, "stirred": 400000, "tower": 131072,
              "excavation": 800000}[scene]
        n = _log(rng, 1000, hi)
        return {"kind": kind, "scene": scene, "n": n, "steps": rng.randint(1, 8 if n < 70000 else 2),
                "tune_table": rng.random() < 0.5}
    if kind == "batch":
        lo = _log(rng, 1500, 12000)
        return {"kind": kind, "envs": rng.randint(2, 48), "n_min": lo, "n_max": lo + _log(rng, 1000, 30000),
                "steps": rng.randint(1, 2)}
    if kind == "io":
        return {"kind": kind, "n": _log(rng, 1000, 300000)}
    if kind == "grad":
        return {"kind": kind, "n": _log(rng, 1500, 32000), "steps": rng.randint(4, 16), "every": rng.randint(4, 12)}
    if kind == "views":
        return {"kind": kind, "n": _log(rng, 4000, 600000), "sky_w": rng.randint(24, 160), "sky_h": rng.randint(24, 96),
                "ego_w": rng.randint(24, 96), "ego_h": rng.randint(24, 96)}
    return {"kind": kind, "n": _log(rng, 2000, 1 << 20), "factor": rng.choice([1, 2])}


# --------------------------------------------------------------------------- #
# scenes
# --------------------------------------------------------------------------- #

OFFSETS = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1) if (a, b, c) > (0, 0, 0)]


def _slices(d, n):
    return (slice(0, n - d), slice(d, n)) if d >= 0 else (slice(-d, n), slice(0, n + d))


def _packed(dims, r0, jit, gen, spread=1.015, relax=40):
    """(nx, ny, nz) lattice of touching spheres, z-major, as float64 (n, 3) and radii (n,);
    the lower corner of the lattice is at the origin, pitch = 2 r0 spread.  Overlaps are
    relaxed by moving each overlapping lattice neighbour pair half-way apart."""
    nx, ny, nz = dims
    pitch = 2.0 * r0 * spread
    r = r0 * (1.0 + jit * (2.0 * torch.rand((nz, ny, nx), generator=gen, device=DEV, dtype=F64) - 1.0))
    x = torch.empty((nz, ny, nx, 3), device=DEV, dtype=F64)
    x[..., 0] = (torch.arange(nx, device=DEV, dtype=F64) + 0.5) * pitch
    x[..., 1] = ((torch.arange(ny, device=DEV, dtype=F64) + 0.5) * pitch)[:, None]
    x[..., 2] = ((torch.arange(nz, device=DEV, dtype=F64) + 0.5) * pitch)[:, None, None]
    x += 0.1 * r0 * (2.0 * torch.rand(x.shape, generator=gen, device=DEV, dtype=F64) - 1.0)
    # walls and floor: a small penetration, another one per axis (a corner sphere's nearest
    # wall is then decided by more than rounding)
    lo = r[..., None] * torch.tensor([0.998, 0.9965, 0.995], device=DEV, dtype=F64)
    hi = torch.tensor([nx * pitch, ny * pitch, 1e9], device=DEV, dtype=F64) - lo
    for _ in range(relax):
        move = torch.zeros_like(x)
        for a, b, c in OFFSETS:
            if abs(a) + abs(b) + abs(c) == 3 or min(nz - abs(a), ny - abs(b), nx - abs(c)) <= 0:
                continue
            (z0, z1), (y0, y1), (x0, x1) = _slices(a, nz), _slices(b, ny), _slices(c, nx)
            d = x[z0, y0, x0] - x[z1, y1, x1]
            dist = d.norm(dim=-1).clamp_min(1e-9)
            push = (0.5 * (r[z0, y0, x0] + r[z1, y1, x1] - dist).clamp_min(0.0) / dist)[..., None] * d
            move[z0, y0, x0] += push
            move[z1, y1, x1] -= push
        x += 0.4 * move
        x = torch.minimum(torch.maximum(x, lo), torch.maximum(hi, lo))
    return x.reshape(-1, 3), r.reshape(-1), pitch


class Case:
    """Inputs of one case: device arrays, bodies per environment, parameters."""

    def __init__(self, x, r, gen, bodies, params, offsets=None, twist=None, speed=0.02, fall=None):
        n = x.shape[0]
        self.pos = torch.empty((n, 4), device=DEV, dtype=F32)
        self.pos[:, :3] = x
        self.pos[:, 3] = r
        v = speed * torch.randn((n, 3), generator=gen, device=DEV, dtype=F64)
        if fall is not None:
            v[:, 2] -= fall
        self.vel = v.to(F32).contiguous()
        self.mass = (scenes.DENSITY * (4.0 / 3.0) * math.pi * self.pos[:, 3].double() ** 3).to(F32)
        self.bodies = bodies              # list per environment
        self.params = params
        self.offsets = offsets            # numpy (E + 1) or None
        self.twist = twist or {}          # (environment, body) -> float32 (steps, 6)
        self.n = n

    def sim(self, tune_table=False, wrench_history=1, max_bodies=8):
        free = sum(int(b.is_free) for env in self.bodies for b in env)
        s = gg.Sim(self.pos, self.vel, self.mass, params=self.params, env_offsets=self.offsets,
                   wrench_history=wrench_history, max_bodies=max_bodies, max_free_bodies=free,
                   hash_tune=int(tune_table))
        for e, env in enumerate(self.bodies):
            s.set_bodies(env, e)
        for (e, b), tw in self.twist.items():
            s.set_trajectory(b, tw, e)
        return s


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _side(n, layers):
    return max(2, int(math.ceil(math.sqrt(n / layers))))


@functools.lru_cache(maxsize=1)
def _gear():
    return scenes.gear_body(10, 0.003, 0.012, margin=0.005).grid     # one geometry, baked once


def _bed(n, r0, jit, layers, seed, cubes, steps=64):
    """A packed bed in a container with a scoop dug in (spheres its walls would cut left
    out), on the first steps of a seeded dig path; optionally two free cubes on top."""
    gen = _gen(seed)
    side = _side(n, layers)
    layers = -(-n // (side * side)) + max(2, layers // 8) + 1
    x, r, pitch = _packed((side, side, layers), r0, jit, gen, 1.035 if jit > 0.12 else 1.02)
    foot = side * pitch
    x[:, :2] -= 0.5 * foot
    height = n / (side * side) * pitch
    scale = min(1.0, foot / 0.6) * r0 / 2e-3 if foot > 0.15 else 0.35 * foot / 0.12
    tw, rv, p0 = scenes.waypoint_twists(seed * 7 + 3, steps, 1e-4, (-0.2 * foot, 0.0, height - 0.02 * scale),
                                        0.5 * height, 0.6 * foot, pos_jit=0.02 * scale, rot_range=0.2)
    scoop = scenes.scoop_body(scale, pos=p0, rotvec=rv)
    box = scenes.Body(kind=scenes.OPEN_BOX, shape=(0.5 * foot, 0.5 * foot, 0.0))
    f = _sdf(scoop, _to_body(scoop, x.to(F32), F32), F32)[0].double()
    keep = f > 0.97 * r
    keep &= torch.cumsum(keep.long(), 0) <= n
    x, r = x[keep], r[keep]
    assert x.shape[0] == n
    bodies = [box, scoop]
    if cubes:
        s = 0.03 if foot > 0.3 else 0.1 * foot
        m = scenes.DENSITY * s ** 3
        top = float(x[:, 2].max()) + 0.5 * s + 0.6 * r0
        for cx in (0.15 * foot, 0.32 * foot):
            bodies.append(scenes.Body(kind=scenes.BOX, shape=(0.5 * s,) * 3, pos=(cx, 0.2 * foot, top), is_free=1,
                                      mass=m, inertia=(m * s * s / 6.0,) * 3))
    return x, r, gen, bodies, tw


def _scene(case, seed):
    """The case's inputs, from the seed alone."""
    kind = case["kind"]
    if kind == "batch":
        u = np.random.RandomState(case["n_min"] * 64 + case["envs"]).rand(case["envs"], 2)   # sizes: the case's
        ne = np.rint(np.exp(math.log(case["n_min"]) + u[:, 0] * math.log(case["n_max"] / case["n_min"]))).astype(int)
        xs, rs, bodies, twist, off = [], [], [], {}, [0]
        for e in range(case["envs"]):
            x, r, gen, bl, tw = _bed(int(ne[e]), 2e-3 + 2e-3 * float(u[e, 1]), 0.10, 16, seed * 131 + e, False)
            xs.append(x)
            rs.append(r)
            bodies.append(bl)
            twist[(e, 1)] = tw
            off.append(off[-1] + x.shape[0])
        return Case(torch.cat(xs), torch.cat(rs), _gen(seed), bodies, scenes.Params(dt=1e-4, mu=0.5, pja_iters=20),
                    offsets=np.asarray(off, np.uint32), twist=twist)
    n = case["n"]
    scene = case.get("scene", {"io": "bed", "grad": "bed", "views": "bed", "bin": "column"}.get(kind))
    if scene in ("bed", "excavation"):
        big = scene == "excavation"
        layers = 64 if n >= 128 * 128 * 48 else max(8, int(round(n ** (1.0 / 3.0) * 0.6)))
        x, r, gen, bodies, tw = _bed(n, 2e-3, 0.15 if big else 0.10, layers, seed, big)
        return Case(x, r, gen, [bodies], scenes.Params(dt=1e-4, mu=0.5, pja_iters=30 if big else 20),
                    twist={(0, 1): tw})
    gen = _gen(seed)
    if scene == "tower":
        radius, r0, gap = 0.06, 2e-3, 0.04
        side = int(2.0 * radius / (2.0 * r0)) + 1
        layers = int(1.6 * n / (side * side)) + 24
        x, r, pitch = _packed((side, side, layers), r0, 0.10, gen)
        x[:, :2] -= 0.5 * side * pitch
        bodies = [scenes.Body(kind=scenes.TUBE, shape=(radius,))]
        u = np.random.RandomState(seed + 1).rand(10, 4)
        keep = x[:, :2].norm(dim=1) < radius - 0.985 * r
        for k in range(10):
            q = np.concatenate([[1.0], (2.0 * u[k, :3] - 1.0)])
            q /= np.linalg.norm(q)
            a, b, c, d = q
            axis = np.array([2 * (b * d + a * c), 2 * (c * d - a * b), 1 - 2 * (b * b + c * c)])
            body = scenes.Body(kind=scenes.GRID, pos=(0.0, 0.0, gap * (k + 1)), quat=tuple(float(v) for v in q),
                               ang_vel=tuple(float(v) for v in 4.0 * (2.0 * u[k, 3] - 1.0) * axis), grid=_gear())
            keep &= _sdf(body, _to_body(body, x.to(F32), F32), F32)[0].double() > 0.97 * r
            bodies.append(body)
        keep &= torch.cumsum(keep.long(), 0) <= n
        x, r = x[keep], r[keep]
        assert x.shape[0] == n
        top = max(float(x[:, 2].max()) + 2.0 * r0, 11.0 * gap)
        return Case(x, r, gen, [bodies], scenes.Params(dt=1e-4, mu=0.5, pja_iters=20, cyclic_z=(0.0, top)))
    if scene == "box":
        side = max(2, int(math.ceil((n * 17.0 * 17.0 / 4096.0 * 1.0) ** 0.5))) if n >= 4096 else max(4, int(n ** 0.37))
        layers = -(-n // (side * side))
        x, r, pitch = _packed((side, side, layers), 5e-3, 0.10, gen)
        half = 0.5 * side * pitch
        body = scenes.Body(kind=scenes.OPEN_BOX, shape=(half, half, 0.0), pos=(half, half, 0.0))
        return Case(x[:n], r[:n], gen, [[body]], scenes.Params(dt=1e-4, mu=0.5, pja_iters=20))
    if scene == "stirred":
        side = max(4, int(round(n ** (1.0 / 3.0))) + 2)
        x, r, pitch = _packed((side, side, -(-n // (side * side))), 2e-3, 0.10, gen)
        order = torch.randperm(n, generator=gen, device=DEV)
        half = 0.5 * side * pitch
        body = scenes.Body(kind=scenes.OPEN_BOX, shape=(half, half, 0.0), pos=(half, half, 0.0))
        return Case(x[:n][order], r[:n][order], gen, [[body]], scenes.Params(dt=1e-4, mu=0.5, pja_iters=20))
    # columns on a ground plane: packed through ("column") or only at the foot ("collapse")
    side = 40 if n >= 40 * 40 * 4 else max(2, int(round((n / 4.0) ** (1.0 / 3.0))))
    layers = -(-n // (side * side))
    ground = scenes.Body(kind=scenes.PLANE)
    params = scenes.Params(dt=5e-5, mu=0.6, pja_iters=20)
    if scene == "column":
        x, r, _ = _packed((side, side, layers), 2e-3, 0.10, gen)
        return Case(x[:n], r[:n], gen, [[ground]], params)
    foot = max(1, int(0.16 * layers))
    xa, ra, pitch = _packed((side, side, foot), 2e-3, 0.10, gen)
    xb, rb, pb = _packed((side, side, layers - foot if layers > foot else 1), 2e-3, 0.10, gen, spread=1.122, relax=0)
    xb[:, :2] += 0.5 * side * (pitch - pb)
    xb[:, 2] += foot * pitch + 2e-4
    x, r = torch.cat([xa, xb])[:n], torch.cat([ra, rb])[:n]
    fall = torch.zeros(x.shape[0], device=DEV, dtype=F64)
    fall[xa.shape[0]:] = 0.25
    return Case(x, r, gen, [[ground]], params, speed=0.005, fall=fall)


# --------------------------------------------------------------------------- #
# what is timed
# --------------------------------------------------------------------------- #

TOOL = 1     # the scoop's index in a bed's bodies


def _cameras(case, foot):
    sky = scenes.Camera(kind=scenes.HEIGHT_CAMERA, width=case["sky_w"], height=case["sky_h"],
                        extent=(foot, 0.5 * foot), empty=0.0)
    ego = scenes.Camera(kind=scenes.DEPTH_CAMERA, width=case["ego_w"], height=case["ego_h"],
                        pos=(-0.45 * foot, 0.0, 0.45), quat=(math.cos(1.205), 0.0, math.sin(1.205), 0.0), fov_y=1.2,
                        near=0.01, far=1.5, march_steps=96, march_eps=1e-4)
    return sky, ego


def _seeds(sc, case):
    """dL/dx, dL/dv, dL/dpose of a smooth loss: the mass near the scoop's cavity."""
    scoop = sc.bodies[0][TOOL]
    c = torch.tensor(scoop.pos, device=DEV, dtype=F64)
    d = sc.pos[:, :3].double() - c
    s = 0.5 * max(scoop.shape[0:3])
    w = sc.mass.double() * torch.exp(-(d * d).sum(1) / (2 * s * s)) / s
    gpos = (w[:, None] * d / s).to(F32).contiguous()
    gvel = (1e-3 * w[:, None] * torch.ones_like(d)).to(F32).contiguous()
    gpose = torch.tensor([0.3, -0.2, 0.5, 0.0, 0.02, -0.01, 0.03], device=DEV, dtype=F32) * float(w.sum())
    return gpos, gvel, gpose


def prepare(case, seed):
    kind = case["kind"]
    sc = _scene(case, seed)
    st = {"case": case, "scene": sc}
    if kind == "bin":
        n = sc.n
        st["cell"] = float(np.float32(2.002 * float(sc.pos[:, 3].max())))
        st["nh"] = int(case["factor"]) * n
        st["out"] = [torch.empty(m, device=DEV, dtype=torch.int32) for m in (n, n, st["nh"] + 1)]
        return st
    if kind == "grad":
        sim = sc.sim()
        sim.autotune()
        sim.tape_reserve(case["steps"], case["every"])
        st["start"] = sim.state()
        st["seeds"] = _seeds(sc, case)
        st["out"] = torch.empty(7 * sc.n, device=DEV, dtype=F32)
    elif kind == "views":
        sim = sc.sim()
        foot = 2.0 * sc.bodies[0][0].shape[0]
        st["cams"] = _cameras(case, foot)
        st["out"] = [torch.empty((c.height, c.width), device=DEV, dtype=F32) for c in st["cams"]]
    elif kind == "io":
        sim = sc.sim(tune_table=True)
        sim.autotune()
        st["pos"], st["vel"] = sc.pos.cpu().pin_memory(), sc.vel.cpu().pin_memory()
        st["out"] = torch.empty(7 * sc.n, dtype=F32).pin_memory()
    else:
        steps = case["steps"]
        nb = max(len(b) for b in sc.bodies)
        sim = sc.sim(tune_table=case.get("tune_table", True), wrench_history=steps, max_bodies=max(8, nb))
        sim.autotune()
        st["out"] = torch.empty(7 * sc.n, device=DEV, dtype=F32)
        st["wrench"] = torch.empty((steps, sim.n_envs * sim.max_bodies, 6), device=DEV, dtype=F32)
    st["sim"] = sim
    return st


def run(state):
    case, sc = state["case"], state["scene"]
    stream = torch.cuda.current_stream()
    kind = case["kind"]
    if kind == "bin":
        keys, perm, start = state["out"]
        rc = gg.load().gg_bin_sort_noalloc(ctypes.c_void_p(sc.pos.data_ptr()), sc.n, ctypes.c_float(state["cell"]),
                                           state["nh"], ctypes.c_void_p(keys.data_ptr()),
                                           ctypes.c_void_p(perm.data_ptr()), ctypes.c_void_p(start.data_ptr()),
                                           ctypes.c_void_p(stream.cuda_stream))
        if rc != gg.OK:
            raise RuntimeError(f"gg_bin_sort_noalloc: status {rc}")
        return [keys, perm, start]
    sim = state["sim"]
    if kind == "views":
        for cam, img in zip(state["cams"], state["out"]):
            sim.render(cam, out=img, stream=stream)
        return list(state["out"])
    if kind == "io":
        sim.step_io(state["pos"], state["vel"], state["out"], stream=stream)
        return [state["out"]]
    if kind == "grad":
        sim.set_state(state["start"], stream=stream)
        sim.step_taped(TOOL, case["steps"], stream=stream)
        sim.pos_vel(out=state["out"], stream=stream)
        dtw, dmu = sim.backward(*state["seeds"], stream=stream)
        return [state["out"], dtw, dmu]
    sim.set_particles(sc.pos, sc.vel, stream=stream)
    sim.step(case["steps"], stream=stream)
    sim.pos_vel(out=state["out"], stream=stream)
    sim.read("BODY_WRENCH", out=state["wrench"], stream=stream)
    return [state["out"], state["wrench"]]


def work(case):
    """Bytes a pass must move (each input read and each output written once) and the
    arithmetic of its sweeps: about 60 operations per directed contact and sweep, at 3
    contacts a sphere (0.5 for a column in collapse)."""
    kind = case["kind"]
    if kind == "batch":
        lo, hi = case["n_min"], case["n_max"]
        n = case["envs"] * ((hi - lo) / math.log(hi / lo) if hi > lo else lo)
        return {"bytes": 60.0 * n, "flops": 60.0 * 3.0 * n * 20 * case["steps"]}
    n = case["n"]
    if kind == "bin":
        return {"bytes": 16.0 * n + 8.0 * n + 4.0 * (case["factor"] * n + 1), "flops": 10.0 * n}
    if kind == "views":
        px = case["sky_w"] * case["sky_h"] + case["ego_w"] * case["ego_h"]
        return {"bytes": 2 * 16.0 * n + 4.0 * px, "flops": 40.0 * n + 3000.0 * px}
    if kind == "io":
        return {"bytes": 60.0 * n, "flops": 60.0 * 3.0 * n * 20}
    if kind == "grad":
        return {"bytes": 60.0 * n + 28.0 * n + 24.0 * case["steps"], "flops": 4.0 * 60.0 * 3.0 * n * 20 * case["steps"]}
    c = 0.5 if case["scene"] == "collapse" else 3.0
    iters = 30 if case["scene"] == "excavation" else 20
    return {"bytes": 60.0 * n, "flops": 60.0 * c * n * iters * case["steps"]}


# --------------------------------------------------------------------------- #
# the same in 64 bits
# --------------------------------------------------------------------------- #

def _quat_R(q, dt):
    """Rotation matrix (3, 3) of a quaternion (w, x, y, z), each entry in the order the
    FP32 decisions document."""
    w, x, y, z = [torch.as_tensor(v, dtype=dt, device=DEV) for v in q] if not torch.is_tensor(q) else q.to(dt)
    return torch.stack([
        torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)]),
        torch.stack([2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)]),
        torch.stack([2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)])])


def _unit_q(b):
    q = np.asarray(b.quat, np.float64)
    nq = float(np.linalg.norm(np.asarray(b.quat, np.float32).astype(np.float64)))
    return np.asarray(b.quat, np.float32).astype(np.float64) if abs(nq - 1.0) < 1e-6 else np.float32(q / nq).astype(float)


def _rotT(R, d):
    """R^T d, the first two products summed first (FP32 decisions depend on the order)."""
    return torch.stack([(R[0, k] * d[:, 0] + R[1, k] * d[:, 1]) + R[2, k] * d[:, 2] for k in range(3)], 1)


def _to_body(b, x, dt, p=None, q=None):
    p = torch.tensor(np.asarray(b.pos, np.float32).astype(np.float64), device=DEV).to(dt) if p is None else p.to(dt)
    R = _quat_R(torch.tensor(_unit_q(b), device=DEV) if q is None else q, dt)
    return _rotT(R, x.to(dt) - p)


def _box(y, h):
    """Box SDF and its unit gradient."""
    q = y.abs() - h
    m = q.clamp_min(0.0)
    s = (m[:, 0] * m[:, 0] + m[:, 1] * m[:, 1]) + m[:, 2] * m[:, 2]
    out = s > 0
    mx = q.max(dim=1).values
    f = torch.where(out, s, torch.ones_like(s)).sqrt() * out + mx.clamp_max(0.0)
    ax = torch.where((q[:, 0] >= q[:, 1]) & (q[:, 0] >= q[:, 2]), 0, torch.where(q[:, 1] >= q[:, 2], 1, 2))
    sg = torch.where(y < 0, -1.0, 1.0).to(y.dtype)
    g_in = torch.nn.functional.one_hot(ax, 3).to(y.dtype) * sg
    g_out = m * sg / torch.where(out, s, torch.ones_like(s)).sqrt()[:, None]
    return f, torch.where((mx > 0)[:, None], g_out, g_in)


def _sdf(b, y, dt):
    """(f, unit gradient) of body b at body-frame points y, arithmetic in dt."""
    sh = torch.tensor(np.asarray(b.shape12(), np.float32).astype(np.float64), device=DEV).to(dt)
    if b.kind == scenes.PLANE:
        g = torch.zeros_like(y)
        g[:, 2] = 1.0
        return y[:, 2], g
    if b.kind == scenes.BOX:
        return _box(y, sh[:3])
    if b.kind == scenes.BOX_MINUS_BOX:
        fa, ga = _box(y, sh[:3])
        fb, gb = _box(y - sh[6:9], sh[3:6])
        a = fa >= -fb
        return torch.where(a, fa, -fb), torch.where(a[:, None], ga, -gb)
    if b.kind == scenes.OPEN_BOX:
        w = torch.stack([sh[0] - y[:, 0], y[:, 0] + sh[0], sh[1] - y[:, 1], y[:, 1] + sh[1], y[:, 2] + sh[2]], 1)
        f, k = w.min(dim=1)
        nrm = torch.tensor([[-1.0, 0, 0], [1, 0, 0], [0, -1, 0], [0, 1, 0], [0, 0, 1]], device=DEV, dtype=dt)
        return f, nrm[k]
    if b.kind == scenes.TUBE:
        rho = (y[:, 0] * y[:, 0] + y[:, 1] * y[:, 1]).clamp_min(1e-30).sqrt()
        return sh[0] - rho, torch.stack([-y[:, 0] / rho, -y[:, 1] / rho, torch.zeros_like(rho)], 1)
    v = torch.as_tensor(b.grid.values, device=DEV).to(dt)
    nz, ny, nx = v.shape
    h = np.float32(b.grid.spacing)
    ih = torch.tensor(float(np.float32(1.0 / np.float64(h))), device=DEV, dtype=dt)
    u = (y - sh[:3]) * ih
    lim = torch.tensor([nx - 1, ny - 1, nz - 1], device=DEV, dtype=dt)
    ok = ((u >= 0) & (u <= lim)).all(dim=1)
    i = torch.minimum(u.floor().clamp_min(0.0), lim - 1).clamp_max(float(max(nx, ny, nz))).nan_to_num(0.0).long()
    t = u - i.to(dt)
    at = lambda a, c, e: v[i[:, 2] + a, i[:, 1] + c, i[:, 0] + e]        # noqa: E731
    lerp = lambda a, c, w: a + w * (c - a)                                # noqa: E731
    tx, ty, tz = t[:, 0], t[:, 1], t[:, 2]
    c00, c10 = lerp(at(0, 0, 0), at(0, 0, 1), tx), lerp(at(0, 1, 0), at(0, 1, 1), tx)
    c01, c11 = lerp(at(1, 0, 0), at(1, 0, 1), tx), lerp(at(1, 1, 0), at(1, 1, 1), tx)
    f = lerp(lerp(c00, c10, ty), lerp(c01, c11, ty), tz)
    d0 = lerp(lerp(at(0, 0, 1) - at(0, 0, 0), at(0, 1, 1) - at(0, 1, 0), ty),
              lerp(at(1, 0, 1) - at(1, 0, 0), at(1, 1, 1) - at(1, 1, 0), ty), tz)
    d1, d2 = lerp(c10 - c00, c11 - c01, tz), lerp(c01 - c00, c11 - c10, ty)
    g = torch.stack([d0, d1, d2], 1)
    g = g / g.norm(dim=1, keepdim=True).clamp_min(1e-30)
    return torch.where(ok, f, torch.full_like(f, float("inf"))), g


def _pairs(pos, env):
    """Directed touching pairs (i, j) by the FP32 sphere test, sorted by (i, j)."""
    n = pos.shape[0]
    c = 2.01 * float(pos[:, 3].max())
    k = (pos[:, :3].double() / c).floor().long()
    k -= k.min(dim=0).values - 1
    dim = k.max(dim=0).values + 2
    key = ((env * dim[2] + k[:, 2]) * dim[1] + k[:, 1]) * dim[0] + k[:, 0]
    order = key.argsort()
    sk = key[order]
    me = torch.arange(n, device=DEV)
    found = []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            want = key + (dz * dim[1] + dy) * dim[0]
            a, b = torch.searchsorted(sk, want - 1), torch.searchsorted(sk, want + 2)
            for s in range(int((b - a).max())):
                live = a + s < b
                i, j = me[live], order[(a + s)[live]]
                p, q = pos[i], pos[j]
                d = p[:, :3] - q[:, :3]
                d2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
                rs = p[:, 3] + q[:, 3]
                hit = (d2 <= rs * rs) & (i != j)
                found.append(i[hit] * n + j[hit])
    code = torch.cat(found).sort().values
    return code // n, code % n


def _project(s, nn, mu):
    ln = (s * nn).sum(1)
    lnp = ln.clamp_min(0.0)
    t = s - ln[:, None] * nn
    t2 = (t * t).sum(1)
    lim = mu * lnp
    slide = t2 > lim * lim
    sc = torch.where(slide, lim / torch.where(slide, t2, torch.ones_like(t2)).sqrt(), torch.ones_like(t2))
    return lnp[:, None] * nn + sc[:, None] * t


def _qmul(a, b):
    return torch.stack([a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3],
                        a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2],
                        a[0] * b[2] - a[1] * b[3] + a[2] * b[0] + a[3] * b[1],
                        a[0] * b[3] + a[1] * b[2] - a[2] * b[1] + a[3] * b[0]])


def _rollout(sc, steps, twist=None, mu=None):
    """`steps` time steps in float64: (x, v, wrenches (steps, bodies, 6), poses).
    twist: differentiable table of the scoop of environment 0; mu: likewise."""
    P = sc.params
    dt = float(np.float32(P.dt))
    grav = torch.tensor(np.asarray(P.gravity, np.float32).astype(np.float64), device=DEV)
    mu = float(np.float32(P.mu)) if mu is None else mu
    ab = float(np.float32(P.alpha)) / dt
    n = sc.n
    env = torch.zeros(n, device=DEV, dtype=torch.long)
    if sc.offsets is not None:
        env = torch.repeat_interleave(torch.arange(len(sc.bodies), device=DEV),
                                      torch.as_tensor(np.diff(sc.offsets.astype(np.int64)), device=DEV))
    x, v, m = sc.pos[:, :3].double(), sc.vel.double(), sc.mass.double()
    r32, r = sc.pos[:, 3], sc.pos[:, 3].double()
    flat = [(e, k, b) for e, bl in enumerate(sc.bodies) for k, b in enumerate(bl)]
    f64 = lambda a: torch.tensor(np.asarray(a, np.float32).astype(np.float64), device=DEV)   # noqa: E731
    pose = [[f64(b.pos), torch.tensor(_unit_q(b), device=DEV), f64(b.lin_vel), f64(b.ang_vel)] for _, _, b in flat]
    rows = [torch.arange(int(sc.offsets[e]), int(sc.offsets[e + 1]), device=DEV) if sc.offsets is not None
            else torch.arange(n, device=DEV) for e, _, _ in flat]
    wrenches = []
    for step in range(steps):
        for (e, k, b), s in zip(flat, pose):
            tw = sc.twist.get((e, k))
            if twist is not None and (e, k) == (0, TOOL):
                s[2], s[3] = twist[step, :3], twist[step, 3:]
            elif tw is not None and step < tw.shape[0]:
                s[2], s[3] = f64(tw[step, :3]), f64(tw[step, 3:])
            elif tw is not None:
                s[2], s[3] = f64(b.lin_vel), f64(b.ang_vel)
        x32 = x.detach().to(F32)
        pi, pj = _pairs(torch.cat([x32, r32[:, None]], 1), env)
        d = x[pi] - x[pj]
        dist = d.norm(dim=1)
        nn = d / dist[:, None]
        psi = r[pi] + r[pj] - dist
        cnt = torch.bincount(pi, minlength=n).double()
        con = []
        for (e, k, b), s, own in zip(flat, pose, rows):
            y32 = _to_body(b, x32[own], F32, s[0].detach(), s[1].detach())
            idx = own[_sdf(b, y32, F32)[0] <= r32[own]]
            y = _to_body(b, x[idx], F64, s[0], s[1])
            f, g = _sdf(b, y, F64)
            if b.kind == scenes.GRID:      # outside the decision's cell by rounding: no value there
                f = f.nan_to_num(posinf=0.0)
            nb = g @ _quat_R(s[1], F64).T
            xc = x[idx] - f[:, None] * nb
            cnt = cnt + torch.bincount(idx, minlength=n)
            con.append([idx, nb, r[idx] - f, xc, torch.zeros_like(nb)])
        uw = cnt / m
        base = v + dt * grav
        free = [float(b.is_free) for _, _, b in flat]
        vw = [[s[2] + dt * grav * fr, s[3]] for s, fr in zip(pose, free)]
        own = [list(t) for t in vw]
        inv = []
        for (e, k, b), s, c in zip(flat, pose, con):
            if not b.is_free:
                inv.append(0.0)
                continue
            R = _quat_R(s[1], F64)
            a = torch.linalg.cross(c[3] - s[0], c[1]) @ R
            inv.append(c[0].shape[0] * (1.0 / b.mass + (a * a / f64(b.inertia)).sum(1)))
        lam = torch.zeros_like(nn)
        U = base
        w = (1.0 / (uw[pi] + uw[pj]))[:, None]
        for _ in range(P.pja_iters):
            lam = _project(lam - w * (U[pi] - U[pj] - ab * psi[:, None] * nn), nn, mu)
            S = torch.zeros_like(U).index_add(0, pi, lam)
            for q, c in enumerate(con):
                if c[0].numel() == 0:
                    continue
                ub = vw[q][0] + torch.linalg.cross(vw[q][1].expand_as(c[3]), c[3] - pose[q][0])
                wb = (1.0 / (uw[c[0]] + inv[q]))[:, None]
                c[4] = _project(c[4] - wb * (U[c[0]] - ub - ab * c[2][:, None] * c[1]), c[1], mu)
                S = S.index_add(0, c[0], c[4])
            for q, (e, k, b) in enumerate(flat):
                if b.is_free:
                    R = _quat_R(pose[q][1], F64)
                    L = -torch.linalg.cross(con[q][3] - pose[q][0], con[q][4]).sum(0)
                    vw[q] = [own[q][0] - con[q][4].sum(0) / b.mass, own[q][1] + R @ ((R.T @ L) / f64(b.inertia))]
            U = base + S / m[:, None]
        wr = torch.zeros((len(flat), 6), device=DEV, dtype=F64)
        with torch.no_grad():
            for q, c in enumerate(con):
                F = -c[4] / dt
                wr[q, :3], wr[q, 3:] = F.sum(0), torch.linalg.cross(c[3] - pose[q][0], F).sum(0)
        wrenches.append(wr)
        v = U
        x = x + dt * U
        if P.cyclic_z[1] > P.cyclic_z[0]:
            lo = float(np.float32(P.cyclic_z[0]))
            up = float(np.float32(P.cyclic_z[1]) - np.float32(P.cyclic_z[0]))
            x = x + torch.where(x[:, 2] < lo, up, 0.0)[:, None] * torch.tensor([0.0, 0.0, 1.0], device=DEV, dtype=F64)
        for q, s in enumerate(pose):
            V, W = vw[q]
            s[0] = s[0] + dt * V
            a = dt * W
            a2 = (a * a).sum()
            ang = (a2 + 1e-300).sqrt()
            half = torch.where(a2 > 1e-24, torch.sin(0.5 * ang) / ang, 0.5 - a2 / 48.0)
            s[1] = _qmul(torch.cat([torch.cos(0.5 * ang)[None], a * half]), s[1])
            s[1] = s[1] / s[1].norm()
            if flat[q][2].is_free:
                s[2], s[3] = V, W
    return x, v, torch.stack(wrenches), pose, flat


def _pos_vel(sc, x, v):
    return torch.cat([torch.cat([x, sc.pos[:, 3:].double()], 1).reshape(-1), v.reshape(-1)])


def exact(case, seed):
    kind = case["kind"]
    if kind == "bin":
        return None                     # whole numbers
    sc = _scene(case, seed)
    if kind == "views":
        return _views(case, sc)
    if kind == "grad":
        steps = case["steps"]
        tw = torch.tensor(sc.twist[(0, TOOL)][:steps].astype(np.float64), device=DEV, requires_grad=True)
        mu = torch.tensor(float(np.float32(sc.params.mu)), device=DEV, dtype=F64, requires_grad=True)
        x, v, _, pose, _ = _rollout(sc, steps, twist=tw, mu=mu)
        gp, gv, gb = [t.double() for t in _seeds(sc, case)]
        L = (gp * x).sum() + (gv * v).sum() + (gb * torch.cat([pose[TOOL][0], pose[TOOL][1]])).sum()
        L.backward()
        return [_pos_vel(sc, x.detach(), v.detach()), tw.grad, mu.grad.reshape(1)]
    with torch.no_grad():
        x, v, wr, _, flat = _rollout(sc, case.get("steps", 1))
        if kind == "io":
            return [_pos_vel(sc, x, v).cpu()]
        mb = max(8, max(len(b) for b in sc.bodies))
        full = torch.zeros((wr.shape[0], len(sc.bodies) * mb, 6), device=DEV, dtype=F64)
        for q, (e, k, _) in enumerate(flat):
            full[:, e * mb + k] = wr[:, q]
        return [_pos_vel(sc, x, v), full]


def _views(case, sc):
    """Height and depth images in 64 bits (spheres by brute force over the pixels)."""
    foot = 2.0 * sc.bodies[0][0].shape[0]
    sky, ego = _cameras(case, foot)
    f = lambda a: float(np.float32(a))                                   # noqa: E731
    x, r = sc.pos[:, :3].double(), sc.pos[:, 3].double()
    px = f(-0.5 * foot) + (torch.arange(sky.width, device=DEV, dtype=F64) + 0.5) * (f(foot) / sky.width)
    py = f(-0.25 * foot) + (torch.arange(sky.height, device=DEV, dtype=F64) + 0.5) * (f(0.5 * foot) / sky.height)
    height = torch.zeros((sky.height, sky.width), device=DEV, dtype=F64)
    for row in range(sky.height):
        near = ((x[:, 1] - py[row]).abs() <= r).nonzero()[:, 0]
        if near.numel() == 0:
            continue
        d2 = (x[near, 0][None] - px[:, None]) ** 2 + ((x[near, 1] - py[row]) ** 2)[None]
        up = r[near][None] ** 2 - d2
        z = torch.where(up >= 0, x[near, 2][None] + up.clamp_min(0.0).sqrt(), -1e30).max(dim=1).values
        height[row] = torch.where(z > -1e29, z, 0.0)
    W, H = ego.width, ego.height
    foc = 0.5 * H / math.tan(0.5 * f(ego.fov_y))
    ax = (torch.arange(W, device=DEV, dtype=F64) + 0.5 - 0.5 * W) / foc
    ay = (torch.arange(H, device=DEV, dtype=F64) + 0.5 - 0.5 * H) / foc
    ray = torch.stack([ax[None, :].expand(H, W), ay[:, None].expand(H, W), torch.ones((H, W), device=DEV, dtype=F64)], -1)
    ray = ray / ray.norm(dim=-1, keepdim=True)
    ray = ray.reshape(-1, 3) @ _quat_R(torch.tensor([f(q) for q in ego.quat], device=DEV, dtype=F64), F64).T
    o = torch.tensor([f(q) for q in ego.pos], device=DEV, dtype=F64)
    near_c, far = f(ego.near), f(ego.far)
    oc = x - o
    cc = (oc * oc).sum(1) - r * r
    best = torch.full((H * W,), float("inf"), device=DEV, dtype=F64)
    for s in range(0, sc.n, 1 << 15):
        b = ray @ oc[s:s + (1 << 15)].T
        disc = b * b - cc[s:s + (1 << 15)]
        t = b - disc.clamp_min(0.0).sqrt()
        t = torch.where((disc >= 0) & (t >= near_c) & (t <= far), t, float("inf"))
        best = torch.minimum(best, t.min(dim=1).values)
    t = torch.full_like(best, near_c)
    live = torch.ones_like(best, dtype=torch.bool)
    eps = f(ego.march_eps)
    for _ in range(ego.march_steps):
        p = o + t[:, None] * ray
        d = torch.stack([_sdf(b, _to_body(b, p, F64), F64)[0] for b in sc.bodies[0]]).min(dim=0).values
        hit = live & (d < eps)
        best = torch.where(hit, torch.minimum(best, t), best)
        t = torch.where(live & ~hit, t + d, t)
        live &= ~hit & (t <= far)
    return [height, torch.where(best <= far, best, far).reshape(H, W)]
