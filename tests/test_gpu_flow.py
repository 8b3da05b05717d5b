"""The dataflow sweeps (launch-shape sets with GG_TUNE_FLOW: every sweep in one launch, the
contact records on chip, partners' estimates exchanged as tagged values) against the
per-launch sweeps: bit-identical positions, velocities, wrenches and impulses at the sizes
where tiles, blocks and ranges end, with free bodies, several particle ranges, records
that do not fit on chip, lists cut by the contact capacity, and bounded waits."""
import dataclasses
import os
import subprocess
import sys
import time

import numpy as np
import pytest

from gpu_helpers import need_gpu
from paper_2306_01369_gb300 import scenes as S

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def gg():
    need_gpu()
    from paper_2306_01369_gb300 import gg as g
    return g


def flow_sets(gg):
    return [k for k in range(1, gg.load().gg_tuning_count() + 1) if "flow" in gg.tuning_flags(k)]


def squeezed(n, seed=11, factor=0.95, shuffle=False, **params):
    """A box of overlapping spheres (about three contacts each)."""
    sc = S.settle_box(n=max(n, 64), seed=seed)
    pr = sc.pos_r[:n].copy()
    pr[:, :3] *= np.float32(factor)
    if shuffle:
        pr = pr[np.argsort(S.uniform(seed, n), kind="stable")]
    return S.Scene("squeezed", np.ascontiguousarray(pr), np.zeros((n, 3), np.float32), S.sphere_mass(pr[:, 3]), sc.bodies,
                   dataclasses.replace(sc.params, **params), 10)


def outputs(gg, sc, tuning, steps, check=True, **kw):
    sim = gg.Sim.from_scene(sc, tuning=tuning, wrench_history=steps, **kw)
    sim.step(steps)
    out = [sim.read(f, check=check) for f in ("POS", "VEL", "BODY_STATE", "BODY_WRENCH", "CONTACT_IMPULSE",
                                              "BODY_CONTACT_IMPULSE")]
    out.append(sim.read("CONTACTS", np.uint32, check=check))
    flags = sim.stats()["status_flags"]
    sim.close()
    return out, flags


def same(gg, sc, steps=3, ref=7, sets=None, **kw):
    want, wf = outputs(gg, sc, ref, steps, **kw)
    for k in sets or flow_sets(gg):
        got, gf = outputs(gg, sc, k, steps, **kw)
        assert gf == wf
        for a, b in zip(got, want):
            assert np.array_equal(a, b), (sc.name, k)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 1000, 4096])
def test_sizes_around_a_tile(gg, n):
    same(gg, squeezed(n))


@pytest.mark.parametrize("iters", [1, 2, 3])
def test_few_iterations(gg, iters):
    same(gg, squeezed(2000, pja_iters=iters))


def test_ids_in_no_spatial_order(gg):
    same(gg, squeezed(4000, shuffle=True))


def test_free_and_moving_bodies(gg):
    same(gg, S.excavation(n=6000, n_steps=20), steps=12, sets=[flow_sets(gg)[-1]])


def test_more_free_bodies_than_the_launch_takes(gg):
    """Nine free bodies: the set runs the split launches."""
    sc = squeezed(600)
    top = float(sc.pos_r[:, 2].max())
    sc.bodies = sc.bodies + [S.Body(kind=S.BOX, shape=(0.004,) * 3, pos=(0.03 + 0.015 * k, 0.05, top + 0.006), is_free=1,
                                    mass=0.01, inertia=(1e-6,) * 3) for k in range(7)]
    sc.bodies += [S.Body(kind=S.BOX, shape=(0.004,) * 3, pos=(0.03, 0.08 + 0.02 * k, top + 0.006), is_free=1, mass=0.01,
                         inertia=(1e-6,) * 3) for k in range(2)]
    same(gg, sc, max_bodies=16)


def test_several_particle_ranges(gg):
    """A batch of more spheres than one range takes, its environments uneven."""
    b = S.batched_beds(n_envs=14, n_steps=4, n_min=15000, n_max=40000)
    assert b.n > 300000
    for e in range(14):
        a, z = int(b.env_offsets[e]), int(b.env_offsets[e + 1])
        b.pos_r[a:z, 1:3] *= np.float32(0.97)
    same(gg, b, steps=2, sets=[flow_sets(gg)[1]])


def test_records_beyond_the_shared_memory(gg):
    """A crowded cloud in random order: about ten partners a sphere, most of them other
    blocks' (their records do not all fit on chip)."""
    n = 90000
    pr, vel = S.random_cloud(n, 5, box=0.135, vel_scale=0.05)
    sc = S.Scene("cloud", pr, vel, S.sphere_mass(pr[:, 3]), [S.Body(kind=S.PLANE, pos=(0.0, 0.0, -0.01))],
                 S.Params(dt=1e-5, max_contacts=32), 4)
    same(gg, sc, steps=1, sets=[flow_sets(gg)[1]])


def test_lists_cut_by_the_capacity(gg):
    """One-sided lists (a sphere with more partners than its capacity): the plain sweeps
    run, as bit-identical as before."""
    sc = squeezed(3000, factor=0.9, max_contacts=2)
    want, wf = outputs(gg, sc, 7, 1, check=False)
    assert wf & 1
    for k in flow_sets(gg):
        if "half" in gg.tuning_flags(k):
            continue      # (which partners a half-stencil pass loses depends on its atomics)
        got, gf = outputs(gg, sc, k, 1, check=False)
        assert gf == wf
        for a, b in zip(got, want):
            assert np.array_equal(a, b), k


def test_waits_run_out_and_report(gg):
    """A phantom participant (tags that nothing writes): every wait runs out within its
    bound, the step reports it, and the context stays usable."""
    sc = squeezed(3000)
    k = flow_sets(gg)[0]
    sim = gg.Sim(sc.pos_r, sc.vel, sc.mass, sc.params, tuning=k, barrier_test_phantoms=1, wait_limit_us=20000)
    sim.set_bodies(sc.bodies)
    t0 = time.perf_counter()
    sim.step(1)
    with pytest.raises(gg.GGError) as e:
        sim.sync()
    assert e.value.status == gg.ERR_DEVICE_TIMEOUT
    assert time.perf_counter() - t0 < 5.0
    sim.close()
    same(gg, sc, steps=2, sets=[k])


def test_going_back_to_a_checkpoint(gg):
    """Steps taken again from a restored state (the same step indices) equal the first
    time's: no value published then is taken for one of now."""
    sc = squeezed(3000)
    sim = gg.Sim.from_scene(sc, tuning=flow_sets(gg)[1])
    sim.step(2)
    blob = sim.state()
    sim.step(3)
    first = [sim.pos(), sim.vel()]
    for _ in range(2):
        sim.set_state(blob)
        sim.step(3)
        assert np.array_equal(first[0], sim.pos()) and np.array_equal(first[1], sim.vel())
    sim.close()


def test_spheres_larger_than_the_cells(gg):
    """Radii raised after creation above half a cell: a full-stencil search then lists pairs
    for one of their spheres only (the larger one walks cells the smaller one does not), and
    the plain sweeps run, as bit-identical as before."""
    sc = squeezed(3000, max_contacts=32)
    big = sc.pos_r.copy()
    big[::7, 3] *= np.float32(1.7)
    for k in flow_sets(gg):
        ref = 21 if "half" in gg.tuning_flags(k) else 7
        got = []
        for tuning in (ref, k):
            sim = gg.Sim.from_scene(sc, tuning=tuning)
            sim.set_particles(big)
            sim.step(1)
            c = sim.contacts()
            own = np.repeat(np.arange(sc.n), np.diff(c["pp_off"].astype(np.int64)))
            pairs = set(zip(own.tolist(), c["pp_j"].tolist()))
            if "half" not in gg.tuning_flags(k):
                assert any((j, i) not in pairs for i, j in pairs)
            got.append([sim.read(f) for f in ("POS", "VEL", "BODY_WRENCH", "CONTACT_IMPULSE")])
            assert sim.stats()["status_flags"] == 0
            sim.close()
        for a, b in zip(*got):
            assert np.array_equal(a, b), k


def pressed_boxes(n=3000, v=(0.0, 0.0, 0.0)):
    """Two free boxes in use: one sunk into the top of a squeezed bed, a plate pressing on its
    corners, one with corners in a wall of the container and its side among the spheres."""
    sc = squeezed(n)
    mid = float(np.median(sc.pos_r[:, 2]))
    free = dict(is_free=1, mass=0.05, inertia=(4e-6,) * 3, lin_vel=v)
    sc.bodies = sc.bodies + [
        S.Body(kind=S.BOX, shape=(0.02,) * 3, pos=(0.1, 0.1, 0.115), **free),
        S.Body(kind=S.BOX, shape=(0.01, 0.02, 0.01), pos=(0.0095, 0.1, mid), **free),
        S.Body(kind=S.BOX, shape=(0.05, 0.05, 0.01), pos=(0.1, 0.1, 0.1445), lin_vel=(0.02, 0.0, -0.1))]
    return sc


def test_free_bodies_in_contact(gg):
    """Spheres, a wall and a moving plate act on two free boxes: what the boxes' blocks and
    the spheres' exchange in every sweep, for every set."""
    sc = pressed_boxes()
    sim = gg.Sim.from_scene(sc, tuning=flow_sets(gg)[0])
    sim.step(1)
    b = sim.contacts()["bc_b"]
    assert all((b == k).sum() >= 5 for k in (1, 2))           # spheres on both boxes
    assert np.abs(sim.wrench()[-1, 3]).max() > 0              # and a box's corners on the plate
    sim.close()
    same(gg, sc, steps=4)
    sc.params = dataclasses.replace(sc.params, pja_iters=3)
    same(gg, sc, steps=2)


RESTART = r"""
import dataclasses, sys
import numpy as np
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
from paper_2306_01369_gb300 import gg
from test_gpu_flow import flow_sets, pressed_boxes, same
sc = pressed_boxes()
sc.params = dataclasses.replace(sc.params, pja_iters=3, gravity=(0.0, 0.0, 0.0))
later = pressed_boxes(v=(0.3, -0.2, 0.4)).bodies
apart = sc.pos_r.copy()
apart[:, :3] *= np.float32(1.5)
for k in flow_sets(gg):
    same(gg, pressed_boxes(), steps=30, sets=[k])     # the tags start over every five steps
    out = []
    for idle in (0, 20):
        sim = gg.Sim.from_scene(sc, tuning=k)
        if idle:        # tags 1 and 2 published, then no free body until the tags have started over
            sim.step(1)
            sim.set_bodies([])
            sim.set_particles(apart, np.zeros((sc.n, 3), np.float32))
            sim.step(idle)
            assert sim.stats()["n_pp"] == 0
        sim.set_bodies(later)
        sim.set_particles(sc.pos_r, sc.vel)
        sim.step(1)
        out.append([sim.read(f) for f in ("POS", "VEL", "BODY_STATE", "BODY_WRENCH")])
        sim.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out)), k
print("equal")
"""


def test_tags_that_start_over():
    """The checked build starts its tags over after a hundred: runs across that equal the
    split sweeps, and a free body that was out of use meanwhile is not met by the twist
    published under the same tag before."""
    need_gpu()
    from paper_2306_01369_gb300 import _build
    _build.build(debug=True)
    r = subprocess.run([sys.executable, "-c", RESTART, ROOT], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, GG_DEBUG="1"))
    assert r.returncode == 0 and "equal" in r.stdout, r.stderr[-3000:]


@pytest.mark.parametrize("n", [700, 3000, 20000])
def test_crowded_clouds_on_little_scratch(gg, n):
    """The scratch is sized by what the capacities allow: none for records where a block's
    share fits on chip whatever the contacts, some at 20,000 spheres."""
    pr, vel = S.random_cloud(n, 6, box=0.135 * (n / 90000) ** (1 / 3), vel_scale=0.05)
    sc = S.Scene("cloud", pr, vel, S.sphere_mass(pr[:, 3]), [S.Body(kind=S.PLANE, pos=(0.0, 0.0, 0.0))],
                 S.Params(dt=1e-5, max_contacts=32), 4)
    same(gg, sc, steps=1)


def test_memory_of_small_simulations(gg):
    """A simulation whose set never runs the dataflow sweeps holds none of their scratch, and
    a small one little (152 blocks' worth would be 87 MB): 32 bytes a sphere, and at 4,096
    spheres 16 bytes for each of 131 blocks' at most 1,279 + 656 contacts with bodies, a few
    MB, with cudaMalloc's 2 MB granularity for each of the seven buffers."""
    torch = need_gpu()
    sc = squeezed(4096)

    def held(**kw):
        before = torch.cuda.mem_get_info()[0]
        sims = [gg.Sim.from_scene(sc, **kw) for _ in range(8)]
        after = torch.cuda.mem_get_info()[0]
        for s in sims:
            s.close()
        return (before - after) / 8e6
    gg.Sim.from_scene(sc).close()                 # (the context's own allocations)
    plain, flow = held(tuning=7), held(tuning=flow_sets(gg)[1])
    lit = dataclasses.replace(sc.params, pja_weight=1)
    sc.params, params = lit, sc.params
    off = held(tuning=flow_sets(gg)[1])
    sc.params = params
    assert flow - plain < 22 and off - plain < 2, (plain, flow, off)


def test_two_simulations_in_two_streams(gg):
    """Small simulations claim the blocks they can use, so two run side by side: each as on
    its own, the waits of neither held up by the other."""
    torch = need_gpu()
    k = flow_sets(gg)[-1]
    scenes = [squeezed(4096), squeezed(3000, seed=12)]
    want = []
    for sc in scenes:
        sim = gg.Sim.from_scene(sc, tuning=k)
        sim.step(60)
        want.append((sim.pos(), sim.vel()))
        sim.close()
    sims = [gg.Sim.from_scene(sc, tuning=k) for sc in scenes]
    streams = [torch.cuda.Stream() for _ in sims]
    torch.cuda.synchronize()
    for _ in range(20):
        for sim, st in zip(sims, streams):
            sim.step(3, stream=st.cuda_stream)
    torch.cuda.synchronize()
    for sim, (x, v) in zip(sims, want):
        assert np.array_equal(sim.pos(), x) and np.array_equal(sim.vel(), v)
        sim.close()


def test_lists_that_outgrow_the_chip(gg):
    """One bed too large for the chip and a small one beside it: the large one's range gets
    the plain sweeps in the same launch, bit-identical, wrenches too."""
    big, small = squeezed_column(420000), squeezed_column(20000)
    for scenes_ in ([big], [small, big, small]):
        pr = np.concatenate([s.pos_r for s in scenes_])
        offs = np.concatenate([[0], np.cumsum([s.n for s in scenes_])])
        out = []
        for tuning in [7] + flow_sets(gg):
            sim = gg.Sim(pr, np.zeros((len(pr), 3), np.float32), S.sphere_mass(pr[:, 3]), big.params,
                         env_offsets=offs, tuning=tuning)
            for e, s in enumerate(scenes_):
                sim.set_bodies(s.bodies, e)
            sim.step(2)
            out.append([sim.read(f) for f in ("POS", "VEL", "BODY_WRENCH", "CONTACT_IMPULSE")])
            assert sim.stats()["n_pp"] > 3 * 420000 and sim.stats()["status_flags"] == 0
            sim.close()
            assert all(np.array_equal(a, b) for a, b in zip(out[0], out[-1])), tuning


def squeezed_column(n):
    """A column of overlapping spheres, 3.4 contacts each: 3.9 units of cost a sphere, of which
    the chip takes about 1.26 million."""
    sc = S.column_collapse(n=n)
    sc.pos_r[:, :3] *= np.float32(0.88)
    return sc


def test_leaving_a_set_that_no_longer_fits(gg):
    """Tuned while nothing touches, packed afterwards: the dataflow sweeps report that the
    bed does not fit, and the simulation goes over to a split set with the same results."""
    sc = squeezed_column(420000)
    loose = S.column_collapse(n=420000)
    sim = gg.Sim.from_scene(loose)
    sim.step(1)
    sim.sync()
    chosen = gg.load().gg_tuning_selected(sim.h)
    assert "flow" in gg.tuning_flags(chosen)
    ref = gg.Sim.from_scene(loose, tuning=7)
    ref.step(1)
    for s in (sim, ref):
        s.set_particles(sc.pos_r, sc.vel)
        for _ in range(3):
            s.step(1)
            s.sync()
    assert "flow" not in gg.tuning_flags(gg.load().gg_tuning_selected(sim.h))
    for f in ("POS", "VEL", "BODY_WRENCH"):
        assert np.array_equal(sim.read(f), ref.read(f)), f
    again = gg.load().gg_tuning_selected(sim.h)
    sim.step(2)
    ref.step(2)
    assert gg.load().gg_tuning_selected(sim.h) == again and np.array_equal(sim.pos(), ref.pos())
    sim.close()
    ref.close()


def test_free_bodies_with_lists_cut_by_the_capacity(gg):
    """The plain sweeps with free bodies: their updates between the grid barriers."""
    sc = pressed_boxes()
    sc.params = dataclasses.replace(sc.params, max_contacts=2)
    want, wf = outputs(gg, sc, 7, 3, check=False)
    assert wf & 1
    for k in flow_sets(gg):
        if "half" in gg.tuning_flags(k):
            continue
        got, gf = outputs(gg, sc, k, 3, check=False)
        assert gf == wf
        for a, b in zip(got, want):
            assert np.array_equal(a, b), k


def test_free_bodies_in_a_small_batch(gg):
    """Several environments in one range, free bodies in each: the dataflow launch takes them."""
    a, b = pressed_boxes(), pressed_boxes(2500, v=(0.1, 0.0, -0.1))
    pr = np.concatenate([a.pos_r, b.pos_r])
    want = None
    for tuning in [7] + flow_sets(gg):
        sim = gg.Sim(pr, np.zeros((len(pr), 3), np.float32), S.sphere_mass(pr[:, 3]), a.params,
                     env_offsets=[0, a.n, a.n + b.n], tuning=tuning, max_free_bodies=4)
        for e, s in enumerate((a, b)):
            sim.set_bodies(s.bodies, e)
        sim.step(3)
        got = [sim.read(f) for f in ("POS", "VEL", "BODY_STATE", "BODY_WRENCH")]
        sim.close()
        want = want or got
        assert all(np.array_equal(x, y) for x, y in zip(got, want)), tuning
