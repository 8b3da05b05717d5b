"""Both sides of the lines at which a launch changes its shape: the depth camera's warp per
body, the half-stencil search's thread per row, the reverse pass's kept graphs and lanes."""
import numpy as np
import pytest

from gpu_helpers import F32, need_gpu
from paper_2306_01369_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gg():
    need_gpu()
    from paper_2306_01369_gb300 import gg
    return gg


@pytest.mark.parametrize("nb,w,h", [(1, 1, 1), (2, 31, 1), (4, 33, 7), (5, 40, 30), (32, 36, 36)])
def test_traced_bodies(gg, orc, nb, w, h):
    """Bodies alone: the tracing is the oracle's FP32 one to the bit, whatever the split."""
    rng = np.random.default_rng(nb)
    bodies = [S.Body(kind=S.PLANE, pos=(0.0, 0.0, -0.3))]
    for k in range(1, nb):
        pos, rv = rng.uniform(-0.3, 0.3, 3), tuple(rng.uniform(-1.0, 1.0, 3))
        bodies.append(S.scoop_body(1.0, pos, rv) if k % 2 else
                      S.Body(kind=S.BOX, shape=tuple(rng.uniform(0.02, 0.06, 3)), pos=tuple(pos),
                             quat=S._quat_from_rotvec(rv)))
    cam = S.Camera(kind=S.DEPTH_CAMERA, width=w, height=h, pos=(0.0, 0.0, 0.8), quat=S._quat_from_rotvec((np.pi, 0.0, 0.0)),
                   fov_y=0.9, near=0.01, far=1.5, march_steps=50, march_eps=1e-4)
    sim = gg.Sim(np.zeros((0, 4), F32), np.zeros((0, 3), F32), np.zeros(0, F32), S.Params(), max_bodies=nb)
    sim.set_bodies(bodies)
    got = sim.render(cam)
    sim.close()
    assert np.array_equal(got, orc.render(cam, np.zeros((0, 3)), np.zeros(0), bodies).astype(F32))


@pytest.mark.parametrize("n", [1, 127, 129, 262144, 262145])
def test_half_stencil_rows(gg, n):
    """Up to 262,144 spheres a thread per row, above that a thread per sphere: the same
    contacts and state as the full-stencil search, with small (shared) and large buckets."""
    side = round(n ** (1 / 3)) + 1
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    rng = np.random.default_rng(n)
    pr = np.empty((n, 4), F32)
    pr[:, :3] = 0.0195 * (g - side / 2) + rng.uniform(-1e-3, 1e-3, (n, 3))
    pr[:, 3] = 0.01
    pr = np.ascontiguousarray(pr[rng.permutation(n)])
    sets = [k for k in range(1, gg.load().gg_tuning_count() + 1) if "half" in gg.tuning_flags(k)]
    sets = [next(k for k in sets if ("lists" in gg.tuning_flags(k)) == lists) for lists in
            {"lists" in gg.tuning_flags(k) for k in sets}]
    for hf in (1, 4):
        want = None
        for tuning in [7] + sets:
            sim = gg.Sim(pr, None, S.sphere_mass(pr[:, 3]), S.Params(dt=1e-4, pja_iters=3, max_contacts=24), tuning=tuning,
                         hash_factor=hf)
            sim.step(2)
            got = [sim.read("POS"), sim.read("VEL"), sim.read("CONTACTS", np.uint32)]
            sim.close()
            want = want or got
            assert all(np.array_equal(a, b) for a, b in zip(got, want)), (tuning, hf)


def test_reverse_passes_of_changing_length(gg):
    """Reverse passes of one simulation, longer, shorter and of the first length again:
    each gives what a simulation of its own gives."""
    sc = S.diff_scene(n=512, n_steps=6)
    seed = np.random.default_rng(3).normal(size=(sc.n, 3)).astype(F32)

    def fresh():
        sim = gg.Sim(sc.pos_r, sc.vel, sc.mass, sc.params)
        sim.set_bodies(sc.bodies)
        sim.set_trajectory(1, sc.twist[1].astype(F32))
        return sim

    def run(sim, state, steps):
        sim.tape_reserve(steps, 2)
        sim.set_state(state)
        sim.step_taped(1, steps)
        return sim.backward(seed)

    kept = fresh()
    state = kept.state()
    for steps in (4, 6, 3, 4):
        got = run(kept, state, steps)
        one = fresh()
        want = run(one, state, steps)
        one.close()
        assert np.array_equal(got[0], want[0]) and got[1] == want[1]
    kept.close()


@pytest.mark.parametrize("n", [65, 8192, 8193, 65536, 65537])
def test_reverse_pass_lanes(gg, n):
    """The reversed sweeps take 8, 4 or 2 lanes a particle by the particle count.  With the
    scene's ids reversed every sum falls to other lanes and blocks, and the gradient is the
    same.  float32 sums of at most 65,537 terms, in a tree of at most 512 strided terms and
    nine levels: 1e-4 of their size."""
    side = int(np.ceil(np.sqrt(n)))
    g = np.stack(np.meshgrid(np.arange(side), np.arange(side), indexing="ij"), -1).reshape(-1, 2)[:n]
    pr = np.empty((n, 4), F32)
    pr[:, :2] = 0.0198 * (g - side // 2)
    pr[:, 2] = 0.0099
    pr[:, 3] = 0.01
    seed = np.zeros((n, 3), F32)
    seed[:, 0], seed[:, 2] = 1.0, np.where(np.arange(n) % 3 == 0, 1.0, 0.5)
    got = []
    for order in (np.arange(n), np.arange(n)[::-1].copy()):
        sim = gg.Sim(np.ascontiguousarray(pr[order]), None, S.sphere_mass(pr[:, 3]),
                     S.Params(dt=1e-4, mu=0.5, pja_iters=4, max_contacts=8))
        sim.set_bodies([S.Body(kind=S.PLANE, lin_vel=(0.05, 0.0, 0.1))])
        sim.set_trajectory(0, np.tile(np.array([[0.05, 0.0, 0.1, 0.0, 0.0, 0.0]], F32), (2, 1)))
        sim.tape_reserve(2, 2)
        sim.step_taped(0, 2)
        g_tw, g_mu = sim.backward(np.ascontiguousarray(seed[order]))
        sim.close()
        got.append((np.asarray(g_tw, np.float64), float(g_mu)))
    scale = np.abs(got[0][0]).max()
    assert scale > 0 and np.isfinite(got[0][0]).all()
    assert np.abs(got[0][0][:, :3] - got[1][0][:, :3]).max() <= 1e-4 * scale


@pytest.mark.parametrize("nb,w,h", [(1, 40, 30), (2, 400, 250), (2, 400, 251), (3, 317, 316), (4, 800, 500), (4, 800, 501),
                                    (32, 400, 429), (32, 400, 430)])
def test_traced_images_of_either_form(gg, orc, nb, w, h):
    """Both sides of the pixel counts up to which a ray's bodies get a warp each: the oracle's
    tracing to the bit, and with spheres in front the nearer of the two depths."""
    rng = np.random.default_rng(nb)
    bodies = [S.Body(kind=S.PLANE, pos=(0.0, 0.0, -0.3))]
    for k in range(1, nb):
        pos, rv = rng.uniform(-0.3, 0.3, 3), tuple(rng.uniform(-1.0, 1.0, 3))
        bodies.append(S.Body(kind=S.BOX, shape=tuple(rng.uniform(0.02, 0.06, 3)), pos=tuple(pos),
                             quat=S._quat_from_rotvec(rv)))
    cam = S.Camera(kind=S.DEPTH_CAMERA, width=w, height=h, pos=(0.0, 0.0, 0.8), quat=S._quat_from_rotvec((np.pi, 0.0, 0.0)),
                   fov_y=0.9, near=0.01, far=1.5, march_steps=24, march_eps=1e-4)
    pr = np.concatenate([rng.uniform(-0.3, 0.3, (200, 3)), rng.uniform(0.005, 0.03, (200, 1))], 1).astype(F32)
    out = []
    for p, nbodies in ((pr[:0], nb), (pr, 0), (pr, nb)):
        sim = gg.Sim(p, np.zeros((len(p), 3), F32), S.sphere_mass(p[:, 3]), S.Params(), max_bodies=nb)
        sim.set_bodies(bodies[:nbodies])
        out.append(sim.render(cam))
        sim.close()
    assert np.array_equal(out[0], orc.render(cam, np.zeros((0, 3)), np.zeros(0), bodies).astype(F32))
    assert np.array_equal(out[2], np.minimum(out[0], out[1]))
    assert (out[1] < out[0]).any() and (out[0] < out[1]).any()


@pytest.mark.parametrize("n", [700000, 700001])
def test_half_stencil_rows_at_the_line(gg, n):
    """The same on both sides of the count up to which the rows get a thread each."""
    test_half_stencil_rows(gg, n)


def test_one_reservation_other_lengths_and_tools(gg):
    """Reverse passes under one reservation, of other lengths and with another tool: the kept
    graphs are made anew where they must be, and each pass gives what a simulation of its own
    gives."""
    sc = S.diff_scene(n=512, n_steps=6)
    seed = np.random.default_rng(4).normal(size=(sc.n, 3)).astype(F32)
    pr = sc.pos_r.copy()      # squeezed, on the container's floor: spheres on each other and on both bodies
    pr[:, :3] = (pr[:, :3] - pr[:, :3].mean(0)) * np.float32(0.72) + pr[:, :3].mean(0)
    pr[:, 2] -= (pr[:, 2] - np.float32(0.9) * pr[:, 3]).min()

    def fresh():
        sim = gg.Sim(pr, None, sc.mass, S.Params(dt=1e-5, mu=0.5, pja_iters=20))
        sim.set_bodies(sc.bodies)
        sim.set_trajectory(1, sc.twist[1].astype(F32))
        sim.tape_reserve(6, 2)
        return sim

    def run(sim, state, tool, steps):
        sim.set_state(state)
        sim.step_taped(tool, steps)
        return sim.backward(seed)

    kept = fresh()
    state = kept.state()
    for tool, steps in ((1, 4), (1, 6), (1, 6), (0, 6), (0, 3), (1, 3), (1, 4)):
        got = run(kept, state, tool, steps)
        one = fresh()
        want = run(one, state, tool, steps)
        one.close()
        assert np.array_equal(got[0], want[0]) and got[1] == want[1], (tool, steps)
        assert np.abs(got[0]).max() > 0
    kept.close()


@pytest.mark.parametrize("n", [4000, 20000, 70000])
def test_reverse_pass_lanes_against_eight(gg, n):
    """8, 4 and 2 lanes a particle (by the particle count) on the same contacts: a squeezed bed
    of 512 spheres with the scoop, filled up with spheres that touch nothing, against the bed
    alone, whose 8-lane gradients the oracle's tests pin.  Same terms, summed in another order:
    at most 512 particles x 20 sweeps of float32 sums with carried errors, 1e-4 of the largest
    component of each kind (forces, torques, mu)."""
    sc = S.diff_scene(n=512, n_steps=4)
    rng = np.random.default_rng(9)
    pr = sc.pos_r[:512].copy()
    pr[:, :3] = (pr[:, :3] - pr[:, :3].mean(0)) * np.float32(0.6) + pr[:, :3].mean(0)
    k = np.arange(n - 512)
    fill = np.empty((n - 512, 4), F32)
    fill[:, :3] = 0.005 * np.stack([k % 4 - 1.5, k // 4 % 4 - 1.5, k // 16 + 200], -1)   # a tower over the container
    fill[:, 3] = 0.002
    seed = rng.normal(size=(512, 3)).astype(F32)
    out = []
    for extra in (0, n - 512):
        x = np.concatenate([pr, fill[:extra]])
        sim = gg.Sim(x, None, S.sphere_mass(x[:, 3]), S.Params(dt=1e-5, mu=0.5, pja_iters=20, max_contacts=24))
        sim.set_bodies(sc.bodies)
        sim.set_trajectory(1, sc.twist[1].astype(F32))
        sim.tape_reserve(3, 3)
        sim.step_taped(1, 3)
        counts = np.diff(sim.contacts()["pp_off"].astype(np.int64))
        assert counts[:512].max() > 8 and not counts[512:].any()
        tw, mu = sim.backward(np.concatenate([seed, np.zeros((extra, 3), F32)]))
        sim.close()
        out.append((np.asarray(tw, np.float64), float(mu)))
    (a, ma), (b, mb) = out
    for k in (slice(0, 3), slice(3, 6)):
        assert np.abs(a[:, k]).max() > 0
        assert np.abs(a[:, k] - b[:, k]).max() <= 1e-4 * np.abs(a[:, k]).max()
    assert ma != 0 and abs(ma - mb) <= 1e-4 * abs(ma)
