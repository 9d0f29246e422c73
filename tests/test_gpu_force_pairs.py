"""Large blocks by unordered pairs (csrc/force_sym.cuh) against the FP64 oracle and the one-sided kernel."""
import numpy as np
import pytest

import oracle
from synthetic import active_subset, plummer_sphere
from tests.gpu_common import EPS2, check_force, errors, gpu_force, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


def _sim(m, x, v, eps2, mode, **kw):
    from paper_astro_ph_0702058_gb300 import Simulation
    return Simulation(m, x, v, eps2, mode=mode, **kw)


def _masses(n, seed):
    w = np.random.default_rng(seed).uniform(0.1, 10.0, n)
    return w / w.sum()


def _check(mode, m, x, v, eps2, act, got, st, what):
    assert st["last_i_per_thread"] == 4, st  # the pairs took it
    rows = np.unique(np.concatenate([np.arange(130), np.linspace(0, len(act) - 1, 400).astype(int),
                                     np.arange(len(act) - 130, len(act))]))
    ref = oracle.force(m, x, v, eps2, act[rows])
    assert all(np.all(np.isfinite(g)) for g in got)
    check_force(mode, m, x, v, eps2, act[rows], tuple(g[rows] for g in got), ref, what)


# one-warp CTAs up to 32768 rows, four-warp ones above; one and several tiles per superblock; a last superblock
# of one row, of one chunk and of a part of a chunk
@pytest.mark.parametrize("mode", ["plain", "comp"])
@pytest.mark.parametrize("n,eps2", [(8192, EPS2), (8193, EPS2), (16384, 0.0), (16385, EPS2), (32768, EPS2),
                                    (33000, 0.0), (65536, EPS2), (70001, EPS2)])
def test_all_particles(torch, mode, n, eps2):
    m, x, v = plummer_sphere(n, 3)
    m = _masses(n, 3)
    with _sim(m, x, v, eps2, mode) as sim:  # (its set-up takes the pairs of the whole stream)
        st0 = sim.stats()
        assert st0["last_i_per_thread"] == 4, st0
        s = {k: np.zeros((n, 3)) for k in ("a", "k")}
        sim.get_state(**s)
        sim.predict(0.0)
        act = np.random.default_rng(1).permutation(n).astype(np.int32)  # any order of the list
        got = gpu_force(sim, act)
        st = sim.stats()
        assert np.array_equal(got[0], gpu_force(sim, act)[0])  # repeats bit for bit
    if n >= 16384:
        _check(mode, m, x, v, eps2, act, got, st, f"pairs n={n}")
    every = np.arange(n, dtype=np.int32)
    _check(mode, m, x, v, eps2, every, (s["a"], s["k"], got[2][np.argsort(act)]), st0, f"set-up n={n}")


# blocks of a quarter of the particles on, the others outside (one, a part of a tile, many tiles)
@pytest.mark.parametrize("mode", ["plain", "comp"])
@pytest.mark.parametrize("n,n_act", [(20001, 20000), (20500, 20001), (65536, 33000), (80000, 20000), (100003, 40001)])
def test_part_of_the_particles(torch, mode, n, n_act):
    m, x, v = plummer_sphere(n, 4)
    m = _masses(n, 4)
    act = active_subset(n, n_act, 5)
    with _sim(m, x, v, EPS2, mode) as sim:
        sim.predict(0.0)
        got = gpu_force(sim, act)
        st = sim.stats()
    _check(mode, m, x, v, EPS2, act, got, st, f"pairs n={n} n_act={n_act}")


@pytest.mark.parametrize("mode", ["plain", "comp"])
def test_lists_that_repeat_a_particle(torch, mode):
    """A caller's list may hold a particle twice: every row is its particle's force, as from the one-sided kernel."""
    n = 21000
    m, x, v = plummer_sphere(n, 6)
    act = np.arange(n, dtype=np.int32)[:20500].copy()
    act[17] = act[8000]
    with _sim(m, x, v, EPS2, mode) as sim, _sim(m, x, v, EPS2, mode, j_tile=256, i_block=1) as one:
        for s in (sim, one):
            s.predict(0.0)
        got, ref = gpu_force(sim, act), gpu_force(one, act)
        for g, r in zip(got, ref):
            assert np.array_equal(g[17], g[8000])
            np.testing.assert_allclose(g, r, rtol=0, atol=1e-4 * np.abs(r).max())
        full = np.zeros(n, dtype=np.int32)  # the same particle in every row
        got = gpu_force(sim, full)
        assert np.all(got[0] == got[0][0]) and np.all(got[2] == got[2][0])
    rows = np.array([0, 17, 8000])
    check_force(mode, m, x, v, EPS2, act[rows], tuple(g[rows] for g in gpu_force_again(m, x, v, mode, act)),
                oracle.force(m, x, v, EPS2, act[rows]), "repeated")


def gpu_force_again(m, x, v, mode, act):
    with _sim(m, x, v, EPS2, mode) as sim:
        sim.predict(0.0)
        return gpu_force(sim, act)


def test_bad_index(torch):
    from paper_astro_ph_0702058_gb300 import NBodyError
    n = 17000
    m, x, v = plummer_sphere(n, 7)
    act = np.arange(n, dtype=np.int32)
    act[5000] = n
    with _sim(m, x, v, EPS2, "comp") as sim:
        sim.predict(0.0)
        with pytest.raises(NBodyError) as e:
            gpu_force(sim, act)
        assert e.value.code == -1
        got = gpu_force(sim, np.arange(n, dtype=np.int32))
        st = sim.stats()
    _check("comp", m, x, v, EPS2, np.arange(n, dtype=np.int32), got, st, "after a bad index")


# one and several 64-row tiles per superblock, a last superblock of one row
@pytest.mark.parametrize("n,eps2", [(4096, EPS2), (4097, 0.0), (8192, EPS2), (8193, EPS2), (16000, 0.0)])
def test_double_single(torch, n, eps2):
    """The double-single force by pairs: the mode's 1e-10 per row (max over the rows of the relative errors)."""
    m, x, v = plummer_sphere(n, 8)
    m = _masses(n, 8)
    act = np.random.default_rng(2).permutation(n).astype(np.int32)
    with _sim(m, x, v, eps2, "ds") as sim:
        sim.predict(0.0)
        got = gpu_force(sim, act)
        assert sim.stats()["last_i_per_thread"] == 2
        twice = act.copy()
        twice[5] = twice[n - 7]
        rep = gpu_force(sim, twice)  # a repeated particle: the one-sided kernel, each row its particle's force
        assert all(np.array_equal(r[5], r[n - 7]) for r in rep)
    rows = np.unique(np.concatenate([np.arange(70), np.linspace(0, n - 1, 300).astype(int), np.arange(n - 70, n)]))
    for g, a in ((got, act), (rep, twice)):
        e = errors(*(u[rows] for u in g), *oracle.force(m, x, v, eps2, a[rows]))
        for k in ("acc", "jerk", "pot"):
            assert e[k].max() <= 1e-10, (k, e[k].max())


# Units of length and mass that are powers of two change the exponents of every value and nothing else, so the forces
# scale exactly while every intermediate stays within FP32's range; r^-3 by itself does not (2^-159 and 2^156 in plain
# and compensated mode; in double-single mode its low words, 2^-132 with 24 bits, do not).
@pytest.mark.parametrize("mode,n,length,mass", [("plain", 8192, 53, 80), ("comp", 8200, 53, 80), ("plain", 40000, 53, 80),
                                                ("comp", 33000, 53, 80), ("plain", 8192, -44, -30),
                                                ("comp", 8192, -44, -30), ("ds", 4096, 36, 72), ("ds", 4100, 36, 72)])
def test_units_of_any_size(torch, mode, n, length, mass):
    m, x, v = plummer_sphere(n, 12)
    act = np.arange(n, dtype=np.int32)
    got = []
    for ln, ms in ((0, 0), (length, mass)):
        lu, mu = 2.0 ** ln, 2.0 ** ms
        with _sim(m * mu, x * lu, v * lu, EPS2 * lu * lu, mode) as sim:  # (velocities: the unit of time stays)
            s = {k: np.zeros((n, 3)) for k in ("a", "k")}
            sim.get_state(**s)  # the set-up's force, by pairs
            assert sim.stats()["last_i_per_thread"] == (2 if mode == "ds" else 4)
            sim.predict(0.0)
            pot = gpu_force(sim, act)[2]
        got.append((s["a"] * (lu * lu / mu), s["k"] * (lu * lu / mu), pot * (lu / mu)))
    for one, other in zip(*got):
        assert np.array_equal(one, other)


def test_slots_are_given_back(torch):
    """Slots above 2 GiB leave the device with the calls that wait, smaller ones stay; a refused allocation of them
    leaves the one-sided kernels, for that call only."""
    from paper_astro_ph_0702058_gb300 import Simulation, nbody_debug_fail_alloc, nbody_debug_pairs_bytes
    n = 320000
    plan = nbody_debug_pairs_bytes(1, n, n, torch.cuda.get_device_properties(0).multi_processor_count)
    assert plan > 2 << 30
    small = 512 << 20  # the context's other memory and more
    m, x, v = plummer_sphere(n, 13)
    act = torch.arange(n, dtype=torch.int32, device="cuda")
    new = lambda: [torch.zeros(n, 3, dtype=torch.float64, device="cuda") for _ in range(2)] + [  # noqa: E731
        torch.zeros(n, dtype=torch.float64, device="cuda")]
    got, refused = new(), new()
    free0 = torch.cuda.mem_get_info()[0]
    held = lambda: free0 - torch.cuda.mem_get_info()[0]  # noqa: E731
    with Simulation(m, x, v, EPS2, mode="comp") as sim:
        assert sim.stats()["last_i_per_thread"] == 4 and held() < small
        sim.predict(0.0)
        nbody_debug_fail_alloc(1)
        sim.force(act, acc=refused[0], jerk=refused[1], pot=refused[2])
        nbody_debug_fail_alloc(0)
        assert sim.stats()["last_i_per_thread"] == 1
        for _ in range(2):
            sim.force(act, acc=got[0], jerk=got[1], pot=got[2])
            assert sim.stats()["last_i_per_thread"] == 4 and held() > plan
        sim.sync()
        assert held() < small
        s = {k: np.zeros((n, 3)) for k in ("a", "k")}
        sim.get_state(**s)
        assert np.array_equal(got[0].cpu().numpy(), s["a"]) and np.array_equal(got[1].cpu().numpy(), s["k"])
        for a, b in zip(got, refused):  # two summations of the same FP32 terms (64 each, then compensated)
            assert (a - b).norm() <= 64 * 2.0 ** -24 * b.norm()
        sim.step(1.0 / 64, 1)
        assert held() < small
    n = 40000
    with Simulation(m[:n], x[:n], v[:n], EPS2, mode="comp") as sim:
        sim.sync()
        assert held() > nbody_debug_pairs_bytes(1, n, n, 152)


def test_slots_of_a_captured_force_stay(torch):
    """A caller's graph of a force keeps the slots it was captured with, whatever waits in between."""
    from paper_astro_ph_0702058_gb300 import Simulation
    n = 320000
    m, x, v = plummer_sphere(n, 14)
    stream = torch.cuda.Stream()
    act = torch.arange(n, dtype=torch.int32, device="cuda")
    out = [torch.zeros(n, 3, dtype=torch.float64, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    with Simulation(m, x, v, EPS2, mode="comp", stream=stream) as sim:
        sim.predict(0.0)
        sim.force(act, acc=out[0], jerk=out[1])
        sim.sync()
        ref = [o.clone() for o in out]
        sim.force(act, acc=out[0], jerk=out[1])  # (the capture allocates nothing)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
            sim.force(act, acc=out[0], jerk=out[1])
        assert sim.stats()["last_i_per_thread"] == 4
        for _ in range(2):
            sim.sync()  # would give the slots back
            for o in out:
                o.zero_()
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            for a, b in zip(out, ref):
                assert torch.equal(a, b)
        del g
