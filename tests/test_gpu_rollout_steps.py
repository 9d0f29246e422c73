"""The fused steps of a shared-step rollout (csrc/adjoint.cu) against the library's own block-step calls."""
import numpy as np
import pytest

from synthetic import plummer_sphere
from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu
EPS2, LEVEL = (1.0 / 128) ** 2, 9


# one particle, blocks of 32 (component, particle) threads and their edges, several j-ranges, pairs (8192)
@pytest.mark.parametrize("n,mode", [(1, "plain"), (2, "comp"), (11, "plain"), (33, "comp"), (257, "plain"), (1500, "comp"),
                                    (8191, "plain"), (16384, "comp"), (20000, "plain"), (300, "ds"), (300, "sumcheck"),
                                    (100, "sorted")])
def test_rollout_equals_block_steps(n, mode):
    """x_T and v_T of three steps against predict, force and correct called one by one.  From 8192 particles on, and
    in the modes without packed pairs, both add the same FP32 partial sums; only the order of the last additions (to
    ~2^-48) may differ, so x and v agree to ~1e-13.  Below, a rollout splits a row's sum among more threads."""
    need_gpu()
    from paper_astro_ph_0702058_gb300 import MODES, Simulation
    from paper_astro_ph_0702058_gb300._lib import nbody_rollout
    m, x, v = plummer_sphere(n, 50 + n)
    xT, vT = np.zeros((n, 3)), np.zeros((n, 3))
    nbody_rollout(n, m, x, v, EPS2, LEVEL, 3, MODES[mode], xT, vT)
    every = np.arange(n, dtype=np.int32)
    with Simulation(m, x, v, EPS2, lmin=LEVEL, lmax=LEVEL, mode=mode) as sim:
        for k in range(3):
            sim.predict((k + 1) * 2.0 ** -LEVEL)
            sim.force(every)
            sim.correct(every)
        s = {k: np.zeros((n, 3)) for k in ("x", "v")}
        sim.get_state(**s)
    tx, tv = 1e-13 * np.abs(s["x"]).max(), 1e-12 * max(np.abs(s["v"]).max(), 1e-30)
    if mode in ("plain", "comp") and n < 8192:
        # FP32 sums of the same terms in two orders differ by at most 2 n u sum |term| (u = 2^-24).  A step turns a
        # force and jerk off by da, dk into 0.5 dt da + 0.09 dt^2 dk in v and 0.35 dt^2 da + 0.04 dt^3 dk in x at
        # most from either end of it; three steps, then a factor 2 for what the moved particles' forces add.
        da = dk = 0.0
        for i in range(n):
            dx, dv = np.linalg.norm(x - x[i], axis=1), np.linalg.norm(v - v[i], axis=1)
            w = 2 * n * 2.0 ** -24 * m / (dx ** 2 + EPS2) ** 1.5
            da, dk = max(da, (w * dx).sum()), max(dk, (w * 4 * dv).sum())
        dt = 2.0 ** -LEVEL
        ev = 3 * 2 * (0.5 * dt * da + 0.09 * dt ** 2 * dk)
        tv += 2 * ev
        tx += 2 * (3 * 2 * (0.35 * dt ** 2 * da + 0.04 * dt ** 3 * dk) + 3 * dt * ev)
    np.testing.assert_allclose(xT, s["x"], rtol=0, atol=tx)
    np.testing.assert_allclose(vT, s["v"], rtol=0, atol=tv)


@pytest.mark.parametrize("steps", [0, 1])
def test_shortest_rollouts(steps):
    need_gpu()
    from paper_astro_ph_0702058_gb300._lib import nbody_rollout_vjp
    n = 40
    m, x, v = plummer_sphere(n, 9)
    g = np.random.default_rng(1).standard_normal((2, n, 3))
    out = [np.zeros((n, 3)), np.zeros((n, 3)), np.zeros(n)]
    nbody_rollout_vjp(n, m, x, v, EPS2, LEVEL, steps, 16, 0, g[0], g[1], *out)
    from oracle import adjoint
    dt = 2.0 ** -LEVEL
    ref = adjoint.rollout_vjp(m, x, v, EPS2, dt, steps, g[0], g[1])[2:]
    # The force adjoint runs at FP32 positions: a separation is off by 2^-24 (|x_i| + |x_j|), which moves
    # da/dx by at most 6 m / eps^4 of it, and the step weighs the force by ~dt^2 (x) of the cotangents; twice that
    # for the jerk's part and the two forces of a step.
    tol = 2 * 2.0 ** -24 * 2 * np.abs(x).max() * dt ** 2 * 6 * m.max() / EPS2 ** 2 * np.abs(g).max()
    for o, r in zip(out, ref):
        np.testing.assert_allclose(o, r, rtol=0, atol=tol)


def test_segments_where_the_states_are_too_many_to_keep():
    """20000 particles x 600 steps are 1.15 GB of states: segments run again, their length without effect."""
    need_gpu()
    from paper_astro_ph_0702058_gb300._lib import nbody_rollout_vjp
    n, steps = 20000, 600
    m, x, v = plummer_sphere(n, 10)
    g = np.random.default_rng(2).standard_normal((2, n, 3))
    out = []
    for every in (16, 50):
        out.append([np.zeros((n, 3)), np.zeros((n, 3)), np.zeros(n)])
        nbody_rollout_vjp(n, m, x, v, EPS2, LEVEL, steps, every, 0, g[0], g[1], *out[-1])
    for a, b in zip(*out):
        assert np.all(np.isfinite(a)) and np.array_equal(a, b)


def test_nonfinite_steps_are_reported():
    """A run whose velocities leave FP32's range after its first step fails, without a count of rows that is not one."""
    import re
    need_gpu()
    from paper_astro_ph_0702058_gb300 import NBodyError
    from paper_astro_ph_0702058_gb300._lib import nbody_rollout, nbody_rollout_vjp
    n, steps = 2, 3
    m, x, v = np.full(n, 1e25), np.array([[5e-4, 0, 0], [-5e-4, 0, 0]]), np.zeros((n, 3))
    out = [np.zeros((n, 3)), np.zeros((n, 3))]
    for call in (lambda: nbody_rollout(n, m, x, v, 1e-8, 0, steps, 0, *out),
                 lambda: nbody_rollout_vjp(n, m, x, v, 1e-8, 0, steps, 16, 0, np.ones((n, 3)), None, *out, None)):
        with pytest.raises(NBodyError) as e:
            call()
        assert e.value.code == -5 and "non-finite" in str(e.value)
        rows = re.search(r"(\d+) rows", str(e.value))
        assert rows is None or int(rows.group(1)) <= n * steps, str(e.value)
