"""The energy diagnostic by tiles of unordered pairs (csrc/energy.cu) against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from synthetic import plummer_sphere
from tests.gpu_common import EPS2, need_gpu

pytestmark = pytest.mark.gpu


# one tile and its edges (32 rows at least), several tiles, tiles of more than one CTA pass (128 rows and more)
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 65, 1000, 4097, 9001, 40000])
@pytest.mark.parametrize("eps2", [EPS2, 0.0])
def test_energy_sizes(n, eps2):
    """FP64 sums of n^2 / 2 terms of one sign, each within a few 2^-53: 1e-13 (double-single terms: 2^-44 each)."""
    need_gpu()
    from paper_astro_ph_0702058_gb300 import Simulation
    m, x, v = plummer_sphere(n, 30 + n)
    w = np.random.default_rng(n).uniform(0.1, 10.0, n)
    m = w / w.sum()
    ek, ep = oracle.energy(m, x, v, eps2)
    with Simulation(m, x, v, eps2) as sim:
        for ds in (False, True):
            gk, gp = sim.energy(ds_potential=ds)
            assert abs(gk - ek) <= 1e-13 * abs(ek)
            assert abs(gp - ep) <= 1e-13 * abs(ep), (ds, gp, ep)
