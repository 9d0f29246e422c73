"""The rule that gives a force to the kernels by unordered pairs (host arithmetic, no GPU)."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CAP = 8 << 30  # bytes of slots at most
PLAIN, COMP, DS = 0, 1, 4


def _plan(*calls):
    """nbody_debug_pairs_bytes of each (mode, n_act, n, sm_count), in a process that a rule without an end cannot hold."""
    from paper_astro_ph_0702058_gb300 import build
    build.build()
    src = ("from paper_astro_ph_0702058_gb300._lib import nbody_debug_pairs_bytes as f\n"
           f"print(*(f(*c) for c in {list(calls)!r}))")
    r = subprocess.run([sys.executable, "-c", src], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-2000:]
    return [int(w) for w in r.stdout.split()]


# the double-single slots of one superblock alone pass the cap above 76.7 million particles
@pytest.mark.parametrize("mode", [PLAIN, COMP, DS])
def test_every_size_has_a_plan(mode):
    sizes = [1, 4095, 4096, 8191, 8192, 1 << 20, 2_400_000, 76_000_000, 80_000_000, (1 << 31) - 1]
    got = _plan(*((mode, n, n, 152) for n in sizes))
    least = 4096 if mode == DS else 8192
    words = 7 if mode == PLAIN else 14
    for n, b in zip(sizes, got):
        assert 0 <= b <= CAP and b % (words * 4 * n) == 0
        assert (b > 0) == (least <= n <= 2_400_000), (n, b)
