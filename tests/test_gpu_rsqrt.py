"""rsqrt_f64 (csrc/step_impl.cuh), the FP64 reciprocal root of the energy, the loss and the level rule, by itself: a
kernel that calls it, compiled against the library's header, on values and range ends chosen here."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_astro_ph_0702058_gb300", "csrc")

SOURCE = r"""
#include "step_impl.cuh"
__global__ void roots(const double *x, double *y, double *seed, double *exact, long long n)
{
    const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    if (i >= n) return;
    y[i] = nb::rsqrt_f64(x[i]);
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(seed[i]) : "d"(x[i]));
    exact[i] = __ddiv_rn(1.0, __dsqrt_rn(x[i]));
}
extern "C" int run(const double *x, double *y, double *seed, double *exact, long long n)
{
    roots<<<static_cast<unsigned>((n + 255) / 256), 256>>>(x, y, seed, exact, n);
    return static_cast<int>(cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    torch = need_gpu()
    from paper_astro_ph_0702058_gb300 import build
    d = tmp_path_factory.mktemp("rsqrt")
    (d / "roots.cu").write_text(SOURCE)
    lib = str(d / "roots.so")
    r = subprocess.run([build.nvcc(), "-shared", "-Xcompiler", "-fPIC", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(d / "roots.cu"), "-o", lib] + build.ARCH,
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    f = ctypes.CDLL(lib).run

    def call(x):
        t = [torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()]
        t += [torch.zeros_like(t[0]) for _ in range(3)]
        torch.cuda.synchronize()
        assert f(*(ctypes.c_void_p(a.data_ptr()) for a in t), ctypes.c_longlong(len(x))) == 0
        return [a.cpu().numpy() for a in t[1:]]
    return call


def _ulp_error(y, x):
    """Error of y against x^(-1/2) in units of 2^-53 of it: y^2 x - 1 = 2 (y - r) / r, formed exactly from the products
    of 26-bit halves (every partial product and the sums below are exact or off by 2^-100)."""
    s = 134217729.0

    def split(a):
        h = a * s
        h = h - (h - a)
        return h, a - h

    def two_prod(a, b):
        p = a * b
        (ah, al), (bh, bl) = split(a), split(b)
        return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl

    e = np.frexp(x)[1] // 2 * 2  # scaled by an even power of two, exactly
    x, y = np.ldexp(x, -e), np.ldexp(y, e // 2)
    p, pe = two_prod(y, y)
    q, qe = two_prod(p, x)
    return 0.5 * ((q - 1.0) + (qe + pe * x)) * 2.0 ** 53


def test_error_over_the_range(roots):
    """The seed is off by `seed`, so e = 1 - x y0^2 is at most 2 seed + seed^2 and the series stops at 5 e^3 / 16; the
    operations round e and y0 e (each e 2^-53 of the result, halved) and the sum (2^-53 of it)."""
    rng = np.random.default_rng(1)
    grid = 1.0 + np.arange(1, 3 << 19) / float(1 << 19)  # where the seed's steps lie
    x = np.concatenate([np.ldexp(rng.uniform(1.0, 2.0, 1 << 21), rng.integers(-899, 900, 1 << 21)),
                        rng.uniform(1.0, 4.0, 1 << 22), np.ldexp(1.0, np.arange(-900, 901)),
                        1.0 + np.arange(1 << 20) * 2.0 ** -52, 4.0 - np.arange(1, 1 << 20) * 2.0 ** -51,
                        grid, np.nextafter(grid, 0.0), np.nextafter(grid, 9.0)])
    y, seed, exact = roots(x)
    s = np.abs(_ulp_error(seed, x)).max() * 2.0 ** -53
    worst, ieee = np.abs(_ulp_error(y, x)).max(), np.abs(_ulp_error(exact, x)).max()
    print(f"\nseed 2^{np.log2(s):.2f}, rsqrt_f64 {worst:.4f}, IEEE root and division {ieee:.4f} (units of 2^-53)")
    assert s < 2.0 ** -19.9
    e = 2 * s + s * s
    assert worst <= 1.0 + e + 5.0 / 16.0 * e ** 3 * 2.0 ** 53
    assert worst <= ieee


def test_range_ends(roots):
    """Outside [2^-900, 2^900]: the IEEE root and division."""
    tiny = np.array([0.0, -0.0, 5e-324, 1e-310, np.ldexp(1.0, -1022), np.ldexp(1.5, -901), np.nextafter(2.0 ** -900, 0),
                     2.0 ** -900, np.ldexp(1.0, 900), np.nextafter(2.0 ** 901, 0), 2.0 ** 901, 1.7976931348623157e308,
                     np.inf, -1.0, -np.inf, np.nan])
    with np.errstate(all="ignore"):
        y, _, exact = roots(tiny)
        np.testing.assert_allclose(y, exact, rtol=2.0 ** -52, atol=0, equal_nan=True)
        outside = ~((np.abs(tiny) >= 2.0 ** -900) & (np.abs(tiny) < 2.0 ** 901)) | (tiny < 0)
        assert np.array_equal(y[outside], exact[outside], equal_nan=True)
