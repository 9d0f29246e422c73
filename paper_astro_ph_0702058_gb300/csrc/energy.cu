// Energy diagnostic (Sect. 4.2's accuracy measure): E_kin = sum m v^2 / 2 and
// E_pot = -sum_{i<j} m_i m_j / sqrt(eps^2 + |x_j - x_i|^2).
//
// Particles are cut into tiles of T rows; one CTA per unordered pair of tiles
// (I <= J) adds the terms of its pairs i < j, each once, and writes one sum (the
// CTA of (I, I) also the kinetic energy of the rows of I).  One block then adds
// the CTAs' sums in a fixed order.  T is the smallest power of two whose sums
// fit the scratch (as many doubles as particles): enough CTAs at any n.
//
// FP64 potential.  GB300's SM has one FP64 unit that takes ~19 cycles per warp
// instruction, so the pair term is written to use few of its operations: 6 for
// the differences and r^2; then, from the MUFU's approximate y0 (rsqrt.approx.f64,
// a relative error of 2^-20), the root by one step of third order in the
// residual e = 1 - r^2 y0^2, y = y0 (1 + e/2 + 3 e^2/8) (the binomial series of
// (1 - e)^(-1/2); the next term is 5 e^3/16 < 2^-58.7), 5; and the product with m_j
// into the sum, 1.  A pair costs 12 FP64 operations, where an IEEE square root
// and division per ordered pair took about 2 x 28: n = 65536 240 -> 46.5 ms (49 by
// 12 operations of 2^31 pairs at 1.68 per clock per SM).
//
// Double-single potential (~1e-13, for large n), per pair ~130 FP32 operations:
//   x_j, x_i, m_j, eps2: (hi, lo) splits of the FP64 values
//   dx = x_j - x_i, r2 = eps2 + dx.dx        (double-single)
//   1/sqrt(r2): MUFU seed and one Newton step with a double-single residual
//   phi_i -= m_j / r                          (double-single product)
// added in double-single over a j-tile (all of one sign), then in FP64.
#include <algorithm>

#include "ds_arith.cuh"
#include "nbody_internal.cuh"
#include "step_impl.cuh"

namespace nb {

namespace {

using namespace dsa;

constexpr int kEThreads = 128;  // threads of a CTA at most, and j of a shared-memory tile
constexpr int kEMinTile = 32;

__device__ __forceinline__ ds split(const double v)
{
    const float h = __double2float_rn(v);
    return {h, __double2float_rn(v - static_cast<double>(h))};
}

// Rows of a tile and tiles for n particles.
__host__ __device__ inline int energy_tile(const int64_t n)
{
    int t = kEMinTile;
    for (;;) {
        const int64_t s = (n + t - 1) / t;
        if (s * (s + 1) / 2 + s <= n + kEnergyPad) return t;
        t *= 2;
    }
}

template <bool DSP>
__global__ void __launch_bounds__(kEThreads)
    energy_pairs_kernel(const State S, const double eps2, const int T, const int n_tiles,
                        const unsigned long long *__restrict__ trange, double *__restrict__ pot,
                        double *__restrict__ kin)
{
    if (trange[0] != trange[1]) return;  // not synchronised: the host reports it
    __shared__ double sd[DSP ? 1 : 4][DSP ? 1 : kEThreads];
    __shared__ float4 sh[DSP ? kEThreads : 1], sl[DSP ? kEThreads : 1];
    __shared__ double red[32];
    const int nt = blockDim.x, tid = threadIdx.x;
    // the unit (I, J), I <= J
    const long long u = blockIdx.x;
    int J = static_cast<int>((sqrt(8.0 * static_cast<double>(u) + 1.0) - 1.0) * 0.5);
    while (static_cast<long long>(J + 1) * (J + 2) / 2 <= u) ++J;
    while (static_cast<long long>(J) * (J + 1) / 2 > u) --J;
    const int I = static_cast<int>(u - static_cast<long long>(J) * (J + 1) / 2);
    const bool diag = I == J;
    const int64_t i_end = min(S.n, static_cast<int64_t>(I + 1) * T);
    const int64_t j_begin = static_cast<int64_t>(J) * T, j_end = min(S.n, j_begin + T);
    const ds e2 = split(eps2);
    double sum = 0.0, ke = 0.0;
    for (int64_t i0 = static_cast<int64_t>(I) * T; i0 < i_end; i0 += nt) {
        const int64_t i = i0 + tid;
        const bool live = i < i_end;
        const int64_t li = live ? i : i_end - 1;
        const double xi = S.x[0][li], yi = S.x[1][li], zi = S.x[2][li], mi = live ? S.m[li] : 0.0;
        const ds xs[3] = {split(xi), split(yi), split(zi)};
        double p = 0.0;
        for (int64_t j0 = diag ? i0 : j_begin; j0 < j_end; j0 += nt) {
            __syncthreads();
            const int64_t j = j0 + tid;
            if (j < j_end) {
                const double x = S.x[0][j], y = S.x[1][j], z = S.x[2][j], m = S.m[j];
                if constexpr (DSP) {
                    const ds a = split(x), b = split(y), c = split(z), d = split(m);
                    sh[tid] = make_float4(a.h, b.h, c.h, d.h);
                    sl[tid] = make_float4(a.l, b.l, c.l, d.l);
                } else {
                    sd[0][tid] = x;
                    sd[1][tid] = y;
                    sd[2][tid] = z;
                    sd[3][tid] = m;
                }
            }
            __syncthreads();
            const int jn = static_cast<int>(j_end - j0 < nt ? j_end - j0 : nt);
            const int t0 = diag && j0 == i0 ? tid + 1 : 0;  // pairs j > i
            if constexpr (DSP) {
                ds tile = {0.0f, 0.0f};
#pragma unroll 2
                for (int t = t0; t < jn; ++t) {
                    const float4 h = sh[t], l = sl[t];
                    const ds dx = ds_add({h.x, l.x}, ds_neg(xs[0]));
                    const ds dy = ds_add({h.y, l.y}, ds_neg(xs[1]));
                    const ds dz = ds_add({h.z, l.z}, ds_neg(xs[2]));
                    const ds r2 = ds_add(ds_add(ds_add(e2, ds_mul(dx, dx)), ds_mul(dy, dy)), ds_mul(dz, dz));
                    tile = ds_add(tile, ds_mul({h.w, l.w}, ds_rsqrt(r2)));
                }
                p += static_cast<double>(tile.h) + static_cast<double>(tile.l);
            } else {
#pragma unroll 4
                for (int t = t0; t < jn; ++t) {
                    const double dx = sd[0][t] - xi, dy = sd[1][t] - yi, dz = sd[2][t] - zi;
                    const double r2 = __fma_rn(dz, dz, __fma_rn(dy, dy, __fma_rn(dx, dx, eps2)));
                    p = __fma_rn(sd[3][t], rsqrt_f64(r2), p);
                }
            }
        }
        if (live) {
            sum -= mi * p;
            if (diag) {
                const double vx = S.v[0][i], vy = S.v[1][i], vz = S.v[2][i];
                ke += 0.5 * mi * (vx * vx + vy * vy + vz * vz);
            }
        }
    }
    __syncthreads();
    sum = block_reduce(sum, AddOp(), red, 0.0);
    if (tid == 0) pot[u] = sum;
    if (diag) {
        ke = block_reduce(ke, AddOp(), red, 0.0);
        if (tid == 0) kin[I] = ke;
    }
}

// out[0] = the sum of kin[0 .. n_kin), out[1] = of pot[0 .. n_pot), in a fixed order.
__global__ void __launch_bounds__(1024)
    energy_sum_kernel(const double *__restrict__ pot, const int64_t n_pot, const double *__restrict__ kin,
                      const int64_t n_kin, double *out)
{
    __shared__ double red[32];
    double p[4] = {0.0, 0.0, 0.0, 0.0}, k = 0.0;
    for (int64_t i = threadIdx.x; i < n_pot; i += 4096)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (i + 1024 * c < n_pot) p[c] += pot[i + 1024 * c];
    for (int64_t i = threadIdx.x; i < n_kin; i += 1024) k += kin[i];
    const double ps = block_reduce((p[0] + p[1]) + (p[2] + p[3]), AddOp(), red, 0.0);
    const double ks = block_reduce(k, AddOp(), red, 0.0);
    if (threadIdx.x == 0) {
        out[0] = ks;
        out[1] = ps;
    }
}

}  // namespace

cudaError_t energy_launch(const State &S, double eps2, double *scratch, const unsigned long long *trange, double *out,
                          cudaStream_t s, int64_t *launches, bool ds_potential)
{
    const int T = energy_tile(S.n);
    const int64_t n_t = (S.n + T - 1) / T, units = n_t * (n_t + 1) / 2;
    double *pot = scratch, *kin = scratch + units;
    const int nt = std::min(T, kEThreads);
    if (ds_potential)
        energy_pairs_kernel<true><<<static_cast<unsigned>(units), nt, 0, s>>>(S, eps2, T, static_cast<int>(n_t), trange,
                                                                              pot, kin);
    else
        energy_pairs_kernel<false><<<static_cast<unsigned>(units), nt, 0, s>>>(S, eps2, T, static_cast<int>(n_t),
                                                                               trange, pot, kin);
    energy_sum_kernel<<<1, 1024, 0, s>>>(pot, units, kin, n_t, out);
    *launches += 2;
    return cudaGetLastError();
}

}  // namespace nb
