// Reverse mode (adjoint) of a shared-step Hermite rollout: the predictor and
// corrector of Sect. 2 of Portegies Zwart, Belleman & Geldof (2007) are
// linear in (x, v, a, k, a_p, k_p), so their adjoints are their transposes;
// the force of Eq. (Force) with the Appendix A pair term needs a vector-
// Jacobian product, evaluated here in FP32 pair arithmetic like the forward
// force, with FP64 totals.  With R = (eps^2 + |d|^2)^(-1/2), d = x_j - x_i,
// e = v_j - v_i, the pair (i, j) sends to x_j (and minus it to x_i)
//   m_j [R^3 g_a - 3 R^5 (d.g_a) d]
//     + m_j [-3 R^5 (e.g_k) d - 3 R^5 (d.g_k) e + 15 R^7 (d.e)(d.g_k) d - 3 R^5 (d.e) g_k],
// to v_j (minus to v_i) m_j [R^3 g_k - 3 R^5 (d.g_k) d], and to m_j
// R^3 (d.g_a) + R^3 (e.g_k) - 3 R^5 (d.e)(d.g_k), where (g_a, g_k) are the
// upstream gradients of particle i's acceleration and jerk.  For one particle
// p both of its roles combine linearly: with G_a = m_p g_a,q - m_q g_a,p and
// G_k likewise, one evaluation per pair (p, q) gives p's position and
// velocity gradients.
#include <algorithm>
#include <cmath>

#include "force_impl.cuh"  // fold_ds_rn; nbody_internal.cuh, ptx.cuh
#include "step_impl.cuh"

namespace nb {

namespace {

constexpr int kVjpThreads = 128;
constexpr int kVjpTile = 128;

// grid (i-blocks, j-ranges): block (x, y) takes the particles p of i-block x
// against the j-tiles of range y and writes its totals to part[y][7][n]; the
// kernel that follows adds the ranges in ascending order (deterministic).
__global__ void __launch_bounds__(kVjpThreads)
    force_vjp_kernel(const float4 *__restrict__ posm, const float4 *__restrict__ vel,
                     const float4 *__restrict__ gA, const float4 *__restrict__ gK, int n, int n_pad, float eps2,
                     int tiles_per_range, double *__restrict__ part)
{
    __shared__ float4 sp[kVjpTile], sv[kVjpTile], sa[kVjpTile], sk[kVjpTile];
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int pl = p < n ? p : 0;
    const float4 xi = posm[pl], vi = vel[pl], ga = gA[pl], gk = gK[pl];
    const float mp = xi.w;
    // running totals over the tiles as double-single pairs on the FP32 pipe (fold_ds_rn;
    // GB300's FP64 unit takes ~19 cycles per warp instruction), hi + lo in FP64 at the end
    float hx[3] = {0, 0, 0}, lx[3] = {0, 0, 0}, hv[3] = {0, 0, 0}, lv[3] = {0, 0, 0}, hm = 0.f, lm = 0.f;
    const int j_begin = blockIdx.y * tiles_per_range * kVjpTile;
    const int j_end = min(j_begin + tiles_per_range * kVjpTile, n_pad);
    for (int j0 = j_begin; j0 < j_end; j0 += kVjpTile) {
        __syncthreads();
        for (int t = threadIdx.x; t < kVjpTile; t += blockDim.x) {
            sp[t] = posm[j0 + t];
            sv[t] = vel[j0 + t];
            sa[t] = gA[j0 + t];
            sk[t] = gK[j0 + t];
        }
        __syncthreads();
        float px[3] = {0, 0, 0}, pv[3] = {0, 0, 0}, pm = 0.f;
#pragma unroll 4
        for (int t = 0; t < kVjpTile; ++t) {
            const float4 xq = sp[t], vq = sv[t], gaq = sa[t], gkq = sk[t];
            const float mq = xq.w;
            const float d0 = xi.x - xq.x, d1 = xi.y - xq.y, d2 = xi.z - xq.z;  // d = x_p - x_q
            const float e0 = vi.x - vq.x, e1 = vi.y - vq.y, e2 = vi.z - vq.z;
            const float r2 = fmaf(d2, d2, fmaf(d1, d1, fmaf(d0, d0, eps2)));
            const float R = rsqrt_mufu(r2);
            const float R2 = R * R, R3 = R2 * R, R5 = R3 * R2, R7 = R5 * R2;
            const float A0 = fmaf(-mq, ga.x, mp * gaq.x), A1 = fmaf(-mq, ga.y, mp * gaq.y),
                        A2 = fmaf(-mq, ga.z, mp * gaq.z);
            const float K0 = fmaf(-mq, gk.x, mp * gkq.x), K1 = fmaf(-mq, gk.y, mp * gkq.y),
                        K2 = fmaf(-mq, gk.z, mp * gkq.z);
            const float dA = fmaf(d2, A2, fmaf(d1, A1, d0 * A0));
            const float eK = fmaf(e2, K2, fmaf(e1, K1, e0 * K0));
            const float dK = fmaf(d2, K2, fmaf(d1, K1, d0 * K0));
            const float de = fmaf(d2, e2, fmaf(d1, e1, d0 * e0));
            const float cd = fmaf(15.0f * R7 * de, dK, -3.0f * R5 * (dA + eK));
            const float ce = -3.0f * R5 * dK;
            const float cg = -3.0f * R5 * de;
            px[0] += fmaf(cg, K0, fmaf(ce, e0, fmaf(cd, d0, R3 * A0)));
            px[1] += fmaf(cg, K1, fmaf(ce, e1, fmaf(cd, d1, R3 * A1)));
            px[2] += fmaf(cg, K2, fmaf(ce, e2, fmaf(cd, d2, R3 * A2)));
            pv[0] += fmaf(ce, d0, R3 * K0);
            pv[1] += fmaf(ce, d1, R3 * K1);
            pv[2] += fmaf(ce, d2, R3 * K2);
            // p as the source of q's force: d . g_a,q etc.
            const float dga = fmaf(d2, gaq.z, fmaf(d1, gaq.y, d0 * gaq.x));
            const float egk = fmaf(e2, gkq.z, fmaf(e1, gkq.y, e0 * gkq.x));
            const float dgk = fmaf(d2, gkq.z, fmaf(d1, gkq.y, d0 * gkq.x));
            pm += fmaf(R3, dga + egk, -3.0f * R5 * de * dgk);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            fold_ds_rn(hx[c], lx[c], px[c]);
            fold_ds_rn(hv[c], lv[c], pv[c]);
        }
        fold_ds_rn(hm, lm, pm);
    }
    if (p >= n) return;
    double tx[3], tv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        tx[c] = static_cast<double>(hx[c]) + static_cast<double>(lx[c]);
        tv[c] = static_cast<double>(hv[c]) + static_cast<double>(lv[c]);
    }
    const double tm = static_cast<double>(hm) + static_cast<double>(lm);
    double *b = part + static_cast<size_t>(blockIdx.y) * 7 * n + p;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        b[static_cast<size_t>(c) * n] = tx[c];
        b[static_cast<size_t>(3 + c) * n] = tv[c];
    }
    b[static_cast<size_t>(6) * n] = tm;
}

// One thread per (particle, component): adds the component's ranges in order.
__global__ void vjp_reduce_kernel(const double *__restrict__ part, int ranges, int n, DiffGrads G)
{
    const int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (idx >= 7LL * n) return;
    const int c = static_cast<int>(idx / n);
    const int p = static_cast<int>(idx - static_cast<int64_t>(c) * n);
    double t = 0.0;
    for (int y = 0; y < ranges; ++y) t += part[(static_cast<size_t>(y) * 7 + c) * n + p];
    if (c < 3)
        G.gxp[c][p] += t;
    else if (c < 6)
        G.gvp[c - 3][p] += t;
    else
        G.gm[p] += t;
}

// One forward step's end and the next one's start, one thread per (component,
// particle): the force on the particle (its j-range partials, or acc and jerk),
// the corrector from the state at src to the state at dst, and (predict) the
// j-stream at the prediction from there.  src, dst: x[3], v[3], a[3], k[3] of n
// doubles each.  A shared step has no criterion or level, so the components are
// independent: three short FP64 chains in parallel instead of the general
// corrector's one with its roots and division, and no kernel boundary between
// the reduction, the corrector, the copy of the state and the predictor
// (n = 4096: 7.5 + 11.0 + 2 + 4.7 us before).
template <bool DSW>
__global__ void roll_step_kernel(const double *src, double *dst, const int n, const double *__restrict__ acc,
                                 const double *__restrict__ jerk, const float *__restrict__ part, const int split,
                                 const CorrDt d, const bool predict, const JStream J, DevStatus *st)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 3 * n) return;
    const int c = idx / n, i = idx - c * n;
    double ap, kp;
    if (part) {
        constexpr int NC = DSW ? 14 : 7;
        float ah = 0.0f, al = 0.0f, kh = 0.0f, kl = 0.0f;
        const float *b = part + static_cast<size_t>(c) * n + i;
#pragma unroll 4
        for (int r = 0; r < split; ++r, b += static_cast<size_t>(NC) * n) {
            ds2_add(ah, al, b[0], DSW ? b[static_cast<size_t>(7) * n] : 0.0f);
            ds2_add(kh, kl, b[static_cast<size_t>(3) * n], DSW ? b[static_cast<size_t>(10) * n] : 0.0f);
        }
        ap = f2d(ah) + f2d(al);
        kp = f2d(kh) + f2d(kl);
    } else {
        ap = acc[3 * static_cast<size_t>(i) + c];
        kp = jerk[3 * static_cast<size_t>(i) + c];
    }
    const size_t e = static_cast<size_t>(idx), n3 = 3 * static_cast<size_t>(n);
    double xn, vn, a2e, a3;
    corr_dim(src[e], src[n3 + e], src[2 * n3 + e], src[3 * n3 + e], ap, kp, d, xn, vn, a2e, a3);
    if (!(isfinite(xn) && isfinite(vn) && isfinite(ap) && isfinite(kp))) {
        atomicOr(&st->flags, static_cast<unsigned>(kFlagNonfinite));
        atomicAdd(&st->nonfinite, 1ull);
    }
    dst[e] = xn;
    dst[n3 + e] = vn;
    dst[2 * n3 + e] = ap;
    dst[3 * n3 + e] = kp;
    if (!predict) return;
    double xp, vp;
    predict_dim(xn, vn, ap, kp, d.pd, xp, vp);
    const float h = d2f_rn(xp);
    J.soa[static_cast<size_t>(c) * J.n_pad + i] = h;
    J.soa[static_cast<size_t>(4 + c) * J.n_pad + i] = d2f_rn(vp);
    if (DSW) J.soa[static_cast<size_t>(7 + c) * J.n_pad + i] = d2f_rn(xp - f2d(h));
}

// Coefficients of the transposed corrector and predictor of a step dt.
struct AdjDt {
    double dt, dt2h, dt3s;      // dt, dt^2 / 2, dt^3 / 6
    double c1, c2, c3, c4;      // dt^4 / 24, dt^5 / 120, dt^3 / 6, dt^4 / 24
    double i1, i2, i3;          // 1 / dt, 1 / dt^2, 1 / dt^3
    PredDt pd;
};

// Between two force adjoints of the backward sweep, one thread per (component,
// particle).  With `after` (> 0) the totals of the last one (its `after` ranges
// of part) join the gradients of the predicted state and the masses, and the
// transposed predictor leads to the gradients of the state the step began
// with.  Then, with `corrector`, the transposed corrector of the step before:
// from the gradients of the corrected state (gx, gv, ga, gk) to those of the
// predicted one (gxp, gvp), of the force (gA, gK, FP32) and of the start's a, k
// (left in ga, gk); without it the force at t = 0, whose upstream is (ga, gk)
// itself.  Last, the j-stream the force adjoint reads, at the prediction of
// that step from its state `src` (dt = 0 at t = 0).
__global__ void adj_step_kernel(const double *__restrict__ part, const int after, const DiffGrads G, const int n,
                                const AdjDt d, const bool corrector, const double *__restrict__ src, const JStream J)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 3 * n) return;
    const int c = idx / n, i = idx - c * n;
    const size_t e = static_cast<size_t>(idx), n3 = 3 * static_cast<size_t>(n);
    // (the component arrays of each gradient are contiguous: gx[0][e] is component c of particle i)
    double gx = G.gx[0][e], gv = G.gv[0][e], ga = G.ga[0][e], gk = G.gk[0][e];
    if (after > 0) {
        double tx = 0.0, tv = 0.0, tm = 0.0;
        for (int y = 0; y < after; ++y) {
            const double *b = part + static_cast<size_t>(y) * 7 * n + e;
            tx += b[0];
            tv += b[n3];
            if (c == 0) tm += b[2 * n3];
        }
        if (c == 0) G.gm[i] += tm;
        const double gxp = G.gxp[0][e] + tx, gvp = G.gvp[0][e] + tv;
        gx = gxp;
        gv = gxp * d.dt + gvp;
        ga += gxp * d.dt2h + gvp * d.dt;
        gk += gxp * d.dt3s + gvp * d.dt2h;
    }
    float ap = static_cast<float>(ga), kp = static_cast<float>(gk);
    if (corrector) {
        const double g2 = d.c1 * gx + d.c3 * gv, g3 = d.c2 * gx + d.c4 * gv;
        ap = static_cast<float>(6.0 * d.i2 * g2 - 12.0 * d.i3 * g3 + ga);
        kp = static_cast<float>(-2.0 * d.i1 * g2 + 6.0 * d.i2 * g3 + gk);
        ga = -6.0 * d.i2 * g2 + 12.0 * d.i3 * g3;
        gk = -4.0 * d.i1 * g2 + 6.0 * d.i2 * g3;
    }
    G.gxp[0][e] = gx;
    G.gvp[0][e] = gv;
    G.ga[0][e] = ga;
    G.gk[0][e] = gk;
    reinterpret_cast<float *>(G.gA + i)[c] = ap;
    reinterpret_cast<float *>(G.gK + i)[c] = kp;
    double xp = src[e], vp = src[n3 + e];
    if (corrector) predict_dim(xp, vp, src[2 * n3 + e], src[3 * n3 + e], d.pd, xp, vp);
    reinterpret_cast<float *>(J.posm + i)[c] = d2f_rn(xp);
    reinterpret_cast<float *>(J.vel + i)[c] = d2f_rn(vp);
}

// Loss L = sum |x|^2 + E_pot (FP64) and its gradient at the final state:
// dL/dx_i = 2 x_i - m_i a_i, dL/dm_i = phi_i.  Grid (i-blocks, j-ranges): the FP64
// sums (phi, a) of 128 rows over a range of whole 128-particle tiles go to
// part[range][4][n].  FP64-bound (one unit per SM, ~19 cycles per warp
// instruction): 18 operations per pair with rsqrt_f64, about 45 with an IEEE
// root and division, and ranges spread a small n over every SM; n = 4096: 4.2 ms
// in 32 blocks -> 0.7.
__global__ void __launch_bounds__(128)
    loss_pairs_kernel(const State S, double eps2, int tiles_per_range, double *__restrict__ part)
{
    __shared__ double sx[128], sy[128], sz[128], sm[128];
    const int64_t i = blockIdx.x * 128ll + threadIdx.x;
    const bool live = i < S.n;
    const double xi = live ? S.x[0][i] : 0.0, yi = live ? S.x[1][i] : 0.0, zi = live ? S.x[2][i] : 0.0;
    double phi = 0.0, a0 = 0.0, a1 = 0.0, a2 = 0.0;
    const int64_t j_begin = static_cast<int64_t>(blockIdx.y) * tiles_per_range * 128;
    const int64_t j_end = j_begin + static_cast<int64_t>(tiles_per_range) * 128 < S.n
                              ? j_begin + static_cast<int64_t>(tiles_per_range) * 128
                              : S.n;
    for (int64_t j0 = j_begin; j0 < j_end; j0 += 128) {
        __syncthreads();
        const int64_t j = j0 + threadIdx.x;
        if (j < j_end) {
            sx[threadIdx.x] = S.x[0][j];
            sy[threadIdx.x] = S.x[1][j];
            sz[threadIdx.x] = S.x[2][j];
            sm[threadIdx.x] = S.m[j];
        }
        __syncthreads();
        const int jn = static_cast<int>(j_end - j0 < 128 ? j_end - j0 : 128);
#pragma unroll 2
        for (int t = 0; t < jn; ++t) {
            if (j0 + t == i) continue;
            const double dx = sx[t] - xi, dy = sy[t] - yi, dz = sz[t] - zi;
            const double y = rsqrt_f64(__fma_rn(dz, dz, __fma_rn(dy, dy, __fma_rn(dx, dx, eps2))));
            const double my = sm[t] * y, w = my * (y * y);
            phi -= my;
            a0 = __fma_rn(w, dx, a0);
            a1 = __fma_rn(w, dy, a1);
            a2 = __fma_rn(w, dz, a2);
        }
    }
    if (!live) return;
    double *b = part + static_cast<size_t>(blockIdx.y) * 4 * S.n + i;
    b[0] = phi;
    b[S.n] = a0;
    b[2 * S.n] = a1;
    b[3 * S.n] = a2;
}

// Adds the ranges in ascending order; per-particle loss terms in lval.
__global__ void loss_finish_kernel(const State S, const double *__restrict__ part, int ranges, DiffGrads G,
                                   double *__restrict__ lval)
{
    const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (i >= S.n) return;
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    for (int y = 0; y < ranges; ++y)
#pragma unroll
        for (int c = 0; c < 4; ++c) t[c] += part[(static_cast<size_t>(y) * 4 + c) * S.n + i];
    const double xi = S.x[0][i], yi = S.x[1][i], zi = S.x[2][i], mi = S.m[i];
    G.gx[0][i] = 2.0 * xi - mi * t[1];
    G.gx[1][i] = 2.0 * yi - mi * t[2];
    G.gx[2][i] = 2.0 * zi - mi * t[3];
    G.gm[i] = t[0];
    lval[i] = xi * xi + yi * yi + zi * zi + 0.5 * mi * t[0];
}

__global__ void sum_kernel(const double *__restrict__ v, int64_t n, double *out)
{
    __shared__ double s[1024];
    double acc = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) acc += v[i];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if (static_cast<int>(threadIdx.x) < k) s[threadIdx.x] += s[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = s[0];
}

int blocks_of(int64_t n, int t) { return static_cast<int>((n + t - 1) / t); }

}  // namespace

int vjp_ranges(int64_t n, int64_t n_pad, int sm_count)
{
    // enough blocks for about four per SM; ranges of whole tiles
    const int bx = blocks_of(n, kVjpThreads);
    const int tiles = static_cast<int>(n_pad / kVjpTile);
    const int want = (4 * sm_count + bx - 1) / bx;
    const int r = want < 1 ? 1 : (want > tiles ? tiles : want);
    const int tpr = (tiles + r - 1) / r;
    return (tiles + tpr - 1) / tpr;
}

size_t vjp_scratch_doubles(int64_t n, int64_t n_pad, int sm_count)
{
    return static_cast<size_t>(vjp_ranges(n, n_pad, sm_count)) * 7 * static_cast<size_t>(n);
}

cudaError_t force_vjp_launch(const JStream &J, const DiffGrads &G, int64_t n, float eps2, int sm_count,
                             double *scratch, int *ranges, cudaStream_t s, int64_t *launches)
{
    const int tiles = static_cast<int>(J.n_pad / kVjpTile);
    const int r = vjp_ranges(n, J.n_pad, sm_count);
    const int tpr = (tiles + r - 1) / r;
    const dim3 grid(blocks_of(n, kVjpThreads), r);
    force_vjp_kernel<<<grid, kVjpThreads, 0, s>>>(J.posm, J.vel, G.gA, G.gK, static_cast<int>(n),
                                                  static_cast<int>(J.n_pad), eps2, tpr, scratch);
    ++*launches;
    *ranges = r;
    return cudaGetLastError();
}

cudaError_t vjp_finish_launch(const DiffGrads &G, int64_t n, const double *scratch, int ranges, cudaStream_t s,
                              int64_t *launches)
{
    vjp_reduce_kernel<<<blocks_of(7 * n, 256), 256, 0, s>>>(scratch, ranges, static_cast<int>(n), G);
    ++*launches;
    return cudaGetLastError();
}

namespace {
// Threads of the per-(component, particle) kernels: FP64 chains, so a small n is
// spread over all SMs.
int elem_threads(int64_t n) { return 3 * n >= 152 * 512 ? 256 : 32; }
}  // namespace

cudaError_t roll_step_launch(const double *src, double *dst, int64_t n, const double *acc, const double *jerk,
                             const float *part, int split, bool two_word, int level, bool predict, const JStream &J,
                             DevStatus *st, cudaStream_t s, int64_t *launches)
{
    const double dt = std::ldexp(1.0, -level);
    CorrDt d;
    d.dt = dt;
    d.idt = 1.0 / dt;  // (powers of two: every one of these is exact but the third)
    d.idt2 = d.idt * d.idt;
    d.dt3 = dt * dt * dt;
    d.dt4 = d.dt3 * dt;
    d.pd = {dt, 0.5 * dt, dt * (1.0 / 3.0)};
    const int t = elem_threads(n);
    auto *kernel = two_word ? roll_step_kernel<true> : roll_step_kernel<false>;
    kernel<<<blocks_of(3 * n, t), t, 0, s>>>(src, dst, static_cast<int>(n), acc, jerk, part, split, d, predict, J, st);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t adj_step_launch(const double *scratch, int after, const DiffGrads &G, int64_t n, double dt, bool corrector,
                            const double *src, const JStream &J, cudaStream_t s, int64_t *launches)
{
    AdjDt d;
    d.dt = dt;
    d.dt2h = dt * dt / 2.0;
    d.dt3s = dt * dt * dt / 6.0;
    d.c1 = d.c4 = dt * dt * dt * dt / 24.0;
    d.c2 = dt * dt * dt * dt * dt / 120.0;
    d.c3 = d.dt3s;
    d.i1 = 1.0 / dt;
    d.i2 = d.i1 * d.i1;
    d.i3 = d.i2 * d.i1;
    d.pd = {dt, 0.5 * dt, dt * (1.0 / 3.0)};
    const int t = elem_threads(n);
    adj_step_kernel<<<blocks_of(3 * n, t), t, 0, s>>>(scratch, after, G, static_cast<int>(n), d, corrector, src, J);
    ++*launches;
    return cudaGetLastError();
}

namespace {
// j-ranges of the loss (about four CTAs per SM) and tiles per range.
int loss_ranges(int64_t n, int sm_count, int *tiles_per_range)
{
    const int bx = blocks_of(n, 128);
    const int want = std::max(1, std::min((4 * sm_count + bx - 1) / bx, bx));
    *tiles_per_range = (bx + want - 1) / want;
    return (bx + *tiles_per_range - 1) / *tiles_per_range;
}
}  // namespace

size_t loss_scratch_doubles(int64_t n, int sm_count)
{
    int tpr;
    return static_cast<size_t>(loss_ranges(n, sm_count, &tpr)) * 4 * static_cast<size_t>(n);
}

cudaError_t loss_launch(const State &S, double eps2, const DiffGrads &G, int sm_count, double *scratch, double *lval,
                        double *loss, cudaStream_t s, int64_t *launches)
{
    int tpr;
    const int r = loss_ranges(S.n, sm_count, &tpr);
    loss_pairs_kernel<<<dim3(blocks_of(S.n, 128), r), 128, 0, s>>>(S, eps2, tpr, scratch);
    loss_finish_kernel<<<blocks_of(S.n, 64), 64, 0, s>>>(S, scratch, r, G, lval);
    sum_kernel<<<1, 1024, 0, s>>>(lval, S.n, loss);
    *launches += 3;
    return cudaGetLastError();
}

}  // namespace nb
