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
// velocity gradients, and minus them q's.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "force_x2.cuh"  // packed FP32; fold_ds_rn, ds2_add
#include "step_impl.cuh"

namespace nb {

namespace {

// The kernels of a rollout's steps are launched with programmatic stream
// serialisation (launch_after): once every block of this kernel runs, the next
// one's may be scheduled, and each waits here, before its first read or write of
// memory, until the kernel before it is complete and its stores are visible.  A
// step's kernels take 5 to 15 us each, so the 1 to 2 us between two of them
// count (4096 particles, 64 steps, loss and gradient 7.01 -> 6.72 ms; below 2000
// particles the host issues no faster than the kernels end).  What these kernels
// read was written by the one before, so their pointers are not __restrict__ (no
// read-only loads).
__device__ __forceinline__ void after_previous()
{
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

constexpr int kVjpRows = 64;  // rows of a warp

// Sums of a pair that both of its particles need.  Row data packed for two rows
// (force_x2.cuh's packed FP32), the j's values twice.
struct VjpRow {
    f2_t x[3], m, v[3], a[3], k[3];  // position, mass, velocity, upstream of acceleration and jerk
};
struct VjpSum {
    f2_t x[3], v[3], m;
};

__device__ __forceinline__ f2_t dot3(const f2_t (&a)[3], const f2_t (&b)[3])
{
    return f2_fma(a[2], b[2], f2_fma(a[1], b[1], f2_mul(a[0], b[0])));
}

// The pair (p, q): p's share to P, q's to Q.  Exchanging p and q turns d, e, G_a
// and G_k over, so the position and velocity gradients of q are minus p's; the
// mass gradients take the other particle's upstream each.
template <bool DIAG>
__device__ __forceinline__ void vjp_pair(const VjpRow &p, const VjpRow &q, const f2_t E2, const bool ma, const bool mb,
                                         VjpSum &P, VjpSum &Q)
{
    f2_t d[3], e[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        d[c] = f2_sub(p.x[c], q.x[c]);
        e[c] = f2_sub(p.v[c], q.v[c]);
    }
    const f2_t r2 = f2_fma(d[2], d[2], f2_fma(d[1], d[1], f2_fma(d[0], d[0], E2)));
    float a, b;
    f2_unpack(r2, a, b);
    if (DIAG) {  // pairs to leave out: r^-1 = 0
        a = ma ? INFINITY : a;
        b = mb ? INFINITY : b;
    }
    const f2_t R = f2_pack(rsqrt_mufu(a), rsqrt_mufu(b));
    const f2_t R2 = f2_mul(R, R), R3 = f2_mul(R2, R);
    const f2_t t5 = f2_mul(f2_mul(R3, R2), f2_pack(-3.0f, -3.0f));  // -3 R^5
    const f2_t de = dot3(d, e);
    const f2_t aq = dot3(d, q.a), ap = dot3(d, p.a), bq = dot3(e, q.k), bp = dot3(e, p.k);
    const f2_t cq = dot3(d, q.k), cp = dot3(d, p.k);
    const f2_t nmq = f2_sub(0ull, q.m);
    const f2_t sq = f2_add(aq, bq), sp = f2_add(ap, bp);
    const f2_t dAeK = f2_fma(nmq, sp, f2_mul(p.m, sq));  // d.G_a + e.G_k
    const f2_t dK = f2_fma(nmq, cp, f2_mul(p.m, cq));
    const f2_t cg = f2_mul(t5, de), ce = f2_mul(t5, dK);
    const f2_t w = f2_mul(f2_mul(R2, cg), f2_pack(-5.0f, -5.0f));  // 15 R^7 (d.e)
    const f2_t cd = f2_fma(w, dK, f2_mul(t5, dAeK));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const f2_t A = f2_fma(nmq, p.a[c], f2_mul(p.m, q.a[c])), K = f2_fma(nmq, p.k[c], f2_mul(p.m, q.k[c]));
        const f2_t gx = f2_fma(cg, K, f2_fma(ce, e[c], f2_fma(cd, d[c], f2_mul(R3, A))));
        const f2_t gv = f2_fma(ce, d[c], f2_mul(R3, K));
        P.x[c] = f2_add(P.x[c], gx);
        Q.x[c] = f2_sub(Q.x[c], gx);
        P.v[c] = f2_add(P.v[c], gv);
        Q.v[c] = f2_sub(Q.v[c], gv);
    }
    P.m = f2_fma(R3, sq, f2_fma(cg, cq, P.m));
    Q.m = f2_sub(Q.m, f2_fma(R3, sp, f2_mul(cg, cp)));
}

__device__ __forceinline__ f2_t &vjp_at(VjpSum &s, const int c) { return c < 3 ? s.x[c] : c < 6 ? s.v[c - 3] : s.m; }

// Adds x to the total of component c at p (component stride n): FP32 where a slot
// holds one sum of 64 terms, else a double-single pair (lo words 7 further on).
template <bool FOLD>
__device__ __forceinline__ void vjp_fold(float *p, const size_t n, const int c, const float x, const bool first)
{
    float *h = p + static_cast<size_t>(c) * n;
    if (!FOLD) {
        *h = x;
        return;
    }
    float *l = p + static_cast<size_t>(7 + c) * n;
    float hi = first ? 0.0f : *h, lo = first ? 0.0f : *l;
    fold_ds_rn(hi, lo, x);
    *h = hi;
    *l = lo;
}

// Force adjoint by unordered pairs: the structure of force_sym_kernel
// (force_sym.cuh) with one warp per CTA and 64 rows per warp.  Superblocks of 64
// (FOLD: 64 x tiles) rows; one CTA per unordered pair (I, J) of them and per
// j-part h of H (H = 2: the two halves of J's 64, FOLD: J whole, H = 1).  Lane l
// holds rows l and l + 32 of a packed pair and takes j = (l + s) mod 32 in step s;
// the j's sums go down one lane per step.  Slots of part: rows of I in J H + h,
// those of J in I H, the second side of (I, I) in S H.
// One pair costs 96 packed FP32 operations for both particles, 40 of them with
// three different registers (3 cycles each, not 2: force_sym.cuh), where the
// one-sided scalar loop took about 85 per particle: n = 4096 59.8 -> 41.2 us,
// 1500 12.8 -> 9.0 us.
template <int H, bool FOLD>
__global__ void __launch_bounds__(32, 12)
    vjp_pairs_kernel(const float4 *posm, const float4 *vel, const float4 *gA, const float4 *gK, const int n,
                     const float eps2, const int S, const int tiles, float *part)
{
    static_assert(!FOLD || H == 1, "tiles of a superblock whole");
    constexpr int NC = FOLD ? 14 : 7;
    __shared__ float4 sj[4][32];
    const int lane = threadIdx.x;
    const int u = blockIdx.x / H, h = blockIdx.x % H;
    int J = static_cast<int>((sqrtf(8.0f * u + 1.0f) - 1.0f) * 0.5f);
    while ((J + 1) * (J + 2) / 2 <= u) ++J;
    while (J * (J + 1) / 2 > u) --J;
    const int I = u - J * (J + 1) / 2;
    const bool diag = I == J;
    const size_t slot = static_cast<size_t>(NC) * n;
    float *pi_out = part + slot * (J * H + h), *pj_out = part + slot * (diag ? S * H : I * H);
    const int sb = tiles * kVjpRows;
    const int j_end = min(n, (J + 1) * sb);
    const f2_t E2 = f2_pack(eps2, eps2);
    const float4 far = make_float4(kPadPosition, kPadPosition, kPadPosition, 0.f), zero = make_float4(0.f, 0.f, 0.f, 0.f);
    after_previous();
    for (int i0 = I * sb; i0 < min(n, (I + 1) * sb); i0 += kVjpRows) {
        const int r0 = i0 + lane, r1 = r0 + 32;
        VjpRow p;
        {
            const float4 x0 = r0 < n ? posm[r0] : far, x1 = r1 < n ? posm[r1] : far;
            const float4 v0 = r0 < n ? vel[r0] : zero, v1 = r1 < n ? vel[r1] : zero;
            const float4 a0 = r0 < n ? gA[r0] : zero, a1 = r1 < n ? gA[r1] : zero;
            const float4 k0 = r0 < n ? gK[r0] : zero, k1 = r1 < n ? gK[r1] : zero;
            p.x[0] = f2_pack(x0.x, x1.x);
            p.x[1] = f2_pack(x0.y, x1.y);
            p.x[2] = f2_pack(x0.z, x1.z);
            p.m = f2_pack(x0.w, x1.w);
            p.v[0] = f2_pack(v0.x, v1.x);
            p.v[1] = f2_pack(v0.y, v1.y);
            p.v[2] = f2_pack(v0.z, v1.z);
            p.a[0] = f2_pack(a0.x, a1.x);
            p.a[1] = f2_pack(a0.y, a1.y);
            p.a[2] = f2_pack(a0.z, a1.z);
            p.k[0] = f2_pack(k0.x, k1.x);
            p.k[1] = f2_pack(k0.y, k1.y);
            p.k[2] = f2_pack(k0.z, k1.z);
        }
        bool ifirst = true;
        for (int t0 = diag ? i0 : J * sb; t0 < j_end; t0 += kVjpRows) {  // a tile of 64 j
            VjpSum P;
#pragma unroll
            for (int c = 0; c < 7; ++c) vjp_at(P, c) = 0ull;
            for (int j0 = t0 + 32 * h; j0 < min(j_end, H == 2 ? t0 + 32 * h + 32 : t0 + 64); j0 += 32) {
                __syncwarp();
                const int j = j0 + lane;
                sj[0][lane] = j < n ? posm[j] : far;
                sj[1][lane] = j < n ? vel[j] : zero;
                sj[2][lane] = j < n ? gA[j] : zero;
                sj[3][lane] = j < n ? gK[j] : zero;
                __syncwarp();
                VjpSum Q;
#pragma unroll
                for (int c = 0; c < 7; ++c) vjp_at(Q, c) = 0ull;
                auto turn = [&](auto own) {
#pragma unroll 1
                    for (int s = 0; s < 32; ++s) {
                        const int jl = (lane + s) & 31;
                        const float4 x = sj[0][jl], v = sj[1][jl], a = sj[2][jl], k = sj[3][jl];
                        VjpRow q;
                        q.x[0] = f2_pack(x.x, x.x);
                        q.x[1] = f2_pack(x.y, x.y);
                        q.x[2] = f2_pack(x.z, x.z);
                        q.m = f2_pack(x.w, x.w);
                        q.v[0] = f2_pack(v.x, v.x);
                        q.v[1] = f2_pack(v.y, v.y);
                        q.v[2] = f2_pack(v.z, v.z);
                        q.a[0] = f2_pack(a.x, a.x);
                        q.a[1] = f2_pack(a.y, a.y);
                        q.a[2] = f2_pack(a.z, a.z);
                        q.k[0] = f2_pack(k.x, k.x);
                        q.k[1] = f2_pack(k.y, k.y);
                        q.k[2] = f2_pack(k.z, k.z);
                        constexpr bool OWN = decltype(own)::value;
                        vjp_pair<OWN>(p, q, E2, OWN && j0 + jl <= r0, OWN && j0 + jl <= r1, P, Q);
#pragma unroll
                        for (int c = 0; c < 7; ++c) {
                            float a0, a1;
                            f2_unpack(vjp_at(Q, c), a0, a1);
                            a0 = __shfl_sync(0xffffffffu, a0, (lane + 1) & 31);
                            a1 = __shfl_sync(0xffffffffu, a1, (lane + 1) & 31);
                            vjp_at(Q, c) = f2_pack(a0, a1);
                        }
                    }
                };
                if (diag && t0 == i0)
                    turn(std::true_type());
                else
                    turn(std::false_type());
                if (j < j_end) {
#pragma unroll
                    for (int c = 0; c < 7; ++c) {
                        float a0, a1;
                        f2_unpack(vjp_at(Q, c), a0, a1);
                        vjp_fold<FOLD>(pj_out + j, n, c, a0 + a1, i0 == I * sb);
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < 7; ++c) {
                float a0, a1;
                f2_unpack(vjp_at(P, c), a0, a1);
                if (r0 < n) vjp_fold<FOLD>(pi_out + r0, n, c, a0, ifirst);
                if (r1 < n) vjp_fold<FOLD>(pi_out + r1, n, c, a1, ifirst);
            }
            ifirst = false;
        }
    }
}

// The per-(component, particle) kernels: blocks of 32 columns (a warp's width of
// one component's particles) x kLanes warps.  The sums over slots or j-ranges of
// a column are spread over the warps (warp w takes w, w + kLanes, ...), added in
// double-single and then in warp order; warp 0 goes on alone with the column's
// FP64 work.  One thread per column instead took 45 us (65 slots) and 20 us (16
// ranges) at n = 4096, nearly all of it the latency of its own loads.
constexpr int kLanes = 8;

// Sums of NV values over count of them per column: at(s, v, hi, lo) loads value v
// of entry s.  Every thread of the block calls; warp 0 gets the sums.
template <int NV, class At>
__device__ __forceinline__ void column_sums(const int count, At &&at, double (&sum)[NV])
{
    __shared__ float2 sh[NV][kLanes][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float h[NV], l[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) h[v] = l[v] = 0.0f;
#pragma unroll 4
    for (int s = w; s < count; s += kLanes)
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            float a = 0.0f, b = 0.0f;
            at(s, v, a, b);
            ds2_add(h[v], l[v], a, b);
        }
#pragma unroll
    for (int v = 0; v < NV; ++v) sh[v][w][lane] = make_float2(h[v], l[v]);
    __syncthreads();
    if (w == 0)
#pragma unroll
        for (int v = 0; v < NV; ++v) {
#pragma unroll
            for (int k = 1; k < kLanes; ++k) ds2_add(h[v], l[v], sh[v][k][lane].x, sh[v][k][lane].y);
            sum[v] = f2d(h[v]) + f2d(l[v]);
        }
}

// Value of component c of particle i in slot s (zero where the slot has none).
// (part: written by the kernel before, see after_previous.)
__device__ __forceinline__ void vjp_at_slot(const float *part, const VjpSlots V, const int n, const int c,
                                            const int i, const int s, float &a, float &b)
{
    if (V.parts == 2 && s < 2 * (i / V.rows) && (s & 1)) return;  // (as the j of an earlier superblock: one slot)
    const float *p = part + (static_cast<size_t>(s) * (V.two_word ? 14 : 7) + c) * n + i;
    a = p[0];
    if (V.two_word) b = p[static_cast<size_t>(7) * n];
}

// Adds the totals to the gradients.
__global__ void __launch_bounds__(32 * kLanes)
    vjp_reduce_kernel(const float *__restrict__ part, const VjpSlots V, int n, DiffGrads G)
{
    const int64_t idx = blockIdx.x * 32ll + (threadIdx.x & 31);
    const bool live = idx < 7ll * n;
    const int c = live ? static_cast<int>(idx / n) : 0;
    const int p = live ? static_cast<int>(idx - static_cast<int64_t>(c) * n) : 0;
    double t[1];
    column_sums(V.sb * V.parts + 1, [&](int s, int, float &a, float &b) { vjp_at_slot(part, V, n, c, p, s, a, b); }, t);
    if (threadIdx.x >= 32 || !live) return;
    if (c < 3)
        G.gxp[c][p] += t[0];
    else if (c < 6)
        G.gvp[c - 3][p] += t[0];
    else
        G.gm[p] += t[0];
}

// One forward step's end and the next one's start, per (component, particle):
// the force on the particle (its j-range partials, or acc and jerk),
// the corrector from the state at src to the state at dst, and (predict) the
// j-stream at the prediction from there.  src, dst: x[3], v[3], a[3], k[3] of n
// doubles each.  A shared step has no criterion or level, so the components are
// independent: three short FP64 chains in parallel instead of the general
// corrector's one with its roots and division, and no kernel boundary between
// the reduction, the corrector, the copy of the state and the predictor
// (n = 4096: 7.5 + 11.0 + 2 + 4.7 us before).
template <bool DSW>
__global__ void __launch_bounds__(32 * kLanes)
    roll_step_kernel(const double *src, double *dst, const int n, const double *acc, const double *jerk,
                     const float *part, const int split, const CorrDt d, const bool predict, const JStream J,
                     DevStatus *st)
{
    const int idx = blockIdx.x * 32 + (threadIdx.x & 31);
    const bool live = idx < 3 * n;
    const int c = live ? idx / n : 0, i = live ? idx - c * n : 0;
    after_previous();
    double ap, kp;
    if (part) {
        constexpr int NC = DSW ? 14 : 7;
        double f[2];
        column_sums(split, [&](int r, int v, float &a, float &b) {
            const float *q = part + (static_cast<size_t>(r) * NC + 3 * v + c) * n + i;
            a = q[0];
            if (DSW) b = q[static_cast<size_t>(7) * n];
        }, f);
        ap = f[0];
        kp = f[1];
    }
    if (threadIdx.x >= 32 || !live) return;
    if (!part) {
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

// Between two force adjoints of the backward sweep, per (component, particle).
// After the first one (V.sb > 0) the totals of the last one, in the
// slots of part, join the gradients of the predicted state and the masses, and the
// transposed predictor leads to the gradients of the state the step began
// with.  Then, with `corrector`, the transposed corrector of the step before:
// from the gradients of the corrected state (gx, gv, ga, gk) to those of the
// predicted one (gxp, gvp), of the force (gA, gK, FP32) and of the start's a, k
// (left in ga, gk); without it the force at t = 0, whose upstream is (ga, gk)
// itself.  Last, the j-stream the force adjoint reads, at the prediction of
// that step from its state `src` (dt = 0 at t = 0).
__global__ void __launch_bounds__(32 * kLanes)
    adj_step_kernel(const float *part, const VjpSlots V, const DiffGrads G, const int n, const AdjDt d,
                    const bool corrector, const double *src, const JStream J)
{
    const int idx = blockIdx.x * 32 + (threadIdx.x & 31);
    const bool live = idx < 3 * n;
    const int c = live ? idx / n : 0, i = live ? idx - c * n : 0;
    after_previous();
    double t[3];
    if (V.sb > 0)
        column_sums(V.sb * V.parts + 1, [&](int s, int v, float &a, float &b) {
            if (v < 2 || c == 0) vjp_at_slot(part, V, n, v < 2 ? 3 * v + c : 6, i, s, a, b);
        }, t);
    if (threadIdx.x >= 32 || !live) return;
    const size_t e = static_cast<size_t>(idx), n3 = 3 * static_cast<size_t>(n);
    // (the component arrays of each gradient are contiguous: gx[0][e] is component c of particle i)
    double gx = G.gx[0][e], gv = G.gv[0][e], ga = G.ga[0][e], gk = G.gk[0][e];
    if (V.sb > 0) {
        const double tx = t[0], tv = t[1], tm = t[2];
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

// A launch whose blocks may start while the stream's previous kernel still runs; the
// kernel waits for that one in after_previous().
template <class... P, class... A>
cudaError_t launch_after(void (*kernel)(P...), const unsigned grid, const unsigned block, cudaStream_t s, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

int blocks_of(int64_t n, int t) { return static_cast<int>((n + t - 1) / t); }

}  // namespace

// Superblocks of 64 rows up to n = 8192 (128 of them), each pair of them in two
// parts while that leaves fewer warps than the GPU holds (up to n = 3776 on 152 SMs);
// more tiles per superblock beyond, their sums folded in double-single.
VjpSlots vjp_slots(int64_t n, int sm_count)
{
    VjpSlots V{};
    const int64_t tiles = (n + 64 * kVjpRows * 2 - 1) / (64 * kVjpRows * 2);
    V.rows = static_cast<int>(tiles) * kVjpRows;
    V.sb = static_cast<int>((n + V.rows - 1) / V.rows);
    V.two_word = tiles > 1;
    V.parts = tiles == 1 && static_cast<int64_t>(V.sb) * (V.sb + 1) / 2 < 12LL * sm_count ? 2 : 1;
    return V;
}

size_t vjp_scratch_bytes(int64_t n, int sm_count)
{
    const VjpSlots V = vjp_slots(n, sm_count);
    return (static_cast<size_t>(V.sb) * V.parts + 1) * (V.two_word ? 14 : 7) * static_cast<size_t>(n) * sizeof(float);
}

cudaError_t force_vjp_launch(const JStream &J, const DiffGrads &G, int64_t n, float eps2, int sm_count,
                             void *scratch, VjpSlots *slots, cudaStream_t s, int64_t *launches)
{
    const VjpSlots V = vjp_slots(n, sm_count);
    const unsigned units = static_cast<unsigned>(static_cast<int64_t>(V.sb) * (V.sb + 1) / 2 * V.parts);
    auto *kernel = V.two_word ? vjp_pairs_kernel<1, true> : V.parts == 2 ? vjp_pairs_kernel<2, false>
                                                                         : vjp_pairs_kernel<1, false>;
    ++*launches;
    *slots = V;
    return launch_after(kernel, units, 32, s, J.posm, J.vel, G.gA, G.gK, static_cast<int>(n), eps2, V.sb,
                        V.rows / kVjpRows, static_cast<float *>(scratch));
}

cudaError_t vjp_finish_launch(const DiffGrads &G, int64_t n, const void *scratch, const VjpSlots &slots, cudaStream_t s,
                              int64_t *launches)
{
    vjp_reduce_kernel<<<blocks_of(7 * n, 32), 32 * kLanes, 0, s>>>(static_cast<const float *>(scratch), slots,
                                                            static_cast<int>(n), G);
    ++*launches;
    return cudaGetLastError();
}

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
    auto *kernel = two_word ? roll_step_kernel<true> : roll_step_kernel<false>;
    ++*launches;
    return launch_after(kernel, blocks_of(3 * n, 32), 32 * kLanes, s, src, dst, static_cast<int>(n), acc, jerk, part,
                        split, d, predict, J, st);
}

cudaError_t adj_step_launch(const void *scratch, const VjpSlots &slots, const DiffGrads &G, int64_t n, double dt, bool corrector,
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
    ++*launches;
    return launch_after(adj_step_kernel, blocks_of(3 * n, 32), 32 * kLanes, s, static_cast<const float *>(scratch),
                        slots, G, static_cast<int>(n), d, corrector, src, J);
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
