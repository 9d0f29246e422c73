// Device-side steps shared by the single-system and the ensemble kernels:
// the predictor of one component, the corrector of one particle with the
// Aarseth time step and the power-of-two level rule (Portegies Zwart,
// Belleman & Geldof 2007, Sect. 2), and block-wide reductions.
#pragma once

#include "nbody_internal.cuh"

namespace nb {

// Step factors of the predictor: dt/2 (exact) and dt/3.
struct PredDt {
    double dt, half, third;
};
__device__ __forceinline__ PredDt pred_dt(const double dt) { return {dt, 0.5 * dt, __dmul_rn(dt, 1.0 / 3.0)}; }

// Predictor of Sect. 2 for one component, in Horner form with explicit
// roundings so that the predictor and the corrector kernels give the same
// bits:  x_p = x + dt (v + dt/2 (a + dt/3 k)),  v_p = v + dt (a + dt/2 k),
// i.e. x + v dt + a dt^2/2 + k dt^3/6 and v + a dt + k dt^2/2 in five fused
// multiply-adds (GB300's FP64 pipe is ~1/75 of its FP32 pipe).
__device__ __forceinline__ void predict_dim(double x, double v, double a, double k, const PredDt &d,
                                            double &xp, double &vp)
{
    xp = __fma_rn(d.dt, __fma_rn(d.half, __fma_rn(d.third, k, a), v), x);
    vp = __fma_rn(d.dt, __fma_rn(d.half, k, a), v);
}

// Round-to-nearest-even double -> float, and exact float -> double, on the
// integer pipe: GB300 converts at the FP64 rate (~1.8 per clock per SM, the
// predictor's bound).  IEEE 754 binary64 -> binary32: the 52-bit fraction keeps
// its top 23 bits, rounded by the 29 dropped ones (ties to even); a carry out
// of the fraction moves into the exponent, which the addition below does.
// Results outside the normal float range (zero, subnormal, overflow, Inf, NaN)
// take the hardware conversion; every value the predictor writes is normal or
// zero.
__device__ __forceinline__ float d2f_rn(const double d)
{
    const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(d));
    const int ef = static_cast<int>((b >> 52) & 0x7ffull) - 1023 + 127;
    if (ef < 1 || ef > 254) return __double2float_rn(d);
    const unsigned long long frac = b & ((1ull << 52) - 1);
    unsigned int keep = static_cast<unsigned int>(frac >> 29);
    const unsigned int rest = static_cast<unsigned int>(frac & ((1u << 29) - 1));
    keep += (rest > (1u << 28)) | ((rest == (1u << 28)) & (keep & 1u));
    const unsigned int bits = (static_cast<unsigned int>(b >> 63) << 31) + ((static_cast<unsigned int>(ef) << 23) + keep);
    return __uint_as_float(bits);
}

__device__ __forceinline__ double f2d(const float f)
{
    const unsigned int b = __float_as_uint(f);
    const unsigned int ef = (b >> 23) & 0xffu;
    if (ef == 0u || ef == 255u) return static_cast<double>(f);
    const unsigned long long bits = (static_cast<unsigned long long>(b >> 31) << 63) |
                                    (static_cast<unsigned long long>(ef - 127 + 1023) << 52) |
                                    (static_cast<unsigned long long>(b & 0x7fffffu) << 29);
    return __longlong_as_double(static_cast<long long>(bits));
}

// x^(-1/2) in FP64 with 5 operations on the FP64 pipe: the MUFU's approximation y0
// (relative error 2^-20.04 at most, measured) times the binomial series of
// (1 - e)^(-1/2) in e = 1 - x y0^2 to second order; |e| < 2^-19, so the third,
// 5 e^3/16, is below 2^-58.7.  y0 has 21 significant bits at most, so y0^2 is exact.
// With its roundings 1.015 x 2^-53 from the root (measured over the range; an IEEE
// root and division up to 1.5).  Arguments outside [2^-900, 2^900]
// (zero, subnormal, infinite, NaN) take the IEEE root and division.
__device__ __forceinline__ double rsqrt_f64(const double x)
{
    const unsigned int ex = (static_cast<unsigned int>(__double2hiint(x)) >> 20) - 123u;  // (sign: out of range)
    if (ex > 1800u) return __ddiv_rn(1.0, __dsqrt_rn(x));
    double y0;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(x));
    const double e = __fma_rn(-x, __dmul_rn(y0, y0), 1.0);
    return __fma_rn(__dmul_rn(y0, e), __fma_rn(0.375, e, 0.5), y0);
}

// Neither infinite nor NaN, on the integer pipe.
__device__ __forceinline__ bool finite_f64(const double d)
{
    return (static_cast<unsigned int>(__double2hiint(d)) & 0x7ff00000u) != 0x7ff00000u;
}

__device__ __forceinline__ double norm3(const double *u)
{
    return sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
}

// Level L of the largest power of two 2^-L <= dt, clamped to [lmin, lmax];
// returns -1 for NaN.  *clamped is set when dt < 2^-lmax (incl. dt <= 0).
__device__ __forceinline__ int level_of(double dt, int lmin, int lmax, bool *clamped)
{
    *clamped = false;
    if (isnan(dt)) return -1;
    if (!(dt > 0.0)) {
        *clamped = true;
        return lmax;
    }
    if (isinf(dt)) return lmin;
    int e;
    frexp(dt, &e);  // dt = f 2^e with 1/2 <= f < 1, so 2^(e-1) <= dt < 2^e
    int L = 1 - e;
    if (L < lmin) L = lmin;
    if (L > lmax) {
        L = lmax;
        *clamped = true;
    }
    return L;
}

// State loads: through L2 only (CG, for state that another CTA of the same
// launch may have written since this SM last read it) or plain.
template <bool CG>
__device__ __forceinline__ double ld_state(const double *p)
{
    if constexpr (CG) return __ldcg(p);
    return *p;
}
template <bool CG>
__device__ __forceinline__ int64_t ld_state(const int64_t *p)
{
    if constexpr (CG) return static_cast<int64_t>(__ldcg(reinterpret_cast<const long long *>(p)));
    return *p;
}
template <bool CG>
__device__ __forceinline__ int8_t ld_state(const int8_t *p)
{
    if constexpr (CG) return static_cast<int8_t>(__ldcg(reinterpret_cast<const signed char *>(p)));
    return *p;
}

// Step quantities of the corrector of Sect. 2 for a step of `steps` ticks of
// 2^-lmax: dt, 1/dt, 1/dt^2, dt^3, dt^4 and the predictor's factors.
struct CorrDt {
    double dt, idt, idt2, dt3, dt4;
    PredDt pd;
};
__device__ __forceinline__ CorrDt corr_dt(const int64_t steps, const double tick, const int lmax)
{
    CorrDt d;
    // A step of 2^k ticks of 2^-lmax (every particle of a block): dt = 2^e with
    // e = k - lmax, and every quantity but dt/3 is a power of two, dt/3 that power
    // times the rounded 1/3.  They are built from exponent bits on the integer pipe
    // (the conversion and the products below, ~8 dependent operations of ~64 cycles
    // on the FP64 pipe, give the same bits).
    const int e = (__ffsll(steps) - 1) - lmax;
    if (steps > 0 && (steps & (steps - 1)) == 0 && e >= -250 && e <= 250) {
        auto pow2 = [](const int k) { return __longlong_as_double(static_cast<long long>(1023 + k) << 52); };
        d.dt = pow2(e);
        d.idt = pow2(-e);
        d.idt2 = pow2(-2 * e);
        d.dt3 = pow2(3 * e);
        d.dt4 = pow2(4 * e);
        d.pd = {d.dt, pow2(e - 1),
                __longlong_as_double(__double_as_longlong(1.0 / 3.0) + static_cast<long long>(e) * (1ll << 52))};
        return d;
    }
    d.dt = static_cast<double>(steps) * tick;
    d.idt = 1.0 / d.dt;
    d.idt2 = d.idt * d.idt;
    d.dt3 = d.dt * d.dt * d.dt;
    d.dt4 = d.dt3 * d.dt;
    d.pd = pred_dt(d.dt);
    return d;
}

// One component of the corrector: from x, v, a, k at the start of the step and
// the force ap, kp at the predicted state, the corrected xn, vn and a^(2), a^(3)
// at the end of the step.
__device__ __forceinline__ void corr_dim(const double x, const double v, const double a, const double k,
                                         const double ap, const double kp, const CorrDt &d, double &xn,
                                         double &vn, double &a2e, double &a3)
{
    double xp, vp;
    predict_dim(x, v, a, k, d.pd, xp, vp);
    const double da = a - ap;  // Delta a = a - a_p
    const double a2 = -6.0 * da * d.idt2 - (4.0 * k + 2.0 * kp) * d.idt;
    a3 = 12.0 * da * d.idt2 * d.idt + 6.0 * (k + kp) * d.idt2;
    // the Taylor coefficients 1/24, 1/120, 1/6 as products (an FP64 division
    // is a long dependent sequence on this part's narrow FP64 pipe)
    xn = xp + d.dt4 * (a2 * (1.0 / 24.0) + a3 * d.dt * (1.0 / 120.0));
    vn = vp + d.dt3 * (a2 * (1.0 / 6.0) + a3 * d.dt * (1.0 / 24.0));
    a2e = a2 + a3 * d.dt;  // a^(2) at the end of the step
}

__device__ __forceinline__ double square3(const double *u) { return __fma_rn(u[2], u[2], __fma_rn(u[1], u[1], u[0] * u[0])); }

// (a b)^(1/2) for a, b >= 0; products far from the middle of the range take the
// two roots one by one.
__device__ __forceinline__ double sqrt_product(const double a, const double b)
{
    const double p = a * b;
    const unsigned int ex = (static_cast<unsigned int>(__double2hiint(p)) >> 20) - 123u;
    return ex <= 1800u ? p * rsqrt_f64(p) : sqrt(a) * sqrt(b);
}

// Level of Eq. (timestep)'s dt = [eta (|a||a2| + |k|^2) / (|k||a3| + |a2|^2)]^(1/2)
// (as level_of) from the squared norms.  A level only needs floor(log2 dt): with
// numerator N and denominator D, floor(log2 (N / D)) is the difference of their
// exponents, less one where N's fraction is the smaller, and dt's exponent half of
// that, rounded down.  So neither a division nor the outer root is taken, and two
// roots of products replace the four norms': ~30 operations on the FP64 pipe (one
// unit per SM, ~64 cycles each in a dependent chain) where the four norms, the
// division and the root took over 100.
__device__ __forceinline__ int crit_level(const double a2, const double k2, const double s2, const double t2,
                                          const double eta, const int lmin, const int lmax, bool *clamped)
{
    const double num = eta * (sqrt_product(a2, s2) + k2), den = sqrt_product(k2, t2) + s2;
    const long long nb = __double_as_longlong(num), db = __double_as_longlong(den);
    const int ne = static_cast<int>(nb >> 52), de = static_cast<int>(db >> 52);  // (negative: sign set)
    if (ne < 1 || ne > 2046 || de < 1 || de > 2046)  // zero, subnormal, infinite, NaN
        return level_of(den == 0.0 ? static_cast<double>(INFINITY) : sqrt(num / den), lmin, lmax, clamped);
    const long long frac = (1ll << 52) - 1;
    const int lq = ne - de - ((nb & frac) < (db & frac) ? 1 : 0);
    const int L = -(lq >> 1);
    *clamped = L > lmax;
    return L < lmin ? lmin : L > lmax ? lmax : L;
}

// Eq. (timestep) from |a|^2, |k|^2, |a^(2)|^2, |a^(3)|^2 at the end of the step,
// then the level rule: shrink at once, grow one level when the new time allows.
// Raises the non-finite and dt_min flags; returns the new level.
__device__ __forceinline__ int corr_level(const double a2, const double k2, const double s2, const double t2,
                                          const double eta, const int lmin, const int lmax, const int l_old,
                                          const int64_t t_new, const bool finite, DevStatus *st)
{
    bool clamped = false;
    const int lc = crit_level(a2, k2, s2, t2, eta, lmin, lmax, &clamped);
    int l_new;
    if (!finite || lc < 0) {
        l_new = lmax;
        atomicOr(&st->flags, kFlagNonfinite);
        atomicAdd(&st->nonfinite, 1ull);
    } else if (lc >= l_old) {
        l_new = lc;  // shrink at once (or keep)
    } else {
        // grow one level, only if the new time is a multiple of twice the old step
        const int64_t two_old = int64_t(2) << (lmax - l_old);
        l_new = (l_old - 1 >= lmin && (t_new & (two_old - 1)) == 0) ? l_old - 1 : l_old;
    }
    if (clamped) {
        atomicOr(&st->flags, kFlagDtMin);
        atomicAdd(&st->below_min, 1ull);
    }
    return l_new;
}

// Where the corrector and the predictor find particle i's state: the State's global
// arrays (CG: loads through L2 only), or a copy of the particles lo .. in shared
// memory, 13 arrays of 8-byte words (x, v, a, k by component, then t) and one of levels.
template <bool CG>
struct GlobalRows {
    const State &S;
    __device__ __forceinline__ double x(const int c, const int64_t i) const { return ld_state<CG>(S.x[c] + i); }
    __device__ __forceinline__ double v(const int c, const int64_t i) const { return ld_state<CG>(S.v[c] + i); }
    __device__ __forceinline__ double a(const int c, const int64_t i) const { return ld_state<CG>(S.a[c] + i); }
    __device__ __forceinline__ double k(const int c, const int64_t i) const { return ld_state<CG>(S.k[c] + i); }
    __device__ __forceinline__ int64_t t(const int64_t i) const { return ld_state<CG>(S.t + i); }
    __device__ __forceinline__ int level(const int64_t i) const { return ld_state<CG>(S.level + i); }
    __device__ __forceinline__ void put(const int c, const int64_t i, const double x, const double v, const double a,
                                        const double k) const
    {
        S.x[c][i] = x;
        S.v[c][i] = v;
        S.a[c][i] = a;
        S.k[c][i] = k;
    }
    __device__ __forceinline__ void put_time(const int64_t i, const int64_t t, const int level) const
    {
        S.t[i] = t;
        S.level[i] = static_cast<int8_t>(level);
    }
};

constexpr int kRowWords = 13;  // 8-byte words of a particle's state besides its level
template <int STRIDE>
struct SharedRows {
    double *w;  // word q of particle i at w[q STRIDE + i - lo]
    int lo;
    __device__ __forceinline__ double x(const int c, const int64_t i) const { return w[c * STRIDE + static_cast<int>(i) - lo]; }
    __device__ __forceinline__ double v(const int c, const int64_t i) const { return w[(3 + c) * STRIDE + static_cast<int>(i) - lo]; }
    __device__ __forceinline__ double a(const int c, const int64_t i) const { return w[(6 + c) * STRIDE + static_cast<int>(i) - lo]; }
    __device__ __forceinline__ double k(const int c, const int64_t i) const { return w[(9 + c) * STRIDE + static_cast<int>(i) - lo]; }
    __device__ __forceinline__ int64_t t(const int64_t i) const { return __double_as_longlong(w[12 * STRIDE + static_cast<int>(i) - lo]); }
    __device__ __forceinline__ int8_t *levels() const { return reinterpret_cast<int8_t *>(w + kRowWords * STRIDE); }
    __device__ __forceinline__ int level(const int64_t i) const { return levels()[static_cast<int>(i) - lo]; }
    __device__ __forceinline__ void put(const int c, const int64_t i, const double x, const double v, const double a,
                                        const double k) const
    {
        double *p = w + c * STRIDE + static_cast<int>(i) - lo;
        p[0] = x;
        p[3 * STRIDE] = v;
        p[6 * STRIDE] = a;
        p[9 * STRIDE] = k;
    }
    __device__ __forceinline__ void put_time(const int64_t i, const int64_t t, const int level) const
    {
        w[12 * STRIDE + static_cast<int>(i) - lo] = __longlong_as_double(t);
        levels()[static_cast<int>(i) - lo] = static_cast<int8_t>(level);
    }
};

// Corrector of Sect. 2 for particle i (its forces at the predicted state in
// ap_in[3], kp_in[3]), then Eq. (timestep) and the new level; the step ends
// at tick t_new.  Updates x, v, a, k, t, level of i and returns the new level.
template <class Rows>
__device__ __forceinline__ int correct_row_at(const Rows &R, const int64_t i, const double *ap_in, const double *kp_in,
                                              const int64_t t_new, const double tick, const double eta, const int lmin,
                                              const int lmax, DevStatus *st)
{
    const int l_old = R.level(i);
    const CorrDt d = corr_dt(t_new - R.t(i), tick, lmax);
    double ap[3], kp[3], a2e[3], a3[3];
    bool finite = true;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        ap[c] = ap_in[c];
        kp[c] = kp_in[c];
        double xn, vn;
        corr_dim(R.x(c, i), R.v(c, i), R.a(c, i), R.k(c, i), ap[c], kp[c], d, xn, vn, a2e[c], a3[c]);
        finite = finite && finite_f64(xn) && finite_f64(vn) && finite_f64(ap[c]) && finite_f64(kp[c]);
        R.put(c, i, xn, vn, ap[c], kp[c]);
    }
    // Eq. (timestep) with end-of-step quantities.
    const int l_new = corr_level(square3(ap), square3(kp), square3(a2e), square3(a3), eta, lmin, lmax, l_old, t_new,
                                 finite, st);
    R.put_time(i, t_new, l_new);
    return l_new;
}
__device__ __forceinline__ int correct_row(const State &S, const int64_t i, const double *ap_in, const double *kp_in,
                                           const int64_t t_new, const double tick, const double eta, const int lmin,
                                           const int lmax, DevStatus *st)
{
    return correct_row_at(GlobalRows<false>{S}, i, ap_in, kp_in, t_new, tick, eta, lmin, lmax, st);
}

// Block-wide reduction; `id` is the identity of `op` (pads missing warps).
template <typename T, typename Op>
__device__ __forceinline__ T block_reduce(T v, Op op, T *sh, T id)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    const int nw = blockDim.x >> 5;
    v = static_cast<int>(threadIdx.x) < nw ? sh[threadIdx.x] : id;
    if (w == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (l == 0) sh[0] = v;
    }
    __syncthreads();
    v = sh[0];
    __syncthreads();
    return v;
}

// Minimum over the warp, in every lane: the high words first, then the low words of
// the lanes that have the smallest (two warp reductions instead of ten shuffles).
__device__ __forceinline__ unsigned long long warp_min(const unsigned long long v)
{
    const unsigned hi = static_cast<unsigned>(v >> 32), lo = static_cast<unsigned>(v);
    const unsigned mh = __reduce_min_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_min_sync(0xffffffffu, hi == mh ? lo : ~0u);
    return static_cast<unsigned long long>(mh) << 32 | ml;
}

// Minimum over the block, in every thread, with one barrier.  sh: one word per warp,
// not stored to again before the block's next barrier.
__device__ __forceinline__ unsigned long long block_min(unsigned long long v, unsigned long long *sh)
{
    v = warp_min(v);
    const int lane = threadIdx.x & 31;
    if (lane == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    return warp_min(lane < static_cast<int>(blockDim.x >> 5) ? sh[lane] : ~0ull);
}

struct MinOp {
    __device__ unsigned long long operator()(unsigned long long a, unsigned long long b) const { return a < b ? a : b; }
};
struct MaxOp {
    __device__ unsigned long long operator()(unsigned long long a, unsigned long long b) const { return a > b ? a : b; }
};
struct AddOp {
    __device__ double operator()(double a, double b) const { return a + b; }
};
struct SumOp {
    __device__ long long operator()(long long a, long long b) const { return a + b; }
};

}  // namespace nb
