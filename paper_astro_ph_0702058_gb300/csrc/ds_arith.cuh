// Double-single arithmetic on the FP32 pipe: a value is the unevaluated sum
// hi + lo of two floats (~46 significant bits).  Building blocks (Dekker 1971;
// Knuth TAOCP vol. 2, 4.2.2): TwoSum, Fast2Sum and the FMA form of the exact
// product, written with round-to-nearest intrinsics so that no operation is
// contracted or fused.  Used by the double-single force mode and the
// double-single potential of the energy diagnostic.
#pragma once

#include "ptx.cuh"

namespace nb {
namespace dsa {

struct ds {
    float h, l;
};

__device__ __forceinline__ ds two_sum(const float a, const float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

__device__ __forceinline__ ds fast_two_sum(const float a, const float b)  // |a| >= |b| or a == 0
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ ds ds_add(const ds x, const ds y)
{
    const ds s = two_sum(x.h, y.h);
    return fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(x.l, y.l)));
}

__device__ __forceinline__ ds ds_neg(const ds x) { return {-x.h, -x.l}; }

__device__ __forceinline__ ds ds_mul(const ds x, const ds y)
{
    const float p = __fmul_rn(x.h, y.h);
    float e = __fmaf_rn(x.h, y.h, -p);
    e = __fmaf_rn(x.h, y.l, e);
    e = __fmaf_rn(x.l, y.h, e);
    return fast_two_sum(p, e);
}

__device__ __forceinline__ ds ds_mul_f(const ds x, const float f)
{
    const float p = __fmul_rn(x.h, f);
    float e = __fmaf_rn(x.h, f, -p);
    e = __fmaf_rn(x.l, f, e);
    return fast_two_sum(p, e);
}

__device__ __forceinline__ ds ds_rsqrt(const ds r2)
{
    const float y0 = rsqrt_mufu(r2.h);
    const float p = __fmul_rn(y0, y0);
    const ds y0sq = {p, __fmaf_rn(y0, y0, -p)};      // exact
    const ds t = ds_mul(r2, y0sq);                    // 1 - rho
    const ds rho = ds_add({1.0f, 0.0f}, ds_neg(t));  // small: its hi carries the needed bits
    const float c = y0 * (rho.h * fmaf(0.375f, rho.h, 0.5f));
    return fast_two_sum(y0, c);
}

// x y as the rounded product of the high words, exactly, and the rest: its error
// and the cross products (unnormalised: |e| is a few ulp of h).
__device__ __forceinline__ ds ds_prod(const ds x, const ds y)
{
    const float p = __fmul_rn(x.h, y.h);
    return {p, __fmaf_rn(x.l, y.h, __fmaf_rn(x.h, y.l, __fmaf_rn(x.h, y.h, -p)))};
}

// x + p for a ds_prod p: unnormalised, and normalised.
__device__ __forceinline__ ds ds_acc(const ds x, const ds p)
{
    const ds s = two_sum(x.h, p.h);
    return {s.h, __fadd_rn(x.l, __fadd_rn(s.l, p.l))};
}
__device__ __forceinline__ ds ds_add_prod(const ds x, const ds p)
{
    const ds s = ds_acc(x, p);
    return fast_two_sum(s.h, s.l);
}

// One pair term of Appendix A in double-single arithmetic, j given by its
// (hi, lo) position and mass a, b = (x, y, z, m) and velocity u, w4 = (vx, vy, vz, .),
// i by xi, vi: dx = x_j - x_i, dv = v_j - v_i, r2 = eps2 + dx.dx, rinv = r2^-1/2,
// then a += m r^-3 dx, k += m r^-3 (dv - 3 (dx.dv) r^-2 dx), phi -= m r^-1 into
// sum[0..2], sum[3..5], sum[6].  About 325 FP32 operations: products that only
// join a sum are not normalised first, and r^-1 and r^-2 come from one residual,
// rho = 1 - r^2 y0^2 (1 minus the rounded product is exact, so one word holds rho
// to 2^-46): r^-1 = y0 (1 + rho/2 + 3 rho^2/8), r^-2 = y0^2 (1 + rho + rho^2).
__device__ __forceinline__ void ds_pair_term(const float4 a, const float4 b, const float4 u, const float4 w4,
                                             const ds (&xi)[3], const ds (&vi)[3], const ds eps2, ds (&sum)[7])
{
    const ds dx[3] = {ds_add({a.x, b.x}, ds_neg(xi[0])), ds_add({a.y, b.y}, ds_neg(xi[1])),
                      ds_add({a.z, b.z}, ds_neg(xi[2]))};
    const ds dv[3] = {ds_add({u.x, w4.x}, ds_neg(vi[0])), ds_add({u.y, w4.y}, ds_neg(vi[1])),
                      ds_add({u.z, w4.z}, ds_neg(vi[2]))};
    ds r2 = eps2, xv = ds_prod(dx[0], dv[0]);
#pragma unroll
    for (int c = 0; c < 3; ++c) r2 = ds_acc(r2, ds_prod(dx[c], dx[c]));
    r2 = fast_two_sum(r2.h, r2.l);
    xv = ds_acc(ds_acc(xv, ds_prod(dx[1], dv[1])), ds_prod(dx[2], dv[2]));
    xv = fast_two_sum(xv.h, xv.l);
    const float y0 = rsqrt_mufu(r2.h);
    const float p = __fmul_rn(y0, y0), pe = __fmaf_rn(y0, y0, -p);  // y0^2, exactly
    const float t = __fmul_rn(r2.h, p);
    const float te = __fmaf_rn(r2.h, pe, __fmaf_rn(r2.l, p, __fmaf_rn(r2.h, p, -t)));
    const float rho = __fsub_rn(__fsub_rn(1.0f, t), te);
    const ds rinv = fast_two_sum(y0, __fmul_rn(y0, __fmul_rn(rho, __fmaf_rn(0.375f, rho, 0.5f))));
    const ds rinv2 = fast_two_sum(p, __fmaf_rn(p, __fmaf_rn(rho, rho, rho), pe));
    const ds mr = ds_mul({a.w, b.w}, rinv);
    const ds mr3 = ds_mul(mr, rinv2);
    const ds w = ds_mul(xv, ds_mul_f(rinv2, -3.0f));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        sum[c] = ds_add_prod(sum[c], ds_prod(mr3, dx[c]));
        sum[3 + c] = ds_add_prod(sum[3 + c], ds_prod(mr3, ds_add_prod(dv[c], ds_prod(w, dx[c]))));
    }
    sum[6] = ds_add(sum[6], ds_neg(mr));
}

}  // namespace dsa
}  // namespace nb
