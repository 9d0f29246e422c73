// The double-single force of all particles by unordered pairs: the pair term of
// ds_arith.cuh once per pair, for both of its particles, on packed FP32 (two
// rows per register, force_x2.cuh).
//
// Units, turns, slots and the sum over the slots are those of force_sym.cuh, with
// one warp per CTA, 64 rows per warp (rows l and l + 32 in lane l) and 64-row
// tiles.  Every value is a (hi, lo) pair; the sums of both sides take 8 terms
// with TwoSum on the high words and the low words added in FP32 before they are
// renormalised (32 terms: the potential's error 2.7e-14 instead of 0.8e-14 at
// n = 16384), and join their slot as a pair.
//
// An unordered pair takes about 410 FP32 operations, 205 per interaction (the
// one-sided loop 325, 396 before its products joined their sums unnormalised).
// Bound by the FMA pipe and its operand reads (force_sym.cuh): about 815 + 90 cycles
// of two pairs' 1140 measured; 8 to 12 resident warps make no difference.  Full
// forces, one-sided -> pairs, us: n = 4096 303 -> 196, 16384 3340 -> 1967, 30000
// 11151 -> 6656 (before the mass came first).
//
// The assembler fuses a packed product into a packed addition that uses it, also
// where both are written as separate round-to-nearest instructions; a product
// whose rounding error is kept (FMA form) would then count that error twice.
// Each such product leaves through an XOR with a sign mask the compiler cannot
// see (it is negated by it), and is subtracted.
#pragma once

#include "force_sym.cuh"

namespace nb {

constexpr int kSymDsRows = 64;

namespace dsx {

struct d2 {
    f2_t h, l;
};

// hi - b and its error, a - b exactly: Knuth's TwoSum for a - b.
__device__ __forceinline__ d2 two_diff(const f2_t a, const f2_t b)
{
    const f2_t s = f2_sub(a, b);
    const f2_t bb = f2_sub(s, a);
    return {s, f2_sub(f2_sub(a, f2_sub(s, bb)), f2_add(b, bb))};
}
__device__ __forceinline__ d2 fast_sum(const f2_t a, const f2_t b)  // |a| >= |b|
{
    const f2_t s = f2_add(a, b);
    return {s, f2_sub(b, f2_sub(s, a))};
}
__device__ __forceinline__ d2 diff(const d2 x, const d2 y)
{
    const d2 s = two_diff(x.h, y.h);
    return fast_sum(s.h, f2_add(s.l, f2_sub(x.l, y.l)));
}

// x y = -n + e: n the negated rounded product of the high words, e its error and
// the cross products (that of the low words, below 2^-48, is left out).
struct prod2 {
    f2_t n, e;
};
__device__ __forceinline__ prod2 prod(const d2 x, const d2 y, const f2_t sign)
{
    prod2 r;
    r.n = f2_opaque(f2_mul(x.h, y.h), sign);
    r.e = f2_fma(x.l, y.h, f2_fma(x.h, y.l, f2_fma(x.h, y.h, r.n)));
    return r;
}
__device__ __forceinline__ d2 norm(const prod2 p)  // |n| >> |e|
{
    const f2_t s = f2_sub(p.e, p.n);
    return {s, f2_sub(p.e, f2_add(s, p.n))};
}
// s += p, the low words unnormalised.
__device__ __forceinline__ void add(d2 &s, const prod2 p)
{
    const d2 t = two_diff(s.h, p.n);
    s.h = t.h;
    s.l = f2_add(s.l, f2_add(t.l, p.e));
}

struct Row {
    d2 x[3], v[3], m;
};

}  // namespace dsx

// One pair of particles i (two rows) and j, its terms added to the sums of both:
// si += m_j term, sj += m_i term with the signs of i (applied when folded).
template <bool DIAG>
__device__ __forceinline__ void sym_ds_pair(const dsx::Row &I, const dsx::Row &J, const dsx::d2 e2, const f2_t sign,
                                            const bool ma, const bool mb, dsx::d2 (&si)[7], dsx::d2 (&sj)[7])
{
    using namespace dsx;
    d2 dx[3], dv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        dx[c] = diff(J.x[c], I.x[c]);
        dv[c] = diff(J.v[c], I.v[c]);
    }
    d2 r2 = e2;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        prod2 q;
        q.n = f2_opaque(f2_mul(dx[c].h, dx[c].h), sign);
        q.e = f2_fma(f2_add(dx[c].h, dx[c].h), dx[c].l, f2_fma(dx[c].h, dx[c].h, q.n));
        add(r2, q);
    }
    r2 = fast_sum(r2.h, r2.l);
    // r^-1 = y0 (1 + rho/2 + 3 rho^2/8) and r^-2 = y0^2 (1 + rho + rho^2), rho = 1 - r^2 y0^2:
    // 1 - (the rounded product) is exact, so one word holds rho to 2^-46
    float a, b;
    f2_unpack(r2.h, a, b);
    if (DIAG) {  // r^-1 = 0 (the residual below is then taken at a finite r^2)
        a = ma ? INFINITY : a;
        b = mb ? INFINITY : b;
    }
    const f2_t one = f2_pack(1.0f, 1.0f);
    const f2_t y0 = f2_pack(rsqrt_mufu(a), rsqrt_mufu(b));
    const f2_t np = f2_opaque(f2_mul(y0, y0), sign);
    const f2_t pe = f2_fma(y0, y0, np), p = f2_sub(0ull, np);
    const f2_t nt = f2_opaque(f2_mul(r2.h, p), sign);
    const f2_t te = f2_fma(r2.h, pe, f2_fma(r2.l, p, f2_fma(r2.h, p, nt)));
    const f2_t rho = f2_sub(f2_add(one, nt), te);
    const f2_t half = f2_pack(0.5f, 0.5f), c38 = f2_pack(0.375f, 0.375f);
    const d2 y = fast_sum(y0, f2_mul(y0, f2_mul(rho, f2_fma(c38, rho, half))));
    const d2 y2 = fast_sum(p, f2_fma(p, f2_fma(rho, rho, rho), pe));
    // -3 (dx.dv) r^-2
    const f2_t m3 = f2_pack(-3.0f, -3.0f);
    prod2 q3;
    q3.n = f2_opaque(f2_mul(m3, y2.h), sign);
    q3.e = f2_fma(m3, y2.l, f2_fma(m3, y2.h, q3.n));
    const prod2 x0 = prod(dx[0], dv[0], sign);
    d2 xv = {f2_sub(0ull, x0.n), x0.e};
    add(xv, prod(dx[1], dv[1], sign));
    add(xv, prod(dx[2], dv[2], sign));
    xv = fast_sum(xv.h, xv.l);
    const d2 w = norm(prod(xv, norm(q3), sign));
    // (the mass first, as in ds_pair_term: r^-3 alone leaves FP32's range sooner)
    const prod2 mrI = prod(J.m, y, sign), mrJ = prod(I.m, y, sign);
    const d2 sI = norm(prod(norm(mrI), y2, sign)), sJ = norm(prod(norm(mrJ), y2, sign));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        d2 u = dv[c];
        add(u, prod(w, dx[c], sign));
        u = fast_sum(u.h, u.l);
        add(si[c], prod(sI, dx[c], sign));
        add(si[3 + c], prod(sI, u, sign));
        add(sj[c], prod(sJ, dx[c], sign));
        add(sj[3 + c], prod(sJ, u, sign));
    }
    add(si[6], mrI);
    add(sj[6], mrJ);
}

struct SymDsParams {
    const float4 *posm, *poslo, *vel, *vello;  // the rows, (hi, lo) of x and m, of v
    int n, n_sb, tiles;
    float eps2, eps2_lo;
    float *part;             // [n_sb + 1][14][n]
    const long long *skip;   // when set and not zero: nothing to do
    unsigned long long sign; // the sign bits of both halves
};

// Adds (x, xl) to the double-single sum of component c at p.
__device__ __forceinline__ void sym_ds_fold(float *p, const size_t n, const int c, const float x, const float xl,
                                            const bool first)
{
    float *h = p + static_cast<size_t>(c) * n, *l = p + static_cast<size_t>(7 + c) * n;
    float hi = first ? 0.0f : *h, lo = first ? 0.0f : *l;
    ds2_add(hi, lo, x, xl);
    const dsa::ds r = dsa::fast_two_sum(hi, lo);
    *h = r.h;
    *l = r.l;
}

__global__ void __launch_bounds__(32, 11) force_sym_ds_kernel(const SymDsParams P)
{
    using namespace dsx;
    __shared__ float4 sj[4][32];
    if (P.skip && *P.skip != 0) return;
    const int lane = threadIdx.x, n = P.n;
    const int u = blockIdx.x;
    int J = static_cast<int>((sqrtf(8.0f * u + 1.0f) - 1.0f) * 0.5f);
    while ((J + 1) * (J + 2) / 2 <= u) ++J;
    while (J * (J + 1) / 2 > u) --J;
    const int I = u - J * (J + 1) / 2;
    const bool diag = I == J;
    const size_t slot = static_cast<size_t>(14) * n;
    float *pi_out = P.part + slot * J, *pj_out = P.part + slot * (diag ? P.n_sb : I);
    const int sb = P.tiles * kSymDsRows;
    const int j_end = min(n, (J + 1) * sb);
    const d2 e2 = {f2_pack(P.eps2, P.eps2), f2_pack(P.eps2_lo, P.eps2_lo)};
    const f2_t sign = P.sign;
    const float4 far = make_float4(kPadPosition, kPadPosition, kPadPosition, 0.f), zero = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i0 = I * sb; i0 < min(n, (I + 1) * sb); i0 += kSymDsRows) {
        const int r0 = i0 + lane, r1 = r0 + 32;
        Row R;
        {
            const float4 x0 = r0 < n ? P.posm[r0] : far, x1 = r1 < n ? P.posm[r1] : far;
            const float4 l0 = r0 < n ? P.poslo[r0] : zero, l1 = r1 < n ? P.poslo[r1] : zero;
            const float4 v0 = r0 < n ? P.vel[r0] : zero, v1 = r1 < n ? P.vel[r1] : zero;
            const float4 w0 = r0 < n ? P.vello[r0] : zero, w1 = r1 < n ? P.vello[r1] : zero;
            R.x[0] = {f2_pack(x0.x, x1.x), f2_pack(l0.x, l1.x)};
            R.x[1] = {f2_pack(x0.y, x1.y), f2_pack(l0.y, l1.y)};
            R.x[2] = {f2_pack(x0.z, x1.z), f2_pack(l0.z, l1.z)};
            R.m = {f2_pack(x0.w, x1.w), f2_pack(l0.w, l1.w)};
            R.v[0] = {f2_pack(v0.x, v1.x), f2_pack(w0.x, w1.x)};
            R.v[1] = {f2_pack(v0.y, v1.y), f2_pack(w0.y, w1.y)};
            R.v[2] = {f2_pack(v0.z, v1.z), f2_pack(w0.z, w1.z)};
        }
        bool ifirst = true;
        for (int j0 = diag ? i0 : J * sb; j0 < j_end; j0 += 32) {
            __syncwarp();
            const int j = j0 + lane;
            sj[0][lane] = j < n ? P.posm[j] : far;
            sj[1][lane] = j < n ? P.poslo[j] : zero;
            sj[2][lane] = j < n ? P.vel[j] : zero;
            sj[3][lane] = j < n ? P.vello[j] : zero;
            __syncwarp();
            d2 si[7], sq[7];
#pragma unroll
            for (int c = 0; c < 7; ++c) si[c] = sq[c] = {0ull, 0ull};
            auto turn = [&](auto own) {
                constexpr bool OWN = decltype(own)::value;
#pragma unroll 1
                for (int s = 0; s < 32; ++s) {
                    if ((s & 7) == 7) {
#pragma unroll
                        for (int c = 0; c < 7; ++c) {
                            si[c] = fast_sum(si[c].h, si[c].l);
                            sq[c] = fast_sum(sq[c].h, sq[c].l);
                        }
                    }
                    const int jl = (lane + s) & 31;
                    const float4 x = sj[0][jl], xl = sj[1][jl], v = sj[2][jl], vl = sj[3][jl];
                    Row Q;
                    Q.x[0] = {f2_pack(x.x, x.x), f2_pack(xl.x, xl.x)};
                    Q.x[1] = {f2_pack(x.y, x.y), f2_pack(xl.y, xl.y)};
                    Q.x[2] = {f2_pack(x.z, x.z), f2_pack(xl.z, xl.z)};
                    Q.m = {f2_pack(x.w, x.w), f2_pack(xl.w, xl.w)};
                    Q.v[0] = {f2_pack(v.x, v.x), f2_pack(vl.x, vl.x)};
                    Q.v[1] = {f2_pack(v.y, v.y), f2_pack(vl.y, vl.y)};
                    Q.v[2] = {f2_pack(v.z, v.z), f2_pack(vl.z, vl.z)};
                    sym_ds_pair<OWN>(R, Q, e2, sign, OWN && j0 + jl <= r0, OWN && j0 + jl <= r1, si, sq);
#pragma unroll
                    for (int c = 0; c < 7; ++c) {  // j's sums go to the lane that takes it next
                        float a, b;
                        f2_unpack(sq[c].h, a, b);
                        sq[c].h = f2_pack(__shfl_sync(0xffffffffu, a, (lane + 1) & 31),
                                          __shfl_sync(0xffffffffu, b, (lane + 1) & 31));
                        f2_unpack(sq[c].l, a, b);
                        sq[c].l = f2_pack(__shfl_sync(0xffffffffu, a, (lane + 1) & 31),
                                          __shfl_sync(0xffffffffu, b, (lane + 1) & 31));
                    }
                }
            };
            if (diag && j0 < i0 + kSymDsRows)
                turn(std::true_type());
            else
                turn(std::false_type());
#pragma unroll
            for (int c = 0; c < 7; ++c) {
                float h0, h1, l0, l1;
                f2_unpack(sq[c].h, h0, h1);
                f2_unpack(sq[c].l, l0, l1);
                ds2_add(h0, l0, h1, l1);  // the two rows' halves
                if (j < j_end) sym_ds_fold(pj_out + j, n, c, -h0, -l0, i0 == I * sb);
                f2_unpack(si[c].h, h0, h1);
                f2_unpack(si[c].l, l0, l1);
                const float s = c == 6 ? -1.0f : 1.0f;
                if (r0 < n) sym_ds_fold(pi_out + r0, n, c, s * h0, s * l0, ifirst);
                if (r1 < n) sym_ds_fold(pi_out + r1, n, c, s * h1, s * l1, ifirst);
            }
            ifirst = false;
        }
    }
}

}  // namespace nb
