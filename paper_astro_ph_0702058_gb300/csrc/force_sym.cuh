// Force of a large block by pairs: an unordered pair (i, j) of active particles
// is formed once and gives both particles their terms of Eq. (Force).
//
// The differences, r^2, r^-1, r^-2 and 3 (dx.dv) r^-2 of Appendix A's pair term
// are the same for (i, j) and (j, i) but for signs that cancel or flip, so the
// second force of a pair costs 9 more FP32 operations instead of 27 (33 in
// compensated mode): 36 (42) operations per unordered pair, packed two pairs to
// an instruction as in force_x2.cuh.
//
// Layout:
//   rows    the block's particles in list order, n of them, as a structure of
//           arrays (the j-stream itself when the block is all particles, else
//           a gathered copy); cut into n_sb superblocks of W x 128 x tiles rows.
//   unit    one CTA per unordered pair (I, J) of superblocks.  Units only share
//           read-only data, so their order does not matter.  The rows' pairs with
//           the particles outside the block are force_kernel_x2's (as more units
//           here, one-sided, they ran at 0.88 of its rate: 12 to 16 warps per SM
//           against 16 to 24).
//   warp    128 rows i, four per lane in two packed registers, against 128 j in
//           four turns of 32: in step s of a turn, lane l takes j = (l + s) mod
//           32 from shared memory; the sums of j move on by one lane per step
//           (a shuffle), so after 32 steps they hold 128 terms and are back at
//           lane j, while the rows' sums stay in registers.
//   window  the W warps of a CTA take the W chunks of 128 j of a tile in turn
//           (warp w chunk (k + w) mod W in window k), one block barrier per
//           window, so no two warps add to one j's sums at a time.
//   sums    FP32 over 128 terms (compensated: two of 64, added), folded into (hi, lo) by TwoSum (compensated) or
//           an FP32 sum (plain), as in force_x2.cuh.  The folded sums live in
//           the unit's own slots of `part`: the rows of I in slot J, those of J
//           in slot I (I = J: the second side in slot n_sb), the j-ranges outside
//           in the slots after.  Every row has every slot written once, and
//           force_sym_reduce_kernel adds them in slot order, so results do not
//           depend on scheduling.
// What bounds it: the register file.  A packed FMA of three different registers
// reads six 32-bit words and issues every 3 cycles, not 2 (measured: 3.01; 2.2
// where consecutive ones share an operand; scalar FMAs 1.0 each, but mixing
// them with packed ones costs their switch, 3344 against 2947 us at n = 65536
// plain).  17 of the 36 operations are such FMAs.
// Measured against the one-sided kernel (force_kernel_x2) with its reduction,
// full forces, us: n = 8192 plain 82 -> 67, compensated 96 -> 78; 16384: 251 ->
// 194, 301 -> 242; 65536: 3566 -> 2840, 4331 -> 3403; 262144: 55672 -> 44100,
// 66448 -> 53130.
// Two rows per lane instead of four (96 registers) took 3276 us at n = 65536
// plain; r^-2 from the MUFU reciprocal instead of a product 0.5-2 % more.
#pragma once

#include "force_x2.cuh"

namespace nb {

constexpr int kSymRows = 128;  // rows of a warp, and j of a chunk

struct SymParams {
    const float *soa;         // rows: x, y, z, m, vx, vy, vz (lx, ly, lz), `stride` floats each
    long long stride;
    int n;                    // rows
    int n_sb;                 // superblocks
    int tiles;                // W x 128-row tiles of a superblock
    float eps2;
    float *part;              // [n_sb + 1][7 or 14][n]
    const long long *skip;    // when set and not zero: nothing to do
    DevStatus *st;
};

// Four rows of a lane, two per packed register.
struct SymI {
    f2_t x[2], y[2], z[2], m[2], vx[2], vy[2], vz[2], lx[2], ly[2], lz[2];
};

// What two pair terms leave for the sums of both sides.
struct SymT {
    f2_t dx, dy, dz, ux, uy, uz, y, y2;
};

// Pair terms of two rows and one j: dx = x_j - x_i, y = r^-1, y2 = r^-2 and
// u = dv - 3 (dx.dv) r^-2 dx.  ma, mb: pairs to leave out (their terms are zero).
template <int MODE, bool MASK>
__device__ __forceinline__ void sym_term(const f2_t (&v)[10], const SymI &I, const int g, const f2_t E2,
                                         const f2_t NEG3, const bool ma, const bool mb, SymT &T)
{
    if (MODE == kModeComp) {
        T.dx = f2_add(f2_sub(v[0], I.x[g]), f2_sub(v[7], I.lx[g]));
        T.dy = f2_add(f2_sub(v[1], I.y[g]), f2_sub(v[8], I.ly[g]));
        T.dz = f2_add(f2_sub(v[2], I.z[g]), f2_sub(v[9], I.lz[g]));
    } else {
        T.dx = f2_sub(v[0], I.x[g]);
        T.dy = f2_sub(v[1], I.y[g]);
        T.dz = f2_sub(v[2], I.z[g]);
    }
    const f2_t dvx = f2_sub(v[4], I.vx[g]), dvy = f2_sub(v[5], I.vy[g]), dvz = f2_sub(v[6], I.vz[g]);
    const f2_t r2 = f2_fma(T.dz, T.dz, f2_fma(T.dy, T.dy, f2_fma(T.dx, T.dx, E2)));
    float a, b;
    f2_unpack(r2, a, b);
    if (MASK) {  // r^-1 = 0
        a = ma ? INFINITY : a;
        b = mb ? INFINITY : b;
    }
    T.y = f2_pack(rsqrt_mufu(a), rsqrt_mufu(b));
    const f2_t xv = f2_fma(T.dz, dvz, f2_fma(T.dy, dvy, f2_mul(T.dx, dvx)));
    T.y2 = f2_mul(T.y, T.y);
    const f2_t w = f2_mul(f2_mul(xv, T.y2), NEG3);
    T.ux = f2_fma(w, T.dx, dvx);
    T.uy = f2_fma(w, T.dy, dvy);
    T.uz = f2_fma(w, T.dz, dvz);
}

// m r^-3 dx, m r^-3 u and m r^-1 added to the sums of both sides (the signs of
// the j side and of the potential are applied when the sums are folded).  The
// mass comes first, as in force_x2.cuh: r^-3 alone leaves FP32's range for r
// above 2^42 or below 2^-42, where m r^-1 r^-2 need not (a cluster in metres).
// That is 6 products and additions of two registers where r^-3 first took 3 and
// 2 FMAs of three.  ORDER is the order the compiler does best with at the
// kernel's registers: 0 one side after the other (plain, four warps: n = 262144 44.1
// ms, 45.0 in order 2), 1 every product first and the sides' FMAs in turn
// (compensated, four warps at 128 registers: 53.1 ms, 53.7 in order 2, 56.2 and more
// spills in order 0), 2 every product first, then side by side (one-warp CTAs: n =
// 32000 plain 746 us, 758 in orders 0 and 1, compensated 886, 888 in order 1).  With
// r^-3 first they took 43.7 and 53.1 ms, 737 and 874 us.
__device__ __forceinline__ void sym_add(const f2_t s, const SymT &T, f2_t (&p)[7])
{
    p[0] = f2_fma(s, T.dx, p[0]);
    p[1] = f2_fma(s, T.dy, p[1]);
    p[2] = f2_fma(s, T.dz, p[2]);
    p[3] = f2_fma(s, T.ux, p[3]);
    p[4] = f2_fma(s, T.uy, p[4]);
    p[5] = f2_fma(s, T.uz, p[5]);
}
template <int ORDER>
__device__ __forceinline__ void sym_add_both(const f2_t mj, const f2_t mi, const SymT &T, f2_t (&pi)[7], f2_t (&pj)[7])
{
    if constexpr (ORDER == 0) {
        const f2_t a = f2_mul(mj, T.y);
        sym_add(f2_mul(a, T.y2), T, pi);
        pi[6] = f2_add(pi[6], a);
        const f2_t b = f2_mul(mi, T.y);
        sym_add(f2_mul(b, T.y2), T, pj);
        pj[6] = f2_add(pj[6], b);
    } else {
        const f2_t a = f2_mul(mj, T.y), b = f2_mul(mi, T.y);
        pi[6] = f2_add(pi[6], a);
        pj[6] = f2_add(pj[6], b);
        const f2_t s = f2_mul(a, T.y2), t = f2_mul(b, T.y2);
        if constexpr (ORDER == 2) {
            sym_add(s, T, pi);
            sym_add(t, T, pj);
        } else {
            pi[0] = f2_fma(s, T.dx, pi[0]);
            pj[0] = f2_fma(t, T.dx, pj[0]);
            pi[1] = f2_fma(s, T.dy, pi[1]);
            pj[1] = f2_fma(t, T.dy, pj[1]);
            pi[2] = f2_fma(s, T.dz, pi[2]);
            pj[2] = f2_fma(t, T.dz, pj[2]);
            pi[3] = f2_fma(s, T.ux, pi[3]);
            pj[3] = f2_fma(t, T.ux, pj[3]);
            pi[4] = f2_fma(s, T.uy, pi[4]);
            pj[4] = f2_fma(t, T.uy, pj[4]);
            pi[5] = f2_fma(s, T.uz, pi[5]);
            pj[5] = f2_fma(t, T.uz, pj[5]);
        }
    }
}

// Adds x to the sum of component c kept at p (component stride n).
template <int MODE>
__device__ __forceinline__ void sym_fold(float *p, const size_t n, const int c, const float x, const bool first)
{
    float *h = p + static_cast<size_t>(c) * n;
    if (MODE == kModeComp) {
        float *l = p + static_cast<size_t>(7 + c) * n;
        float hi = first ? 0.0f : *h, lo = first ? 0.0f : *l;
        fold_ds_rn(hi, lo, x);
        *h = hi;
        *l = lo;
    } else {
        *h = first ? x : __fadd_rn(*h, x);
    }
}

// Floats of a chunk of 128 j in shared memory: (x, y, z, m), (vx, vy, vz, lx)
// and, compensated, (ly, lz) of each.
template <int MODE>
__host__ __device__ constexpr int sym_chunk_floats()
{
    return (MODE == kModeComp ? 10 : 8) * kSymRows;
}

template <int MODE>
__device__ __forceinline__ void sym_load_j(const float *chunk, const int jl, f2_t (&v)[10])
{
    const float4 *q = reinterpret_cast<const float4 *>(chunk);
    const float4 a = q[jl], b = q[kSymRows + jl];
    v[0] = f2_pack(a.x, a.x);
    v[1] = f2_pack(a.y, a.y);
    v[2] = f2_pack(a.z, a.z);
    v[3] = f2_pack(a.w, a.w);
    v[4] = f2_pack(b.x, b.x);
    v[5] = f2_pack(b.y, b.y);
    v[6] = f2_pack(b.z, b.z);
    if (MODE == kModeComp) {
        const float2 c = reinterpret_cast<const float2 *>(chunk + 8 * kSymRows)[jl];
        v[7] = f2_pack(b.w, b.w);
        v[8] = f2_pack(c.x, c.x);
        v[9] = f2_pack(c.y, c.y);
    } else {
        v[7] = v[8] = v[9] = 0ull;
    }
}

// A warp's 128 rows against a chunk of 128 j, both sides.  DIAG: the chunk is
// the rows themselves, of which only the pairs j > i count.  pj_out: the sums
// of the chunk's j (jlive of them exist), component stride n.  Compensated: the
// rows' sums of the first 64 j wait at mid (14 x 32 words of the warp) and are added
// at the end, so an FP32 sum has 64 terms, as each half of force_x2.cuh's (128 terms
// in one made the error at n = 30000 11 % larger than the one-sided kernel's; folded
// twice as often through L2 instead, the full force at 2^20 took 880 ms, not 853).
template <int MODE, bool DIAG, int UNROLL, int ORDER>
__device__ __forceinline__ void sym_both(const float *chunk, const SymI &I, const int lane, const f2_t E2,
                                         const f2_t NEG3, f2_t (&pi)[2][7], float *pj_out, const int jlive,
                                         const size_t n, const bool jfirst, f2_t *mid)
{
#pragma unroll 1
    for (int r = 0; r < kSymRows; r += 32) {
        if (MODE == kModeComp && r == kSymRows / 2)
#pragma unroll
            for (int q = 0; q < 14; ++q) {
                mid[32 * q + lane] = pi[q / 7][q % 7];
                pi[q / 7][q % 7] = 0ull;
            }
        f2_t pj[7];
#pragma unroll
        for (int c = 0; c < 7; ++c) pj[c] = 0ull;
#pragma unroll UNROLL
        for (int s = 0; s < 32; ++s) {
            const int jl = r + ((lane + s) & 31);
            f2_t v[10];
            sym_load_j<MODE>(chunk, jl, v);
            SymT T[2];
#pragma unroll
            for (int g = 0; g < 2; ++g)
                sym_term<MODE, DIAG>(v, I, g, E2, NEG3, DIAG && jl <= lane + 64 * g, DIAG && jl <= lane + 64 * g + 32,
                                     T[g]);
#pragma unroll
            for (int g = 0; g < 2; ++g) sym_add_both<ORDER>(v[3], I.m[g], T[g], pi[g], pj);
            // j goes to the next lane down, and its sums with it
#pragma unroll
            for (int c = 0; c < 7; ++c) {
                float a, b;
                f2_unpack(pj[c], a, b);
                a = __shfl_sync(0xffffffffu, a, (lane + 1) & 31);
                b = __shfl_sync(0xffffffffu, b, (lane + 1) & 31);
                pj[c] = f2_pack(a, b);
            }
        }
        if (r + lane < jlive) {
#pragma unroll
            for (int c = 0; c < 7; ++c) {
                float a, b;
                f2_unpack(pj[c], a, b);
                sym_fold<MODE>(pj_out + r + lane, n, c, -(a + b), jfirst);
            }
        }
    }
    if (MODE == kModeComp)
#pragma unroll
        for (int q = 0; q < 14; ++q) pi[q / 7][q % 7] = f2_add(pi[q / 7][q % 7], mid[32 * q + lane]);
}

// Element e of array a of a structure of arrays of n; past its end a massless
// particle far from every other.
__device__ __forceinline__ float sym_val(const float *soa, const long long stride, const int n, const int a,
                                         const int e)
{
    return e < n ? soa[a * stride + e] : (a < 3 ? kPadPosition : 0.0f);
}

// WARPS: resident warps per SM the registers are limited for.
template <int MODE, int W, int UNROLL, int WARPS>
__global__ void __launch_bounds__(32 * W, WARPS / W) force_sym_kernel(const SymParams P)
{
    constexpr bool DSW = MODE == kModeComp;
    constexpr int NC = DSW ? 14 : 7, NA = DSW ? 10 : 7;
    constexpr int BT = W * kSymRows;  // rows of a tile
    constexpr int CH = sym_chunk_floats<MODE>();
    constexpr int ORDER = W == 1 ? 2 : DSW ? 1 : 0;  // (sym_add_both)
    __shared__ __align__(16) float sj[W * CH];
    __shared__ f2_t s_mid[DSW ? W * 14 * 32 : 1];
    f2_t *mid = s_mid + (DSW ? (threadIdx.x >> 5) * 14 * 32 : 0);
    if (P.skip && *P.skip != 0) return;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int n = P.n;
    const size_t slot = static_cast<size_t>(NC) * n;
    const f2_t E2 = f2_pack(P.eps2, P.eps2), NEG3 = f2_pack(-3.0f, -3.0f);

    // the unit: (I, J) with I <= J
    const int u = blockIdx.x;
    int J = static_cast<int>((sqrtf(8.0f * u + 1.0f) - 1.0f) * 0.5f);
    while ((J + 1) * (J + 2) / 2 <= u) ++J;
    while (J * (J + 1) / 2 > u) --J;
    const int I_sb = u - J * (J + 1) / 2;
    const bool diag = I_sb == J;
    if (!NB_CHECK(I_sb >= 0 && I_sb <= J && J < P.n_sb, P.st, 60)) return;
    float *pi_out = P.part + slot * J;
    float *pj_out = P.part + slot * (diag ? P.n_sb : I_sb);
    const int j_begin = J * P.tiles * BT, j_end = min(n, j_begin + P.tiles * BT);

    // j-tiles in groups: the sums of a group's j stay in L2 while every row tile passes
    // over them (large superblocks: 55 MB for all resident CTAs)
    constexpr int kGroup = 4 * BT;
    for (int g0 = j_begin; g0 < j_end; g0 += kGroup)
    for (int it = 0; it < P.tiles; ++it) {
        const int t0 = (I_sb * P.tiles + it) * BT;
        const int i0 = t0 + w * kSymRows;  // the warp's rows
        if (t0 >= n) break;
        if (diag && t0 >= g0 + kGroup) break;  // (of a superblock's own pairs, those with j >= i)
        SymI I;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const int e0 = i0 + lane + 64 * g, e1 = e0 + 32;
            f2_t q[10];
#pragma unroll
            for (int a = 0; a < NA; ++a)
                q[a] = f2_pack(sym_val(P.soa, P.stride, n, a, e0), sym_val(P.soa, P.stride, n, a, e1));
            I.x[g] = q[0];
            I.y[g] = q[1];
            I.z[g] = q[2];
            I.m[g] = q[3];
            I.vx[g] = q[4];
            I.vy[g] = q[5];
            I.vz[g] = q[6];
            if (DSW) {
                I.lx[g] = q[7];
                I.ly[g] = q[8];
                I.lz[g] = q[9];
            }
        }
        const int j_first = diag ? max(g0, t0) : g0;
        bool ifirst = g0 == j_begin || (diag && t0 >= g0);  // the rows' first j-tile in this unit
        for (int j0 = j_first; j0 < min(j_end, g0 + kGroup); j0 += BT) {
            __syncthreads();
            for (int e = tid; e < BT; e += 32 * W) {
                float *q = sj + (e / kSymRows) * CH;
                const int k = e % kSymRows;
                float v[10];
#pragma unroll
                for (int a = 0; a < NA; ++a) v[a] = sym_val(P.soa, P.stride, j_end, a, j0 + e);
                reinterpret_cast<float4 *>(q)[k] = make_float4(v[0], v[1], v[2], v[3]);
                reinterpret_cast<float4 *>(q)[kSymRows + k] = make_float4(v[4], v[5], v[6], DSW ? v[7] : 0.0f);
                if (DSW) reinterpret_cast<float2 *>(q + 8 * kSymRows)[k] = make_float2(v[8], v[9]);
            }
            const bool own = diag && j0 == t0;  // the tile of the rows themselves
            const int nk = own ? W / 2 + 1 : W;
            for (int k = 0; k < nk; ++k) {
                __syncthreads();
                const int c = (k + w) % W;
                const int jr = j0 + c * kSymRows;
                // (own: windows 0 .. W/2 meet every pair of chunks, the last one twice)
                if (i0 >= n || jr >= j_end || (own && k > 0 && 2 * k == W && w >= W / 2)) continue;
                f2_t pi[2][7];
#pragma unroll
                for (int g = 0; g < 2; ++g)
#pragma unroll
                    for (int q = 0; q < 7; ++q) pi[g][q] = 0ull;
                const bool jfirst = it == 0 && k == 0;  // (each chunk that exists meets a warp in window 0)
                if (own && k == 0)
                    sym_both<MODE, true, 1, ORDER>(sj + c * CH, I, lane, E2, NEG3, pi, pj_out + jr, j_end - jr, n,
                                                   jfirst, mid);
                else
                    sym_both<MODE, false, UNROLL, ORDER>(sj + c * CH, I, lane, E2, NEG3, pi, pj_out + jr, j_end - jr, n,
                                                         jfirst, mid);
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    const int r0 = i0 + lane + 64 * g, r1 = r0 + 32;
#pragma unroll
                    for (int q = 0; q < 7; ++q) {
                        float a, b;
                        f2_unpack(pi[g][q], a, b);
                        if (r0 < n) sym_fold<MODE>(pi_out + r0, n, q, q == 6 ? -a : a, ifirst);
                        if (r1 < n) sym_fold<MODE>(pi_out + r1, n, q, q == 6 ? -b : b, ifirst);
                    }
                }
                ifirst = false;
            }
        }
    }
}

}  // namespace nb
