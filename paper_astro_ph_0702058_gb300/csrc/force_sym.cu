// Launch of the force by unordered pairs (kernel in force_sym.cuh): when a block
// takes it, how it is cut, the rows and the particles outside the block as
// contiguous arrays, and the sum over the slots.
#include <cmath>
#include <type_traits>

#include "ds_arith.cuh"
#include "force_sym.cuh"
#include "force_sym_ds.cuh"

namespace nb {

cudaError_t force_dispatch_plain(const ForceParams &P, const ForceConfig &cfg, cudaStream_t s);
cudaError_t force_dispatch_comp(const ForceParams &P, const ForceConfig &cfg, cudaStream_t s);

namespace {

constexpr int kSymMaxSb = 128;             // superblocks
constexpr int64_t kSymMinRows = 8192;      // rows from which a block may take pairs
constexpr int64_t kSymMinPart = 20000;     // the same for a part of the particles
constexpr int64_t kSymDsMin = 4096;        // particles from which the double-single force may
constexpr int64_t kSymPartCap = int64_t(8) << 30;  // bytes of its slots
constexpr int kSymThreads = 256;
constexpr int kSymScan = 4 * kSymThreads;  // particles of a block of the compaction

// Resident warps per SM the registers are limited for, and the unroll factor of
// the pair loop.  Measured at n = 262144, ms: plain (with r^-3 first, sym_add_both) 12
// warps x 8 43.7, x 4 45.0, 16 warps (128 registers) x 4 45.4, x 8 44.9; compensated
// 16 x 8 53.1, x 4 54.3, 12 x 8 55.0, x 4 56.0; one-warp CTAs (n = 16384, us): plain
// 12 x 8 235, 16 x 4 231, compensated 12 x 8 280, 16 x 4 291.
template <int MODE, int W>
struct SymShape {
    static constexpr int unroll = 8, warps = MODE == kModeComp && W > 1 ? 16 : 12;
};

template <int MODE, int W>
cudaError_t sym_launch(const SymParams &P, const ForceConfig &cfg, cudaStream_t s)
{
    using Sh = SymShape<MODE, W>;
    const int units = cfg.sym_sb * (cfg.sym_sb + 1) / 2;
    force_sym_kernel<MODE, W, Sh::unroll, Sh::warps><<<units, 32 * W, 0, s>>>(P);
    return cudaGetLastError();
}

// Row q <- particle list[q] (a list with an index outside [0, n) or with a
// particle twice sets *rows_general to n_act); marks the block's particles.
__global__ void __launch_bounds__(kSymThreads)
    sym_gather_kernel(const float *__restrict__ soa, const long long stride, const int arrays,
                      const int32_t *__restrict__ list, const int n_act, const int n, float *__restrict__ rows,
                      const long long rows_stride, int *__restrict__ mark, long long *rows_general, DevStatus *st)
{
    const int q = blockIdx.x * kSymThreads + threadIdx.x;
    if (q >= n_act) return;
    const int idx = list[q];
    if (idx < 0 || idx >= n) {
        atomicOr(&st->flags, static_cast<unsigned>(kFlagBadIndex));
        st->bad_index = q;
        *rows_general = n_act;
        return;
    }
    if (atomicExch(mark + idx, 1) != 0) *rows_general = n_act;
    for (int a = 0; a < arrays; ++a) rows[a * rows_stride + q] = soa[a * stride + idx];
}

// The float4 streams of the rows (double-single mode), likewise.
__global__ void __launch_bounds__(kSymThreads)
    sym_gather_ds_kernel(const JStream J, const int32_t *__restrict__ list, const int n_act, const int n,
                         float4 *__restrict__ rows, int *__restrict__ mark, long long *rows_general, DevStatus *st)
{
    const int q = blockIdx.x * kSymThreads + threadIdx.x;
    if (q >= n_act) return;
    const int idx = list[q];
    if (idx < 0 || idx >= n) {
        atomicOr(&st->flags, static_cast<unsigned>(kFlagBadIndex));
        st->bad_index = q;
        *rows_general = n_act;
        return;
    }
    if (atomicExch(mark + idx, 1) != 0) *rows_general = n_act;
    rows[q] = J.posm[idx];
    rows[n_act + q] = J.poslo[idx];
    rows[2ll * n_act + q] = J.vel[idx];
    rows[3ll * n_act + q] = J.vello[idx];
}

// counts[b] <- particles of block b's kSymScan that are not marked.
__global__ void __launch_bounds__(kSymThreads) sym_count_kernel(const int *__restrict__ mark, const int n, int *counts)
{
    __shared__ int sh[kSymThreads / 32];
    int k = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int i = blockIdx.x * kSymScan + e * kSymThreads + threadIdx.x;
        k += i < n && mark[i] == 0;
    }
    k = __reduce_add_sync(0xffffffffu, k);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = k;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < kSymThreads / 32; ++w) t += sh[w];
        counts[blockIdx.x] = t;
    }
}

// The particles that are not marked, ascending, as contiguous arrays of at most n_out.
__global__ void __launch_bounds__(kSymThreads)
    sym_compact_kernel(const float *__restrict__ soa, const long long stride, const int arrays,
                       const int *__restrict__ mark, const int n, const int *__restrict__ counts,
                       float *__restrict__ out, const long long out_stride, const int n_out)
{
    // (and the massless far particles that fill the last tile)
    for (int e = n_out + static_cast<int>(blockIdx.x * kSymThreads + threadIdx.x); e < out_stride;
         e += gridDim.x * kSymThreads)
        for (int a = 0; a < arrays; ++a) out[a * out_stride + e] = a < 3 ? kPadPosition : 0.0f;
    __shared__ int sh[kSymThreads / 32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int before = 0;  // particles of the blocks before this one
    for (int b = t; b < static_cast<int>(blockIdx.x); b += kSymThreads) before += counts[b];
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0) sh[w] = before;
    __syncthreads();
    int base = 0;
    for (int k = 0; k < kSymThreads / 32; ++k) base += sh[k];
    for (int e = 0; e < 4; ++e) {
        const int i = blockIdx.x * kSymScan + e * kSymThreads + t;
        const bool hit = i < n && mark[i] == 0;
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        __syncthreads();
        if (lane == 0) sh[w] = __popc(m);
        __syncthreads();
        int pos = base + __popc(m & ((1u << lane) - 1u));
        for (int k = 0; k < kSymThreads / 32; ++k) {
            if (k < w) pos += sh[k];
            base += sh[k];
        }
        if (hit && pos < n_out)  // (a list with a particle twice leaves more)
            for (int a = 0; a < arrays; ++a) out[a * out_stride + pos] = soa[a * stride + i];
    }
}

// The sums of a row over the slots, in slot order: one thread per row and
// component, reads coalesced over the rows; double-single on the FP32 pipe.
template <int MODE>
__global__ void __launch_bounds__(256)
    force_sym_reduce_kernel(const float *__restrict__ part, const int slots, const int n, double *__restrict__ acc,
                            double *__restrict__ jerk, double *__restrict__ pot, const long long *rows_general,
                            const bool general)
{
    constexpr int NC = MODE == kModeComp ? 14 : 7;
    if (rows_general && (*rows_general != 0) != general) return;  // the other path's rows
    const int q = blockIdx.x * 256 + threadIdx.x;
    const int c = blockIdx.y;
    if (q >= n) return;
    float h = 0.0f, l = 0.0f;
#pragma unroll 8
    for (int s = 0; s < slots; ++s) {
        const float *b = part + (static_cast<size_t>(s) * NC + c) * n + q;
        ds2_add(h, l, b[0], MODE == kModeComp ? b[static_cast<size_t>(7) * n] : 0.0f);
        if (MODE == kModeComp) {  // (double-single mode: a low word left to grow would cost ~2 of its 46 bits)
            const dsa::ds r = dsa::fast_two_sum(h, l);
            h = r.h;
            l = r.l;
        }
    }
    const double t = static_cast<double>(h) + static_cast<double>(l);
    if (c < 3)
        acc[3 * static_cast<size_t>(q) + c] = t;
    else if (c < 6)
        jerk[3 * static_cast<size_t>(q) + c - 3] = t;
    else
        pot[q] = t;
}

// Few rows with many j-ranges, for a caller's own buffers: the sums and their
// order are those of reduce_partials_2d_kernel (8 rows x 32 lanes of one
// component per block); each result goes to the context and to the caller's
// device buffer in one kernel, where a copy each took ~2 us of a call's 35.
template <int MODE>
__global__ void __launch_bounds__(256)
    force_out_kernel(const float *__restrict__ part, const int split, const int n_act, double *__restrict__ acc,
                     double *__restrict__ jerk, double *__restrict__ pot, const ForceUser u)
{
    constexpr int NC = MODE == kModeComp ? 14 : 7, R = 8, L = 32;
    __shared__ float2 sh[L][R];
    const int row = threadIdx.x % R, w = threadIdx.x / R;
    const int c = blockIdx.y;
    const int q = blockIdx.x * R + row;
    float h = 0.0f, l = 0.0f;
    if (q < n_act)
#pragma unroll 4
        for (int sp = w; sp < split; sp += L) {
            const float *b = part + (static_cast<size_t>(sp) * NC + c) * n_act + q;
            ds2_add(h, l, b[0], MODE == kModeComp ? b[static_cast<size_t>(7) * n_act] : 0.0f);
        }
    sh[w][row] = make_float2(h, l);
    __syncthreads();
    if (w != 0 || q >= n_act) return;
#pragma unroll
    for (int k = 1; k < L; ++k) ds2_add(h, l, sh[k][row].x, sh[k][row].y);
    const double t = static_cast<double>(h) + static_cast<double>(l);
    const size_t e = c < 6 ? 3 * static_cast<size_t>(q) + c % 3 : static_cast<size_t>(q);
    (c < 3 ? acc : c < 6 ? jerk : pot)[e] = t;
    double *const o = c < 3 ? u.acc : c < 6 ? u.jerk : u.pot;
    if (o) o[e] = t;
}

// Scratch of a context: the general path's row count, the marks, the
// compaction's counts, then the rows and the other particles (together n).
struct SymScratch {
    long long *rows_general;
    int *mark, *counts;
    float *rows;
};
int64_t up4(const int64_t n) { return (n + 3) / 4 * 4; }
SymScratch sym_scratch(void *p, const int64_t n)
{
    SymScratch S;
    char *b = static_cast<char *>(p);
    S.rows_general = reinterpret_cast<long long *>(b);
    S.mark = reinterpret_cast<int *>(b + 16);
    S.counts = S.mark + up4(n);
    S.rows = reinterpret_cast<float *>(S.counts + up4(n / kSymScan + 1));
    return S;
}

}  // namespace

size_t sym_scratch_bytes(int64_t n)
{
    return 16 + sizeof(int) * (up4(n) + up4(n / kSymScan + 1)) + sizeof(float) * 16 * (n + 8 + kJTile);
}

// All particles take pairs from 8192 on (the kernels alone, one-sided -> pairs, us,
// plain / compensated: n = 8192 82 -> 67 / 96 -> 78; 4096: 30 -> 28 / 34 -> 33, left
// as it was); a caller's list, which is checked and gathered first (~30 us), from
// 16384 (251 -> 231 / 301 -> 280 per call).  Only pairs within a block are shared,
// so a part of the particles gains about 0.2 n_act / n of its time and pays ~25 us
// for the copies and the second kernel.  Measured (us): compensated 33536 of 65536
// rows 2228 -> 2129, 22000: 1481 -> 1474, 40001 of 100003 3962 -> 3834, 26000: 2646
// -> 2563, but 12000 of 32768 433 -> 460; plain 40001 of 100003 3391 -> 3163, 22000
// of 65536 1248 -> 1252.  So from 20000 rows and a quarter of the particles on.
// Superblocks are as small as 128 of them allow, for many units (8256 against 2080
// of twice the size: 4-5 % at n = 65536 and 262144), up to 8 GiB of slots (2^20
// compensated, before the pair loop's last changes: 889 ms with 7.6 GB, 920 with 4.3;
// now 853); CTAs of one warp up to 32768
// rows, of four above (n = 16384: 194 against 240 us plain; 65536: 2894 against 2804).
bool sym_plan(int mode, int64_t n_act, int64_t n, int sm_count, ForceConfig *cfg)
{
    if (mode == kModeDS) {
        // all particles only, from 4096 on (one unit per resident warp and more: 303 -> 196 us there);
        // 64-row tiles, one-warp CTAs
        if (n_act != n || n < kSymDsMin) return false;
        const int64_t slot = 14 * n * static_cast<int64_t>(sizeof(float));
        int64_t tiles = (n + kSymDsRows * kSymMaxSb - 1) / (kSymDsRows * kSymMaxSb), sb;
        for (;; ++tiles) {  // fewer superblocks until their slots fit; too few units end it at any n
            sb = (n + kSymDsRows * tiles - 1) / (kSymDsRows * tiles);
            if (sb * (sb + 1) / 2 < 12LL * sm_count) return false;
            if ((sb + 1) * slot <= kSymPartCap) break;
        }
        cfg->threads = 32;
        cfg->ipt = 2;
        cfg->jsub = 1;
        cfg->slice = 0;
        cfg->n_iblk = static_cast<int>(sb);
        cfg->split = static_cast<int>(sb + 1);
        cfg->tiles_per_split = static_cast<int>(tiles);
        cfg->sym_sb = static_cast<int>(sb);
        cfg->sym_ranges = 0;
        return true;
    }
    if (!NB_PACKED || (mode != kModePlain && mode != kModeComp)) return false;
    if (n_act < kSymMinRows || n_act > n || (n_act < n && (n_act < kSymMinPart || 4 * n_act < n))) return false;
    const int nc = two_word_sums(mode) ? 14 : 7;
    const int W = n_act <= 32768 ? 1 : 4;
    const int64_t bt = static_cast<int64_t>(W) * kSymRows;
    const int64_t n_out = n - n_act;
    const int64_t slot_bytes = static_cast<int64_t>(nc) * n_act * sizeof(float);
    int64_t ranges = 0;  // of the particles outside: as a one-sided force over them takes
    if (n_out > 0) {
        ForceConfig out{};
        if (force_choose(mode, n_act, (n_out + kJTile - 1) / kJTile * kJTile, sm_count, 256, 1, 0, &out) != NBODY_OK)
            return false;
        ranges = out.split;
    }
    const int res = (mode == kModeComp && W > 1 ? 16 : 12) / W;  // resident CTAs per SM (SymShape)
    const int64_t slots = static_cast<int64_t>(res) * sm_count;
    const int64_t t_min = (n_act + bt * kSymMaxSb - 1) / (bt * kSymMaxSb);
    bool found = false;
    double best = 0.0;
    for (int64_t tiles = t_min; !found || tiles <= t_min + t_min / 4; ++tiles) {
        const int64_t sb = (n_act + bt * tiles - 1) / (bt * tiles);
        const int64_t units = sb * (sb + 1) / 2;
        if (units < slots) break;  // too few units
        if ((sb + 1 + ranges) * slot_bytes > kSymPartCap) continue;
        // the last, partly filled wave: an SM that holds k of res CTAs works at
        // about 0.6, 0.87 and 0.97 of its rate with 1/4, 1/2 and 3/4 of them
        const double waves = static_cast<double>(units) / slots, whole = std::floor(waves);
        const double fill = waves - whole;
        const double last = fill == 0.0 ? 0.0 : fill <= 0.25 ? 0.42 : fill <= 0.5 ? 0.57 : fill <= 0.75 ? 0.77 : 1.0;
        const double cost = (whole + last) * static_cast<double>(tiles) * tiles;
        if (found && cost >= 0.99 * best) continue;
        found = true;
        best = cost;
        cfg->threads = 32 * W;
        cfg->ipt = 4;
        cfg->jsub = 1;
        cfg->slice = 0;
        cfg->n_iblk = static_cast<int>(sb);
        cfg->split = static_cast<int>(sb + 1 + ranges);
        cfg->tiles_per_split = static_cast<int>(tiles);
        cfg->sym_sb = static_cast<int>(sb);
        cfg->sym_ranges = static_cast<int>(ranges);
    }
    return found;
}

cudaError_t force_sym_launch(int mode, const JStream &js, int64_t n, const int32_t *active, int64_t n_act,
                             double eps2, const ForceConfig &cfg, bool ascending, double *acc, double *jerk,
                             double *pot, void *partials, void *scratch, const long long **rows_general,
                             DevStatus *st, cudaStream_t s, int64_t *launches)
{
    const SymScratch X = sym_scratch(scratch, n);
    const int na = static_cast<int>(n_act), nn = static_cast<int>(n), n_out = nn - na;
    const int arrays = mode == kModeComp ? 10 : 7;
    if (mode == kModeDS) {
        SymDsParams D{};
        D.posm = js.posm;
        D.poslo = js.poslo;
        D.vel = js.vel;
        D.vello = js.vello;
        D.n = na;
        D.n_sb = cfg.sym_sb;
        D.tiles = cfg.tiles_per_split;
        D.eps2 = static_cast<float>(eps2);
        D.eps2_lo = static_cast<float>(eps2 - static_cast<double>(D.eps2));
        D.part = static_cast<float *>(partials);
        D.sign = 0x8000000080000000ull;
        *rows_general = nullptr;
        if (!ascending) {
            const cudaError_t e = cudaMemsetAsync(scratch, 0, 16 + sizeof(int) * up4(n), s);
            if (e != cudaSuccess) return e;
            float4 *rows = reinterpret_cast<float4 *>(X.rows);
            sym_gather_ds_kernel<<<(na + kSymThreads - 1) / kSymThreads, kSymThreads, 0, s>>>(
                js, active, na, nn, rows, X.mark, X.rows_general, st);
            ++*launches;
            D.posm = rows;
            D.poslo = rows + n_act;
            D.vel = rows + 2 * n_act;
            D.vello = rows + 3 * n_act;
            D.skip = X.rows_general;
            *rows_general = X.rows_general;
        }
        force_sym_ds_kernel<<<cfg.sym_sb * (cfg.sym_sb + 1) / 2, 32, 0, s>>>(D);
        ++*launches;
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        return force_sym_reduce_launch(mode, D.part, cfg.split, n_act, acc, jerk, pot, D.skip, false, s, launches);
    }
    SymParams P{};
    P.n = na;
    P.n_sb = cfg.sym_sb;
    P.tiles = cfg.tiles_per_split;
    P.eps2 = static_cast<float>(eps2);
    P.part = static_cast<float *>(partials);
    P.soa = js.soa;
    P.stride = js.n_pad;
    P.st = st;
    *rows_general = nullptr;
    if (!ascending || n_out > 0) {
        cudaError_t e = cudaMemsetAsync(scratch, 0, 16 + sizeof(int) * up4(n), s);
        if (e != cudaSuccess) return e;
        P.soa = X.rows;
        P.stride = up4(n_act);
        sym_gather_kernel<<<(na + kSymThreads - 1) / kSymThreads, kSymThreads, 0, s>>>(
            js.soa, js.n_pad, arrays, active, na, nn, X.rows, P.stride, X.mark, X.rows_general, st);
        ++*launches;
        if (!ascending) {
            P.skip = X.rows_general;
            *rows_general = X.rows_general;
        }
        if (n_out > 0) {
            float *out = X.rows + kSoaArrays * P.stride;
            const long long out_pad = (n_out + kJTile - 1) / kJTile * kJTile;
            const int nb = (nn + kSymScan - 1) / kSymScan;
            sym_count_kernel<<<nb, kSymThreads, 0, s>>>(X.mark, nn, X.counts);
            sym_compact_kernel<<<nb, kSymThreads, 0, s>>>(js.soa, js.n_pad, arrays, X.mark, nn, X.counts, out, out_pad,
                                                          n_out);
            ForceParams Q{};
            Q.soa = out;
            Q.n_act = na;
            Q.n = nn;
            Q.n_tiles = static_cast<int>(out_pad / kJTile);
            Q.eps2 = P.eps2;
            Q.part = P.part + static_cast<size_t>(cfg.sym_sb + 1) * (mode == kModeComp ? 14 : 7) * na;
            Q.st = st;
            Q.rows = X.rows;
            Q.rows_stride = P.stride;
            Q.skip = P.skip;
            ForceConfig oc{};
            oc.threads = 256;
            oc.ipt = 1;
            oc.split = cfg.sym_ranges;
            oc.n_iblk = (na + 255) / 256;
            e = mode == kModeComp ? force_dispatch_comp(Q, oc, s) : force_dispatch_plain(Q, oc, s);
            if (e != cudaSuccess) return e;
            ++*launches;
            *launches += 2;
        }
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    cudaError_t e;
    if (mode == kModeComp)
        e = cfg.threads == 32 ? sym_launch<kModeComp, 1>(P, cfg, s) : sym_launch<kModeComp, 4>(P, cfg, s);
    else
        e = cfg.threads == 32 ? sym_launch<kModePlain, 1>(P, cfg, s) : sym_launch<kModePlain, 4>(P, cfg, s);
    if (e != cudaSuccess) return e;
    ++*launches;
    return force_sym_reduce_launch(mode, P.part, cfg.split, n_act, acc, jerk, pot, P.skip, false, s, launches);
}

cudaError_t force_out_launch(int mode, const float *part, int split, int64_t n_act, double *acc, double *jerk,
                             double *pot, const ForceUser &u, cudaStream_t s, int64_t *launches)
{
    const int na = static_cast<int>(n_act);
    auto *kernel = mode == kModeComp ? force_out_kernel<kModeComp> : force_out_kernel<kModePlain>;
    kernel<<<dim3((na + 7) / 8, 7), 256, 0, s>>>(part, split, na, acc, jerk, pot, u);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t force_sym_reduce_launch(int mode, const float *part, int slots, int64_t n_act, double *acc, double *jerk,
                                    double *pot, const long long *rows_general, bool general, cudaStream_t s,
                                    int64_t *launches)
{
    const int na = static_cast<int>(n_act);
    const dim3 grid((na + 255) / 256, 7);
    if (two_word_sums(mode))
        force_sym_reduce_kernel<kModeComp><<<grid, 256, 0, s>>>(part, slots, na, acc, jerk, pot, rows_general, general);
    else
        force_sym_reduce_kernel<kModePlain><<<grid, 256, 0, s>>>(part, slots, na, acc, jerk, pot, rows_general,
                                                                 general);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace nb
