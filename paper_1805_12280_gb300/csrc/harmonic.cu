// Harmonic summing of a power plane: the stage that receives the plane from the
// FT-convolution module (Sec. 3 names it; read here as the incoherent harmonic sum).
//
// Rows of the plane are ordered by drift, z = y - c with c = (m-1)/2, and column bin0
// holds frequency bin 0 (for templates centred in a frame of F taps, bin0 = (F-1)/2).
// The k-th harmonic of a signal at bin r with drift z lies at bin k r with drift k z, so for
// the fundamental (r, z), r >= 1,
//     S_h(r, z) = sum_{k=1..h} P[c + k z][bin0 + k r],      h = 1, 2, 4, .., H,
// is defined where |h z| <= c and bin0 + h r <= n - 1, and every S_h above its level's
// threshold becomes a candidate.
//
// A thread takes Q fundamentals of one row, 256 apart: all loads of their harmonics are issued
// before the first is used, then each sum is formed in the order k = 1, 2, .., the running sum
// compared with the threshold at every power of two.  A block takes tiles of 256 Q consecutive
// fundamentals of one row (the k = 1 loads of a warp are one 128-byte line; the k-th are a
// k-strided gather over k lines).
//
// Planes narrower than 2^31 columns take one launch that walks the plane in slope windows (below)
// with code compiled for each number of harmonics that lie in the plane; crossings are staged
// per warp, with no block barrier.  85 x 2^22, 8 harmonics: 310 us, 1.68 GB of DRAM traffic (1.18
// planes), against 599 us and 3.40 GB when rows were launched in runs of equal harmonic
// count and every strided pass fetched its rows again; 32 harmonics 845 -> 404 us, one harmonic
// 276 -> 224 us, 65536 columns and 8 harmonics 55 -> 17 us per call (15 launches -> 1).  What bounds it:
// load latency at 16 warps per SM (issue 40 %, DRAM 80 % of the measured copy rate); three blocks per
// SM, with fewer loads in flight per thread, are slower.
// Planes of more than 513 rows, whose table has little room for windows, go by runs of rows with the
// same number of harmonics in the same launch.  Wider rows take the general kernel with 64-bit indexing.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstdio>
#include <type_traits>

#include "fdas_internal.cuh"

namespace fdas {
namespace {

constexpr int kHsThreads = 256;
constexpr int kHsStage = 256;                        // records staged per block and tile
constexpr int kHsMaxLevels = 6;                      // h = 1 .. 32

struct HsThresholds {
    float t[kHsMaxLevels];
};

struct HsLimits {   // r_lim[k] = (n - 1 - bin0) / k: harmonic k of r lies in the plane iff r <= r_lim[k]
    int r_lim[33];
};

// fundamentals per thread and tile: loads in flight per thread Q H = 64 (8 for H = 1)
template <int H>
__host__ __device__ constexpr int hs_per_thread()
{
    return H <= 8 ? 8 : 64 / H;
}

template <int H>
__global__ void __launch_bounds__(kHsThreads) harmonic_kernel(const float *__restrict__ P, int m, int64_t n,
                                                              int64_t bin0, int64_t tiles_per_row, HsThresholds thr,
                                                              fdas_harmonic_candidate *__restrict__ out,
                                                              int64_t max_cand, unsigned long long *__restrict__ count)
{
    constexpr int Q = hs_per_thread<H>();
    constexpr int64_t TILE = (int64_t)kHsThreads * Q;
    __shared__ fdas_harmonic_candidate stage[kHsStage];
    __shared__ unsigned n_staged, n_flush;
    __shared__ unsigned long long flush_base;
    const int c = (m - 1) / 2;
    const int64_t rmax = n - 1 - bin0;   // fundamentals r = 1 .. rmax
    const int64_t tiles = (int64_t)m * tiles_per_row;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int y = (int)(tile / tiles_per_row);
        const int z = y - c;
        const int az = z < 0 ? -z : z;
        const int kz = az == 0 ? H : min(H, c / az);   // harmonics whose drift k z lies in the plane
        const int64_t r0 = 1 + (tile - (int64_t)y * tiles_per_row) * TILE + threadIdx.x;
        const int64_t origin = (int64_t)c * n + bin0;   // cell of k = 0
        const int64_t step_z = (int64_t)z * n;
        if (threadIdx.x == 0) n_staged = 0;
        __syncthreads();
        float v[Q][H];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t r = r0 + q * kHsThreads;
            const int64_t step = step_z + r;   // from harmonic k to k + 1
#pragma unroll
            for (int k = 1; k <= H; ++k) {
                const bool in = k <= kz && (int64_t)k * r <= rmax;   // r <= rmax is the case k = 1
                v[q][k - 1] = in ? __ldg(P + origin + (int64_t)k * step) : 0.f;
            }
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t r = r0 + q * kHsThreads;
            float acc = 0.f;
#pragma unroll
            for (int k = 1; k <= H; ++k) {
                acc += v[q][k - 1];
                if ((k & (k - 1)) == 0) {   // level h = k
                    const int j = 31 - __clz(k);
                    if (k <= kz && (int64_t)k * r <= rmax && acc > thr.t[j]) {
                        fdas_harmonic_candidate rec;
                        rec.tpl = y;
                        rec.power = acc;
                        rec.bin = bin0 + r;
                        rec.nharm = k;
                        rec.reserved = 0;
                        const unsigned slot = atomicAdd(&n_staged, 1u);
                        if (slot < (unsigned)kHsStage) {
                            stage[slot] = rec;
                        } else {   // staging full: reserve this record on its own
                            const unsigned long long at = atomicAdd(count, 1ull);
                            if ((long long)at < max_cand) out[at] = rec;
                        }
                    }
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned ns = min(n_staged, (unsigned)kHsStage);
            n_flush = ns;
            flush_base = ns ? atomicAdd(count, (unsigned long long)ns) : 0ull;
        }
        __syncthreads();
        for (unsigned i = threadIdx.x; i < n_flush; i += kHsThreads)
            if ((long long)(flush_base + i) < max_cand) out[flush_base + i] = stage[i];
        __syncthreads();   // the stage is read before the next tile refills it
    }
}

// Planes of fewer than 2^31 columns: fundamentals, bins and the in-row offsets are 32-bit.
// Crossings are staged per warp (no block barrier: each warp runs its tiles at its own pace).  Their
// slots come from a ballot and the count of staged records is in a register of every lane, the same
// in all of them; a warp reserves its staged records with one atomic when the next ones may not fit.
// 85 x 2^22, thresholds that 1 / 5 / 20 % of the sums cross: one harmonic 243 / 372 / 1113 us, eight
// 399 / 607 / 1638, against 243 / 1253 / 3124 and 398 / 1752 / 4659 with slots from a shared counter
// and a global reservation of its own for each record past 64 of a tile.
constexpr int kWarpStage = 64;

// All lanes, after their last stores to `stage`; it is free again on return.
__device__ __forceinline__ void warp_flush(const fdas_harmonic_candidate *stage, unsigned staged, int lane,
                                           fdas_harmonic_candidate *__restrict__ out, int64_t max_cand,
                                           unsigned long long *__restrict__ count)
{
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(count, (unsigned long long)staged);
    base = __shfl_sync(0xffffffffu, base, 0);
    __syncwarp();
    for (unsigned i = lane; i < staged; i += 32)
        if ((long long)(base + i) < max_cand) out[base + i] = stage[i];
    __syncwarp();
}

// Slope windows.  Harmonic k of fundamental (r, z) lies in row k z at column k r: on the ray of
// slope r / |z| through (c, bin0).  The cells of all rows with slopes in (S_w, S_{w+1}] are therefore
// closed under the sums, and the plane is walked window by window: row |z| = a takes the
// fundamentals (a S_w, a S_{w+1}], and every harmonic it reads lies in the part of row k a that the
// same window reads as fundamentals, so all but the first read of a cell hit L2.  The z = 0 row
// (its harmonics lie in itself) comes first.  Windows of 64 MB (85 x 2^22, 8 / 32 harmonics: 16 MB 315 /
// 383 us, 32 MB 313 / 370, 64 MB 313 / 405, 128 MB 346 / 433, the whole plane at once 509 / 760).
constexpr int kHsMaxWin = 128, kHsMaxEntries = 2048;   // windows; (window, |z|) entries of one launch
constexpr size_t kHsTableBytes = sizeof(int4) * (kHsMaxEntries + 32);   // with the z = 0 row's
constexpr int64_t kHsWindowBytes = 64ll << 20;
struct HsWindows {
    int count;   // 0: the plane as a whole, by runs of rows with the same number of harmonics
    int slope[kHsMaxWin + 1];
};

// Fundamentals per thread of rows with kz harmonics: 48 to 64 loads in flight, and a bit per
// (fundamental, level) in one mask (85 x 2^22, 8 harmonics: 313 us; with 16 for kz = 1 and 8 for 2 and
// 3: 407; 8 for all of them: 533).
__host__ __device__ constexpr int hs_q(int kz) { return kz == 1 ? 48 : kz == 2 ? 24 : kz == 3 ? 16 : kz <= 8 ? 8 : 64 / kz; }
constexpr int kHsTall = 2, kHsCases = 32;   // tall tiles are compiled for kz <= kHsTall, as cases above kHsCases
__host__ __device__ constexpr int hs_levels(int kz) { return kz < 2 ? 1 : 1 + hs_levels(kz / 2); }

// One tile of 256 Q fundamentals r0 + threadIdx.x + 256 q <= rend of row z, compiled for
// exactly the KZ harmonics that lie in the plane's drift range.  The straight-line part only
// marks crossings in a mask; the marked ones are appended by one short loop, a record per lane and
// round, so that the bodies of all KZ stay small (with an append per sum the kernel was bound by
// instruction fetch).  `staged`: records in the warp's stage, before and after.
// TALL, for rows much shorter than 256 Q: the 256 fundamentals r0 + threadIdx.x of Q rows, from z inwards,
// `rend` of which belong to the run.
template <int KZ, int Q = hs_q(KZ), bool TALL = false>
__device__ __forceinline__ void hs_tile(const float *__restrict__ P, int c, int n, int bin0, int z, int r0, int rend,
                                        const HsThresholds &thr, const HsLimits &lim, fdas_harmonic_candidate *stage,
                                        unsigned &staged, fdas_harmonic_candidate *__restrict__ out, int64_t max_cand,
                                        unsigned long long *__restrict__ count)
{
    constexpr int LV = hs_levels(KZ);
    using Mask = std::conditional_t<(Q * LV > 32), uint64_t, uint32_t>;   // a bit per sum
    constexpr int BITS = Q * LV > 32 ? 6 : 5;
    const int rt = r0 + (int)threadIdx.x;
    float v[Q][KZ];
    Mask valid = ~Mask(0);   // bits of the sums that are defined
    const int64_t step = TALL ? (z < 0 ? n : -(int64_t)n) : kHsThreads;   // cells from q to q + 1
    if (TALL ? r0 + kHsThreads - 1 <= lim.r_lim[KZ] && rend >= Q
             : r0 + kHsThreads * Q - 1 <= min(lim.r_lim[KZ], rend)) {   // every harmonic of the tile lies in the plane
#pragma unroll
        for (int k = 1; k <= KZ; ++k) {
            const float *base = P + ((int64_t)(c + k * z) * n + bin0 + (int64_t)k * rt);   // cell (c + k z, bin0 + k r)
#pragma unroll
            for (int q = 0; q < Q; ++q) v[q][k - 1] = __ldg(base + k * step * q);
        }
    } else {
        valid = 0;
#pragma unroll
        for (int k = 1; k <= KZ; ++k) {
            const float *base = P + ((int64_t)(c + k * z) * n + bin0 + (int64_t)k * rt);
            const int last = TALL ? lim.r_lim[k] : min(lim.r_lim[k], rend);
            const int in = last < rt ? 0 : min(TALL ? rend : (last - rt) / kHsThreads + 1, Q);   // q < in
#pragma unroll
            for (int q = 0; q < Q; ++q) v[q][k - 1] = q < in ? __ldg(base + k * step * q) : 0.f;
            if ((k & (k - 1)) == 0) valid |= (Mask)(in >= 64 ? ~0ull : (1ull << in) - 1) << (Q * (31 - __clz(k)));
        }
    }
    Mask mask = 0;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        float acc = v[q][0];
#pragma unroll
        for (int k = 1; k <= KZ; ++k) {
            if (k > 1) acc += v[q][k - 1];
            if ((k & (k - 1)) == 0) {   // level h = k: the sum replaces its last term
                const int j = 31 - __clz(k);
                if (acc > thr.t[j]) mask |= Mask(1) << (Q * j + q);
                v[q][k - 1] = acc;
            }
        }
    }
    mask &= valid;
    const int lane = threadIdx.x & 31;
    for (unsigned act; (act = __ballot_sync(0xffffffffu, mask != 0)) != 0;) {
        if (staged + __popc(act) > (unsigned)kWarpStage) {
            warp_flush(stage, staged, lane, out, max_cand, count);
            staged = 0;
        }
        if (mask) {
            const int b = (BITS == 6 ? __ffsll((long long)mask) : __ffs((int)mask)) - 1, j = b / Q;
            mask &= mask - 1;
            float t[1 << BITS];   // the sums by bit, then a tree of selects on the bits of b
#pragma unroll
            for (int i = 0; i < (1 << BITS); ++i) t[i] = i < Q * LV ? v[i % Q][(1 << (i / Q < LV ? i / Q : 0)) - 1] : 0.f;
#pragma unroll
            for (int bit = 0; bit < BITS; ++bit) {
                const bool up = (b >> bit) & 1;
#pragma unroll
                for (int i = 0; i < ((1 << BITS) >> (bit + 1)); ++i) t[i] = up ? t[2 * i + 1] : t[2 * i];
            }
            fdas_harmonic_candidate rec;
            const int q = b - Q * j;
            rec.tpl = c + (!TALL ? z : z < 0 ? z + q : z - q);
            rec.power = t[0];
            rec.bin = bin0 + rt + (TALL ? 0 : q * kHsThreads);
            rec.nharm = 1 << j;
            rec.reserved = 0;
            stage[staged + __popc(act & ((1u << lane) - 1u))] = rec;
        }
        staged += __popc(act);
    }
}

// One harmonic (a plain threshold of the plane): no cell is read twice, tiles go row by row.
// Q = 48 for planes that fill the GPU with such tiles, 8 below.
template <int Q>
__global__ void __launch_bounds__(kHsThreads, 2) harmonic_kernel_rows(const float *__restrict__ P, int c, int n, int bin0,
                                                                      int tiles_per_row, HsThresholds thr, HsLimits lim,
                                                                      fdas_harmonic_candidate *__restrict__ out,
                                                                      int64_t max_cand,
                                                                      unsigned long long *__restrict__ count)
{
    __shared__ fdas_harmonic_candidate stage[kHsThreads / 32][kWarpStage];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned staged = 0;
    const int64_t tiles = (int64_t)(2 * c + 1) * tiles_per_row;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int y = (int)(tile / tiles_per_row), first = 1 + (int)(tile - (int64_t)y * tiles_per_row) * kHsThreads * Q;
        hs_tile<1, Q>(P, c, n, bin0, y - c, first, lim.r_lim[1], thr, lim, stage[warp], staged, out, max_cand, count);
    }
    if (staged) warp_flush(stage[warp], staged, lane, out, max_cand, count);
}

// MODE: kWindows, or not by windows but by runs of rows with the same number of harmonics (win.count = 0),
// kTallRuns with tall tiles (a kernel of its own: their code costs 32 harmonics in long rows 9 %).
enum { kWindows, kRuns, kTallRuns };
template <int H, int MODE>
__global__ void __launch_bounds__(kHsThreads, 2) harmonic_kernel_slope(const float *__restrict__ P, int c, int n, int bin0,
                                                                       HsThresholds thr, HsLimits lim, HsWindows win,
                                                                       fdas_harmonic_candidate *__restrict__ out,
                                                                       int64_t max_cand,
                                                                       unsigned long long *__restrict__ count)
{
    __shared__ fdas_harmonic_candidate stage[kHsThreads / 32][kWarpStage];
    // entry (z = 0, number of harmonics inside the row) and entry (window, |z| = c .. 1): its end in tiles,
    // first and last fundamental, |z| << 14 | fundamentals per thread << 6 | harmonics; entry of a run of
    // rows: its end in tiles, tiles per row (or group of rows), largest |z|, rows per tile << 14 (0: one) |
    // fundamentals per thread << 6 | harmonics
    extern __shared__ int4 ent[];
    constexpr bool RUNS = MODE != kWindows, TALL = MODE == kTallRuns;
    __shared__ int part[kHsThreads / 32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rmax = lim.r_lim[1], most = min(H, rmax);   // harmonics inside a row of the plane
    const int zeros = most, runs = min(most, c), entries = zeros + (RUNS ? runs : win.count * c);
    {   // tile counts: each thread sums a run of entries, then a block scan
        const int per = (entries + kHsThreads - 1) / kHsThreads, e0 = min(tid * per, entries), e1 = min(e0 + per, entries);
        int sum = 0;
        for (int i = e0; i < e1; ++i) {
            if (i < zeros) {   // z = 0: fundamentals rmax / (i + 2) < r <= rmax / (i + 1), the rest with the most
                const int kz = i + 1, first = kz == zeros ? 1 : lim.r_lim[kz + 1] + 1, tile = kHsThreads * hs_q(kz);
                sum += (lim.r_lim[kz] - first + tile) / tile;
                ent[i] = make_int4(sum, first, lim.r_lim[kz], (hs_q(kz) << 6) | kz);
                continue;
            }
            const int e = i - zeros;
            if constexpr (RUNS) {   // rows c / (e + 2) < |z| <= c / (e + 1); the last run: all that are left
                const int kz = e + 1, hi = c / kz, rows = hi - (kz == runs ? 0 : c / (kz + 1));
                const int tile = kHsThreads * hs_q(kz), per_row = (rmax + tile - 1) / tile;
                const int cols = (rmax + kHsThreads - 1) / kHsThreads, tall = 2 * ((rows + hs_q(kz) - 1) / hs_q(kz)) * cols;
                const int blocks = gridDim.x, waves = (2 * rows * per_row + blocks - 1) / blocks;
                if (TALL && kz <= kHsTall && 2 * ((tall + blocks - 1) / blocks) <= waves) {
                    sum += tall;
                    ent[i] = make_int4(sum, cols, hi, (hs_q(kz) << 14) | (1 << 6) | (kHsCases + kz));
                } else {
                    sum += 2 * rows * per_row;
                    ent[i] = make_int4(sum, per_row, hi, (hs_q(kz) << 6) | kz);
                }
                continue;
            }
            const int w = e / c, a = c - (e - w * c);
            const int64_t lo = (int64_t)a * win.slope[w], hi = (int64_t)a * win.slope[w + 1];
            const int first = (int)(lo < rmax ? lo : rmax) + 1, last = (int)(hi < rmax ? hi : rmax);
            // the harmonics of its first fundamental inside the plane (rows and columns)
            const int kz = max(1, min(min(H, c / a), rmax / first)), tile = kHsThreads * hs_q(kz);
            sum += 2 * ((last - first + tile) / tile);   // both signs of z
            ent[i] = make_int4(sum, first, last, (a << 14) | (hs_q(kz) << 6) | kz);
        }
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) part[warp] = incl;
        __syncthreads();
        int before = incl - sum;
        for (int i = 0; i < warp; ++i) before += part[i];
        for (int i = e0; i < e1; ++i) ent[i].x += before;
        __syncthreads();
    }
    const int tiles = ent[entries - 1].x;
    unsigned staged = 0;
    // The entry of this block's tile, and its first tile.  A few entries are passed one at a time (most
    // steps of a large plane; the vote at once costs 257 x 1.4e6, 32 harmonics 528 us against 501), many
    // 32 at a time: a table of 750 entries costs a small plane 10 us otherwise (513 x 8000: 27 us against 17).
    int e = 0, begin = 0;
    int4 en = ent[0];
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        for (int i = 0; i < 8 && tile >= en.x; ++i) begin = en.x, en = ent[++e];
        if (tile >= en.x) {   // the last entry's end is past every tile
            int passed;
            do e += passed = __popc(__ballot_sync(0xffffffffu, ent[min(e + lane, entries - 1)].x <= tile));
            while (passed == 32);
            begin = ent[e - 1].x, en = ent[e];
        }
        const int body = en.w & 63, a = en.w >> 14, local = tile - begin;
        int z = 0, last = rmax, at = local;   // tile of the row
        if (!RUNS || e < zeros) {
            const int half = (en.x - begin) >> 1;
            last = en.z;
            if (a) {   // both signs of z
                z = local < half ? a : -a;
                at = local < half ? local : local - half;
            }
        } else {
            const int half = (en.x - begin) >> 1, u = local < half ? local : local - half, group = u / en.y;
            const int az = en.z - (TALL ? group * max(a, 1) : group);
            z = local < half ? az : -az;
            at = u - group * en.y;
            if (TALL && a) last = az - (e + 1 < entries ? ent[e + 1].z : 0);   // rows of the run from here on
        }
        const int first = (!RUNS || e < zeros ? en.y : 1) + at * kHsThreads * ((en.w >> 6) & 255);
#define FDAS_HS_CASE(K)                                                                                                   \
    case K:                                                                                                                \
        if constexpr (K <= H)                                                                                              \
            hs_tile<K>(P, c, n, bin0, z, first, last, thr, lim, stage[warp], staged, out, max_cand, count);                \
        break;
#define FDAS_HS_TALL(K)                                                                                                   \
    case kHsCases + K:                                                                                                     \
        if constexpr (TALL && K <= H)                                                                                      \
            hs_tile<K, hs_q(K), true>(P, c, n, bin0, z, first, last, thr, lim, stage[warp], staged, out, max_cand, count); \
        break;
        switch (body) {
            FDAS_HS_CASE(1) FDAS_HS_CASE(2) FDAS_HS_CASE(3) FDAS_HS_CASE(4) FDAS_HS_CASE(5) FDAS_HS_CASE(6) FDAS_HS_CASE(7)
            FDAS_HS_CASE(8) FDAS_HS_CASE(9) FDAS_HS_CASE(10) FDAS_HS_CASE(11) FDAS_HS_CASE(12) FDAS_HS_CASE(13)
            FDAS_HS_CASE(14) FDAS_HS_CASE(15) FDAS_HS_CASE(16) FDAS_HS_CASE(17) FDAS_HS_CASE(18) FDAS_HS_CASE(19)
            FDAS_HS_CASE(20) FDAS_HS_CASE(21) FDAS_HS_CASE(22) FDAS_HS_CASE(23) FDAS_HS_CASE(24) FDAS_HS_CASE(25)
            FDAS_HS_CASE(26) FDAS_HS_CASE(27) FDAS_HS_CASE(28) FDAS_HS_CASE(29) FDAS_HS_CASE(30) FDAS_HS_CASE(31)
            FDAS_HS_CASE(32)
            FDAS_HS_TALL(1) FDAS_HS_TALL(2)
        }
#undef FDAS_HS_CASE
#undef FDAS_HS_TALL
    }
    if (staged) warp_flush(stage[warp], staged, lane, out, max_cand, count);
}

// Blocks of `fn` that are resident at once (at most `tiles`); asked for once per kernel and device.
cudaError_t resident_grid(const void *fn, int64_t tiles, size_t smem, std::atomic<int> (&known)[64], unsigned *grid)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    int resident = dev >= 0 && dev < 64 ? known[dev].load(std::memory_order_relaxed) : 0;
    if (!resident) {
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kHsThreads, smem)) != cudaSuccess) return e;
        resident = sms * (per_sm > 0 ? per_sm : 1);
        if (dev >= 0 && dev < 64) known[dev].store(resident, std::memory_order_relaxed);
    }
    *grid = (unsigned)(tiles < resident ? tiles : resident);
    return cudaSuccess;
}

cudaError_t launch_hs(int H, const float *P, int m, int64_t n, int64_t bin0, const HsThresholds &thr,
                      fdas_harmonic_candidate *out, int64_t max_cand, unsigned long long *count, cudaStream_t s)
{
    const int64_t rmax = n - 1 - bin0;
    const int c = (m - 1) / 2;
    cudaError_t e;
    unsigned grid = 0;
    // at most one tile per 256 fundamentals of a row and one more for each end of a window
    const int64_t most_tiles = (int64_t)m * (rmax / kHsThreads + 1) + 2 * (int64_t)kHsMaxEntries + 32;
    // 32-bit fundamentals and bins, with room for the last tile's overhang past rmax, and tiles
    const int64_t limit = ((int64_t)1 << 31) - ((int64_t)1 << 16);
    if (n <= limit && (H == 1 || most_tiles <= limit)) {
        HsLimits lim{};
        for (int k = 1; k <= 32; ++k) lim.r_lim[k] = (int)(rmax / k);
        if (H == 1) {
            static std::atomic<int> known[2][64];
            const auto large = harmonic_kernel_rows<hs_q(1)>, small = harmonic_kernel_rows<8>;
            const int64_t tile = (int64_t)kHsThreads * hs_q(1), per_row = (rmax + tile - 1) / tile;
            if ((e = resident_grid((const void *)large, (int64_t)m * per_row, 0, known[0], &grid)) != cudaSuccess) return e;
            // (and not for rows that fill less than half of them: 65537 x 4096 218 us, 289 with them)
            if ((int64_t)m * per_row > 2 * (int64_t)grid && 2 * rmax >= per_row * tile) {
                large<<<grid, kHsThreads, 0, s>>>(P, c, (int)n, (int)bin0, (int)per_row, thr, lim, out, max_cand, count);
            } else {
                const int64_t per_row8 = (rmax + kHsThreads * 8 - 1) / (kHsThreads * 8);
                if ((e = resident_grid((const void *)small, (int64_t)m * per_row8, 0, known[1], &grid)) != cudaSuccess) return e;
                small<<<grid, kHsThreads, 0, s>>>(P, c, (int)n, (int)bin0, (int)per_row8, thr, lim, out, max_cand, count);
            }
            return cudaGetLastError();
        }
        // windows of about kHsWindowBytes of the plane: rows |z| <= rmax / S reach slope S.  Where the
        // table has no room for eight (more than 513 rows; for four, 1025 rows, in planes well beyond
        // L2) the rows go in runs: 1025 rows of 90 MB with two / eight / 32 harmonics 21 / 31 / 58 us, in
        // four windows 32 / 39 / 48, 1400 MB 303 / 481 / 732 against 303 / 480 / 700; 2001 rows of 90 MB
        // 22 / 33 / 65, in two windows 35 / 45 / 63, 1400 MB 308 / 490 / 760 against 328 / 537 / 917
        HsWindows win{};
        const int most = c > 0 ? std::min(kHsMaxWin, kHsMaxEntries / c) : 0;
        const int64_t plane = (int64_t)m * n * 4;
        if (most >= 8 || (most >= 4 && plane > (256ll << 20))) {
            const int64_t bytes = std::max(kHsWindowBytes, plane / most);
            for (int64_t S = 0; S < rmax;) {
                const int64_t a = std::min<int64_t>(c, S > 0 ? rmax / S : c);
                S += std::max<int64_t>(1, bytes / (4 * a * (a + 1)));
                if (win.count == most - 1 || S > rmax) S = rmax;
                win.slope[++win.count] = (int)S;
            }
        }
        const size_t table = sizeof(int4) * (32 + (win.count ? (size_t)win.count * c : 32));
        using Kernel = void (*)(const float *, int, int, int, HsThresholds, HsLimits, HsWindows, fdas_harmonic_candidate *,
                                int64_t, unsigned long long *);
        auto kernel = [&](auto mode) -> Kernel {
            switch (H) {
            case 2: return harmonic_kernel_slope<2, mode()>;
            case 4: return harmonic_kernel_slope<4, mode()>;
            case 8: return harmonic_kernel_slope<8, mode()>;
            case 16: return harmonic_kernel_slope<16, mode()>;
            default: return harmonic_kernel_slope<32, mode()>;
            }
        };
        // tall tiles where a row fills less than half of its kz = 1 tiles (65537 x 4096 with 2 / 8 / 32
        // harmonics 278 / 399 / 824 us, without 329 / 468 / 895)
        const int64_t tile = kHsThreads * hs_q(1), filled = (rmax + tile - 1) / tile * tile;
        const int mode = win.count ? kWindows : 2 * rmax < filled ? kTallRuns : kRuns;
        const Kernel fn = mode == kWindows ? kernel(std::integral_constant<int, kWindows>())
                          : mode == kRuns  ? kernel(std::integral_constant<int, kRuns>())
                                           : kernel(std::integral_constant<int, kTallRuns>());
        // (the occupancy of the largest table, so that one number serves every call)
        static std::atomic<int> known[3][6][64];
        const int level = 31 - __builtin_clz((unsigned)H);
        if ((e = resident_grid((const void *)fn, most_tiles, kHsTableBytes, known[mode][level], &grid)) != cudaSuccess) return e;
        fn<<<grid, kHsThreads, table, s>>>(P, c, (int)n, (int)bin0, thr, lim, win, out, max_cand, count);
        return cudaGetLastError();
    }
    const void *fn = nullptr;
    int64_t tile = 0;
    switch (H) {
    case 1: fn = (const void *)harmonic_kernel<1>; tile = kHsThreads * hs_per_thread<1>(); break;
    case 2: fn = (const void *)harmonic_kernel<2>; tile = kHsThreads * hs_per_thread<2>(); break;
    case 4: fn = (const void *)harmonic_kernel<4>; tile = kHsThreads * hs_per_thread<4>(); break;
    case 8: fn = (const void *)harmonic_kernel<8>; tile = kHsThreads * hs_per_thread<8>(); break;
    case 16: fn = (const void *)harmonic_kernel<16>; tile = kHsThreads * hs_per_thread<16>(); break;
    default: fn = (const void *)harmonic_kernel<32>; tile = kHsThreads * hs_per_thread<32>(); break;
    }
    const int64_t tiles_per_row = (rmax + tile - 1) / tile;
    static std::atomic<int> known[6][64];
    if ((e = resident_grid(fn, (int64_t)m * tiles_per_row, 0, known[31 - __builtin_clz((unsigned)H)], &grid)) != cudaSuccess) return e;
    switch (H) {
    case 1: harmonic_kernel<1><<<grid, kHsThreads, 0, s>>>(P, m, n, bin0, tiles_per_row, thr, out, max_cand, count); break;
    case 2: harmonic_kernel<2><<<grid, kHsThreads, 0, s>>>(P, m, n, bin0, tiles_per_row, thr, out, max_cand, count); break;
    case 4: harmonic_kernel<4><<<grid, kHsThreads, 0, s>>>(P, m, n, bin0, tiles_per_row, thr, out, max_cand, count); break;
    case 8: harmonic_kernel<8><<<grid, kHsThreads, 0, s>>>(P, m, n, bin0, tiles_per_row, thr, out, max_cand, count); break;
    case 16: harmonic_kernel<16><<<grid, kHsThreads, 0, s>>>(P, m, n, bin0, tiles_per_row, thr, out, max_cand, count); break;
    default: harmonic_kernel<32><<<grid, kHsThreads, 0, s>>>(P, m, n, bin0, tiles_per_row, thr, out, max_cand, count); break;
    }
    return cudaGetLastError();
}

int hs_cuda(cudaError_t e, const char *what)
{
    char buf[256];
    snprintf(buf, sizeof buf, "%s: %s (%s)", what, cudaGetErrorString(e), cudaGetErrorName(e));
    return set_error(FDAS_ERR_CUDA, buf);
}

}  // namespace
}  // namespace fdas

extern "C" int fdas_harmonic_sum(const float *plane_dev, int n_templates, int64_t n, int64_t bin0, int max_harm,
                                 const float *thresholds, fdas_harmonic_candidate *cand_dev, int64_t max_cand,
                                 unsigned long long *count_dev, void *stream)
{
    using namespace fdas;
    if (!plane_dev || !count_dev || !thresholds || (max_cand > 0 && !cand_dev))
        return set_error(FDAS_ERR_INVALID_ARG, "null pointer");
    if (max_cand < 0) return set_error(FDAS_ERR_INVALID_ARG, "max_cand must be >= 0");
    if (n_templates < 1 || (n_templates & 1) == 0)
        return set_error(FDAS_ERR_INVALID_ARG, "n_templates must be odd (rows z = -c .. c)");
    if (n < 1 || bin0 < 0 || bin0 >= n) return set_error(FDAS_ERR_INVALID_ARG, "need n >= 1 and 0 <= bin0 < n");
    if (max_harm < 1 || max_harm > 32 || (max_harm & (max_harm - 1)))
        return set_error(FDAS_ERR_INVALID_ARG, "max_harm must be a power of two in [1, 32]");
    if (reinterpret_cast<uintptr_t>(plane_dev) % 4 || reinterpret_cast<uintptr_t>(count_dev) % 8 ||
        reinterpret_cast<uintptr_t>(cand_dev) % 8)
        return set_error(FDAS_ERR_INVALID_ARG, "misaligned plane, counter or candidate array");
    HsThresholds thr{};
    for (int j = 0; (1 << j) <= max_harm; ++j) thr.t[j] = thresholds[j];
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(count_dev, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return hs_cuda(e, "clear candidate counter");
    if (n - 1 - bin0 < 1) return FDAS_OK;   // no fundamental r >= 1 inside the plane
    e = launch_hs(max_harm, plane_dev, n_templates, n, bin0, thr, cand_dev, max_cand, count_dev, s);
    if (e != cudaSuccess) return hs_cuda(e, "harmonic-sum launch");
    return FDAS_OK;
}
