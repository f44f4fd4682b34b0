// Plan-time device kernels: input domain check, radix sort of FP64 values
// with their original indices, the staircase; and the execute-time gather /
// scatter between user order and sorted order.
//
// The subdivision of Algorithm 1 and the complexity theorem of Sec. 4.2 take
// the points and frequencies sorted ascending; the inputs are unsorted, so the
// plan sorts both once and keeps the permutations.
//
// Values are non-negative doubles (checked beside), whose IEEE bit patterns
// compare like unsigned integers.  They are sorted stably by a 32-bit key, the
// leading 31 bits of (pattern - smallest non-zero pattern) within the range
// that the input spans (zero has a key of its own), in four 8-bit passes
// instead of the eight a 64-bit pattern takes and over 8-byte (key, index)
// pairs instead of 12 bytes; the few values that share a key are then ordered
// by their full patterns where they lie, or, if they are many, by passes over the
// bits that the key left out.  Points and frequencies share every
// launch, and up to kSmallSort of each are sorted by one CTA in one launch.
// Measured, both arrays on an idle GPU (sum of the launches): n = m = 1e6
// 0.45 ms in 52 launches on two streams -> 0.17 in 15; 1e5 0.16 -> 0.06; 2000
// 48 launches -> one of 0.02.  Bound by the scatters' 8-byte stores (L2) at
// 1e6 and by launch latency below 1e5.
#include <cooperative_groups.h>
#include <cstdint>

#include "df64.cuh"
#include "nuht_internal.h"

namespace nuht {

// streaming multiprocessors of the current device, cached per device (k_det.cu)
int device_sm_count();

namespace {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 4;                       // elements per thread per tile
constexpr int kSortTile = kSortThreads * kSortItems; // 1024: ~4 CTAs per SM at n = 1e6 (4096 left the scatter passes latency-bound)
constexpr int kRadix = 256;
constexpr int kSortDirectTiles = 128;   // up to this many tiles each scatter CTA sums the tile counts itself
constexpr int kRunMax = 64;             // longest run of equal keys ordered element by element
static_assert(kSortThreads == kRadix, "the scatter kernel scans one digit total per thread");

// Bit pattern with -0.0 folded onto +0.0.
__device__ __forceinline__ uint64_t sort_bits(double v)
{
    return v == 0.0 ? 0ull : (uint64_t)__double_as_longlong(v);
}

// false for negatives, NaN and +-inf; -0.0 is accepted
__device__ __forceinline__ bool in_domain(double v) { return v >= 0.0 && v <= 1.7976931348623157e308; }

// The 32-bit key: 0 for zero, else 1 + (bits - lo) >> shift, lo the smallest
// non-zero pattern and shift such that the largest fits 31 bits.
struct SortQuant {
    uint64_t lo;
    int shift;
    __device__ __forceinline__ uint32_t key(uint64_t b) const { return b == 0 ? 0u : 1u + (uint32_t)((b - lo) >> shift); }
    // the bits below the key (32 at most, for a finite range)
    __device__ __forceinline__ uint32_t low(uint64_t b) const { return (uint32_t)((b - lo) & ((1ull << shift) - 1)); }
};

// stats[0] = the largest ~bits over non-zero values, stats[1] = the largest bits
__device__ __forceinline__ SortQuant sort_quant(const unsigned long long* stats)
{
    const uint64_t hi = stats[1], lo = hi ? ~stats[0] : 0ull;
    const int used = 64 - __clzll((long long)(hi - lo));
    return SortQuant{lo, used > 31 ? used - 31 : 0};
}

__device__ __forceinline__ void warp_range(uint64_t& mn, uint64_t& mx)
{
    for (int off = 16; off > 0; off >>= 1) {
        const uint64_t a = __shfl_xor_sync(0xffffffffu, mn, off), c = __shfl_xor_sync(0xffffffffu, mx, off);
        mn = a > mn ? a : mn;
        mx = c > mx ? c : mx;
    }
}

// Domain check and value range of both arrays (blockIdx.y).
__global__ void __launch_bounds__(kSortThreads) k_sort_range(SortPair S)
{
    const SortArray& A = S.a[blockIdx.y];
    uint64_t mn = 0, mx = 0;   // of ~bits (non-zero), of bits
    int bad = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < A.n; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = A.in[i];
        if (!in_domain(v)) bad = 1;
        const uint64_t b = sort_bits(v);
        if (b && ~b > mn) mn = ~b;
        if (b > mx) mx = b;
    }
    // one pair of global updates per CTA (one per warp cost 80 us at n = m = 1e6)
    __shared__ unsigned long long cmn, cmx;
    if (threadIdx.x == 0) cmn = cmx = 0;
    __syncthreads();
    warp_range(mn, mx);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&cmn, (unsigned long long)mn);
        atomicMax(&cmx, (unsigned long long)mx);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (cmn) atomicMax(A.stats, cmn);
        if (cmx) atomicMax(A.stats + 1, cmx);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(A.flag, 1);
}

// Segment of the element at input index x (offsets off[0..nseg]).
__device__ __forceinline__ uint32_t seg_of(const int64_t* off, int nseg, int64_t x)
{
    int lo = 0, hi = nseg;   // last segment with off[seg] <= x
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= x) lo = mid; else hi = mid;
    }
    return (uint32_t)lo;
}

// What a pass sorts by: the keys formed from the input (first pass), the
// keys of the pairs, or the pairs' segment numbers.
enum { SORT_FIRST, SORT_KEY, SORT_SEG };

template <int KIND>
__device__ __forceinline__ uint2 sort_load(const SortArray& A, const SortQuant& q, const uint2* src, int64_t i)
{
    if (KIND == SORT_FIRST) return make_uint2(q.key(sort_bits(A.in[i])), (uint32_t)i);
    return src[i];
}

template <int KIND>
__device__ __forceinline__ unsigned sort_digit(const SortArray& A, int nseg, uint2 e, int shift)
{
    return ((KIND == SORT_SEG ? seg_of(A.off, nseg, e.y) : e.x) >> shift) & 0xFF;
}

// the array and tile of a CTA: the tiles of a[0], then those of a[1]
__device__ __forceinline__ int sort_tile_of(const SortPair& S, int blk, int* tile)
{
    const int w = blk >= S.a[0].ntiles;
    *tile = w ? blk - S.a[0].ntiles : blk;
    return w;
}

// Adds a tile's digit counts to h.  SKEWED: many elements may share a digit (a
// warp's are then added once).
template <int KIND, bool SKEWED>
__device__ __forceinline__ void sort_count_tile(const SortArray& A, const SortQuant& q, int nseg, int from, int shift,
                                                int tile, uint32_t* h)
{
    const int64_t base = (int64_t)tile * kSortTile;
#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const int64_t i = base + it * kSortThreads + threadIdx.x;
        const unsigned d = i < A.n ? sort_digit<KIND>(A, nseg, sort_load<KIND>(A, q, A.e[from], i), shift) : 0x100u;
        if (SKEWED && __all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0))) {
            if ((threadIdx.x & 31) == 0 && d < 0x100u) atomicAdd(&h[d], 32u);
        } else if (d < 0x100u) {
            atomicAdd(&h[d], 1u);
        }
    }
}

// Digit counts of every tile: hist[tile * kRadix + d].
template <int KIND>
__global__ void __launch_bounds__(kSortThreads) k_sort_hist(SortPair S, int from, int shift)
{
    __shared__ uint32_t h[kRadix];
    int tile;
    const SortArray& A = S.a[sort_tile_of(S, blockIdx.x, &tile)];
    const SortQuant q = KIND == SORT_FIRST ? sort_quant(A.stats) : SortQuant{0, 0};
    h[threadIdx.x] = 0;
    __syncthreads();
    sort_count_tile<KIND, false>(A, q, S.nseg, from, shift, tile, h);
    __syncthreads();
    A.hist[(int64_t)tile * kRadix + threadIdx.x] = h[threadIdx.x];
}

// Per digit (thread), the exclusive prefix of the tile counts in place and the
// digit's total in tot[d]: CTA = 32 digits x 32 runs of tiles.
__global__ void __launch_bounds__(1024) k_sort_colscan(SortPair S)
{
    __shared__ uint32_t part[32][33];
    const SortArray& A = S.a[blockIdx.y];
    const int d = blockIdx.x * 32 + (threadIdx.x & 31), run = threadIdx.x >> 5;
    const int per = (A.ntiles + 31) >> 5, t0 = run * per, t1 = t0 + per < A.ntiles ? t0 + per : A.ntiles;
    uint32_t sum = 0;
    for (int t = t0; t < t1; ++t) sum += A.hist[(int64_t)t * kRadix + d];
    part[run][threadIdx.x & 31] = sum;
    __syncthreads();
    uint32_t acc = 0;
    for (int r = 0; r < run; ++r) acc += part[r][threadIdx.x & 31];
    if (run == 31) A.tot[d] = acc + sum;
    for (int t = t0; t < t1; ++t) {
        const uint32_t v = A.hist[(int64_t)t * kRadix + d];
        A.hist[(int64_t)t * kRadix + d] = acc;
        acc += v;
    }
}

struct ScatterShared {
    uint32_t wcnt[kSortThreads / 32][kRadix];   // per-warp digit counts, then the warps' starts
    uint32_t wsum[kSortThreads / 32];
};

// Start of digit threadIdx.x's bucket from its total v: exclusive scan over the
// digits (blockDim.x == kRadix; all threads).
__device__ __forceinline__ uint32_t digit_start(uint32_t v, ScatterShared& sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += t;
    }
    if (lane == 31) sh.wsum[warp] = x;
    __syncthreads();
    uint32_t pre = 0;
    for (int w = 0; w < warp; ++w) pre += sh.wsum[w];
    return pre + x - v;
}

// Stable scatter of a tile in one pass, its elements of digit threadIdx.x from
// mybase on (returned: where the next tile's go).  Warp w of a tile owns its 128
// consecutive elements, in rounds of 32, so (warp, round, lane) is the input
// order: each warp ranks its elements among equal digits with a per-warp digit
// count in shared memory (warp-synchronous, no CTA barrier per round), then one
// exclusive prefix over the warps per digit places every warp's run after the
// earlier warps' in the tile's part of each digit bucket.
template <int KIND>
__device__ __forceinline__ uint32_t sort_scatter_tile(const SortArray& A, const SortQuant& q, int nseg, int from,
                                                      int shift, int tile, uint32_t mybase, ScatterShared& sh)
{
    constexpr int kWarps = kSortThreads / 32;
    uint32_t (*wcnt)[kRadix] = sh.wcnt;
    uint2* dst = A.e[from ^ 1];
    const int64_t n = A.n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = lane; i < kRadix; i += 32) wcnt[warp][i] = 0;
    __syncwarp();
    const unsigned lt = (1u << lane) - 1u;
    const int64_t wbase = (int64_t)tile * kSortTile + (int64_t)warp * (32 * kSortItems);
    uint2 el[kSortItems];
    unsigned dig[kSortItems];
    uint32_t rk[kSortItems];
#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const int64_t i = wbase + it * 32 + lane;
        el[it] = i < n ? sort_load<KIND>(A, q, A.e[from], i) : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const bool valid = wbase + it * 32 + lane < n;
        const unsigned d = valid ? sort_digit<KIND>(A, nseg, el[it], shift) : 0x100u;
        dig[it] = d;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t prior = valid ? wcnt[warp][d] : 0u;
        __syncwarp();
        if (valid && (peers & lt) == 0) wcnt[warp][d] = prior + __popc(peers);
        __syncwarp();
        rk[it] = prior + __popc(peers & lt);
    }
    __syncthreads();
    uint32_t run = mybase;
    for (int w = 0; w < kWarps; ++w) {
        const uint32_t t = wcnt[w][threadIdx.x];
        wcnt[w][threadIdx.x] = run;
        run += t;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kSortItems; ++it)
        if (dig[it] < 0x100u) dst[wcnt[warp][dig[it]] + rk[it]] = el[it];
    return run;
}

// With DIRECT (few tiles) the CTA forms the counts of the tiles before it and
// the totals itself instead of a scan launch between.
template <int KIND, bool DIRECT>
__global__ void __launch_bounds__(kSortThreads) k_sort_scatter(SortPair S, int from, int shift)
{
    __shared__ ScatterShared sh;
    int tile;
    const SortArray& A = S.a[sort_tile_of(S, blockIdx.x, &tile)];
    const SortQuant q = KIND == SORT_FIRST ? sort_quant(A.stats) : SortQuant{0, 0};
    uint32_t v = 0, mine = 0;
    if (DIRECT) {
#pragma unroll 8
        for (int t = 0; t < A.ntiles; ++t) {
            const uint32_t c = A.hist[(int64_t)t * kRadix + threadIdx.x];
            mine += t < tile ? c : 0u;
            v += c;
        }
    } else {
        v = A.tot[threadIdx.x];
        mine = A.hist[(int64_t)tile * kRadix + threadIdx.x];
    }
    const uint32_t start = digit_start(v, sh) + mine;
    sort_scatter_tile<KIND>(A, q, S.nseg, from, shift, tile, start, sh);
}

__device__ __forceinline__ void sort_put(const SortArray& A, int64_t pos, uint64_t bits, uint32_t idx)
{
    const double v = __longlong_as_double((long long)bits);
    A.out[pos] = v;
    A.perm[pos] = (int32_t)idx;
    const df s = df_from(v);
    A.split[pos] = make_float2(s.h, s.l);
}

// Writes the sorted values, their indices and their double-float parts.  An
// element of a run of equal keys (and segments) goes to its rank by full
// pattern within the run; equal patterns keep their order.  Runs of more than
// kRunMax stay as they are: unsorted[0] is set when two neighbours of one are out
// of order (k_sort_long then sorts the array), unsorted[1] collects the bits in
// which the neighbours of any run differ.  A segment's elements lie where its input does, at
// off[seg].. of the sorted array.
__global__ void __launch_bounds__(kSortThreads) k_sort_finish(SortPair S, int from)
{
    const SortArray& A = S.a[blockIdx.y];
    const uint2* e = A.e[from];
    const SortQuant q = sort_quant(A.stats);
    auto bits_of = [&](int64_t i) { return sort_bits(A.in[e[i].y]); };
    uint32_t differ = 0;
    bool wrong = false;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < A.n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint2 el = e[i];
        const uint64_t b = sort_bits(A.in[el.y]);
        int64_t pos = i;
        if (q.shift > 0 && el.x != 0) {
            int64_t first = 0, end = A.n;
            if (S.nseg > 1) {
                const uint32_t seg = seg_of(A.off, S.nseg, i);
                first = A.off[seg];
                end = A.off[seg + 1];
            }
            auto same = [&](int64_t k) { return k >= first && k < end && e[k].x == el.x; };
            const bool before = same(i - 1);
            if (before || same(i + 1)) {
                int left = 0, right = 0;
                bool over = same(i - kRunMax) || same(i + kRunMax);
                while (!over && same(i - left - 1)) ++left;
                while (!over && same(i + right + 1)) ++right;
                over = over || left + right + 1 > kRunMax;
                if (before) {
                    const uint64_t o = bits_of(i - 1);
                    wrong = wrong || (over && o > b);
                    differ |= q.low(o) ^ q.low(b);
                }
                if (!over) {
                    int rank = 0;
                    for (int k = 1; k <= left; ++k) rank += bits_of(i - k) <= b;
                    for (int k = 1; k <= right; ++k) rank += bits_of(i + k) < b;
                    pos = i - left + rank;
                }
            }
        }
        sort_put(A, pos, b, el.y);
    }
    // one pair of global updates per CTA, and only where it adds something (a store
    // per element took 0.6 ms for 1e6 elements of one run)
    __shared__ uint32_t cta;
    if (threadIdx.x == 0) cta = 0;
    const bool any = __syncthreads_or(wrong || differ != 0);
    if (!any) return;
    differ = __reduce_or_sync(0xffffffffu, differ);
    if ((threadIdx.x & 31) == 0) atomicOr(&cta, differ);
    wrong = __syncthreads_or(wrong);
    if (threadIdx.x == 0) {
        volatile uint32_t* u = A.unsorted;
        if (wrong && u[0] == 0) u[0] = 1u;
        if ((cta & ~u[1]) != 0) atomicOr(A.unsorted + 1, cta);
    }
}

// The arrays with a run of more than kRunMax equal keys out of order (values
// packed more densely than 1 / kRunMax of a 2^-31 step of their range), sorted
// once more by all CTAs together: stable passes over the bits below the keys in
// which a run's values differ, the keys and the segments.  A CTA takes consecutive
// tiles and counts their digits together; grid barriers lie between the counts of
// a pass, their prefix over the CTAs and the scatter.  Returns at once otherwise.
// One CTA per run took 12 ms for 1e6 values of one run; 0.11 here where they differ
// in their last bits, 0.40 for 4e6 that differ in 22.
constexpr int kLongRuns = 32, kLongLen = 20;              // the CTAs' counts: runs of up to kLongLen of them
constexpr int kLongMaxCtas = kLongRuns * kLongLen;

__global__ void __launch_bounds__(kSortThreads, 4) k_sort_long(SortPair S)
{
    if (S.a[0].unsorted[0] == 0 && S.a[1].unsorted[0] == 0) return;
    __shared__ ScatterShared sh;
    __shared__ uint32_t part[kLongRuns][9];
    cooperative_groups::grid_group grid = cooperative_groups::this_grid();
    auto sync = [&]() {
        if (gridDim.x > 1) grid.sync();
        else __syncthreads();
    };
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    SortQuant q[2];
    int low_at[2][4], nlow[2], npass[2], per[2], most = 0;   // the low digits, passes over them and in all, tiles per CTA
    for (int w = 0; w < 2; ++w) {
        const SortArray& A = S.a[w];
        q[w] = sort_quant(A.stats);
        nlow[w] = 0;
        for (uint32_t m = A.unsorted[1]; m != 0; ++nlow[w]) {
            const int at = __ffs(m) - 1;
            low_at[w][nlow[w]] = at;
            m &= ~(0xFFu << at);
        }
        npass[w] = A.unsorted[0] ? nlow[w] + 4 + (S.nseg <= 1 ? 0 : (S.nseg - 1) >> 8 ? 2 : 1) : 0;
        per[w] = (A.ntiles + (int)gridDim.x - 1) / (int)gridDim.x;
        most = npass[w] > most ? npass[w] : most;
        for (int64_t i = t0; npass[w] && i < A.n; i += step)
            A.e[0][i] = make_uint2(q[w].low(sort_bits(A.in[i])), (uint32_t)i);
    }
    for (int pass = 0; pass < most; ++pass) {
        const int from = pass & 1;
        sync();
        bool keys = false;
        for (int w = 0; w < 2; ++w) {
            if (npass[w] == 0 || pass != nlow[w]) continue;
            const SortArray& A = S.a[w];
            keys = true;
            for (int64_t i = t0; i < A.n; i += step) A.e[from][i].x = q[w].key(sort_bits(A.in[A.e[from][i].y]));
        }
        if (keys) sync();
        for (int w = 0; w < 2; ++w) {
            const SortArray& A = S.a[w];
            const int first = blockIdx.x * per[w], end = first + per[w] < A.ntiles ? first + per[w] : A.ntiles;
            if (pass >= npass[w] || first >= end) continue;
            const int p = pass - nlow[w], at = p < 0 ? low_at[w][pass] : 8 * (p & 3);
            uint32_t* h = sh.wcnt[0];
            h[threadIdx.x] = 0;
            __syncthreads();
            for (int t = first; t < end; ++t) {
                if (p < 4) sort_count_tile<SORT_KEY, true>(A, q[w], S.nseg, from, at, t, h);
                else sort_count_tile<SORT_SEG, true>(A, q[w], S.nseg, from, at, t, h);
            }
            __syncthreads();
            A.hist[(int64_t)blockIdx.x * kRadix + threadIdx.x] = h[threadIdx.x];
        }
        sync();
        // prefix of 8 digits' counts over the CTAs
        for (int u = blockIdx.x; u < 2 * kRadix / 8; u += gridDim.x) {
            const int w = u >= kRadix / 8;
            if (pass >= npass[w]) continue;
            const SortArray& A = S.a[w];
            const int nb = (A.ntiles + per[w] - 1) / per[w];   // CTAs with tiles, at most kLongMaxCtas
            const int c = threadIdx.x & 7, d = 8 * (u & (kRadix / 8 - 1)) + c, run = threadIdx.x >> 3;
            uint32_t v[kLongLen], sum = 0;
#pragma unroll
            for (int k = 0; k < kLongLen; ++k) {   // all in flight
                const int b = run * kLongLen + k;
                v[k] = b < nb ? A.hist[(int64_t)b * kRadix + d] : 0u;
            }
#pragma unroll
            for (int k = 0; k < kLongLen; ++k) sum += v[k];
            part[run][c] = sum;
            __syncthreads();
            uint32_t acc = 0;
            for (int r = 0; r < run; ++r) acc += part[r][c];
            if (run == kLongRuns - 1) A.tot[d] = acc + sum;
#pragma unroll
            for (int k = 0; k < kLongLen; ++k) {
                const int b = run * kLongLen + k;
                if (b < nb) A.hist[(int64_t)b * kRadix + d] = acc;
                acc += v[k];
            }
            __syncthreads();   // part is rewritten by the next digits
        }
        sync();
        for (int w = 0; w < 2; ++w) {
            const SortArray& A = S.a[w];
            const int first = blockIdx.x * per[w], end = first + per[w] < A.ntiles ? first + per[w] : A.ntiles;
            if (pass >= npass[w] || first >= end) continue;
            const int p = pass - nlow[w], at = p < 0 ? low_at[w][pass] : 8 * (p & 3);
            uint32_t base = digit_start(A.tot[threadIdx.x], sh) + A.hist[(int64_t)blockIdx.x * kRadix + threadIdx.x];
            for (int t = first; t < end; ++t) {
                if (p < 4) base = sort_scatter_tile<SORT_KEY>(A, q[w], S.nseg, from, at, t, base, sh);
                else base = sort_scatter_tile<SORT_SEG>(A, q[w], S.nseg, from, at, t, base, sh);
                __syncthreads();   // sh is rewritten by the next tile
            }
        }
    }
    sync();
    for (int w = 0; w < 2; ++w) {
        const SortArray& A = S.a[w];
        for (int64_t i = t0; npass[w] && i < A.n; i += step) {
            const uint2 el = A.e[npass[w] & 1][i];
            sort_put(A, i, sort_bits(A.in[el.y]), el.y);
        }
    }
}

// Small arrays: one CTA each (blockIdx.x), everything in one launch.  Thread t
// of warp w holds the pairs w 32 ITEMS + 32 it + lane, so that (warp, it,
// lane) is the current order; each pass ranks them as k_sort_scatter does and
// writes them back to shared memory in their new order.  Elements of equal keys
// are ranked by their full patterns within the run, or, where a run of more than
// kRunMax is out of order (values far closer than their range: radii of points on
// a few circles), sorted once more by the bits below the key and the key: a plan
// of 8000 such radii 5.0 -> 0.15 ms.
constexpr int kSmallThreads = 1024;

template <int ITEMS>
__global__ void __launch_bounds__(kSmallThreads) k_sort_small(SortPair S)
{
    extern __shared__ uint2 pairs[];                     // [1024 ITEMS]
    uint32_t* wcnt = (uint32_t*)(pairs + kSmallThreads * ITEMS);   // [32][kRadix]
    __shared__ uint32_t wsum[32];
    __shared__ unsigned long long st[2];
    const SortArray& A = S.a[blockIdx.x];
    const int n = (int)A.n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int wbase = warp * 32 * ITEMS + lane;
    if (threadIdx.x < 2) st[threadIdx.x] = 0;
    __syncthreads();
    {
        uint64_t mn = 0, mx = 0;
        int bad = 0;
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const int i = wbase + 32 * it;
            const double v = i < n ? A.in[i] : 0.0;
            if (!in_domain(v)) bad = 1;
            const uint64_t b = sort_bits(v);
            if (b && ~b > mn) mn = ~b;
            if (b > mx) mx = b;
        }
        warp_range(mn, mx);
        if (lane == 0) {
            if (mn) atomicMax(&st[0], (unsigned long long)mn);
            if (mx) atomicMax(&st[1], (unsigned long long)mx);
        }
        if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(A.flag, 1);
    }
    const SortQuant q = sort_quant(st);
    uint2 el[ITEMS];
    int nlow = 0;        // passes over the bits below the key, before the key's
    bool ranked = false; // elements of equal keys go to their rank by full pattern
    for (;;) {
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const int i = wbase + 32 * it;
            el[it] = make_uint2(i < n ? q.key(sort_bits(A.in[i])) : 0u, (uint32_t)i);
        }
        for (int pass = 0; pass < nlow + 4; ++pass) {
            for (int i = threadIdx.x; i < 32 * kRadix; i += kSmallThreads) wcnt[i] = 0;
            __syncthreads();
            uint32_t rk[ITEMS];
            unsigned dig[ITEMS];
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {
                const bool valid = wbase + 32 * it < n;
                unsigned d = 0x100u;
                if (valid) d = pass < nlow ? (q.low(sort_bits(A.in[el[it].y])) >> (8 * pass)) & 0xFFu : (el[it].x >> (8 * (pass - nlow))) & 0xFFu;
                dig[it] = d;
                const unsigned peers = __match_any_sync(0xffffffffu, d);
                const uint32_t prior = valid ? wcnt[warp * kRadix + d] : 0u;
                __syncwarp();
                if (valid && (peers & lt) == 0) wcnt[warp * kRadix + d] = prior + __popc(peers);
                __syncwarp();
                rk[it] = prior + __popc(peers & lt);
            }
            __syncthreads();
            uint32_t tot = 0, x = 0;
            if (threadIdx.x < kRadix) {
                for (int w = 0; w < 32; ++w) {
                    const uint32_t t = wcnt[w * kRadix + threadIdx.x];
                    wcnt[w * kRadix + threadIdx.x] = tot;
                    tot += t;
                }
                x = tot;
                for (int off = 1; off < 32; off <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xffffffffu, x, off);
                    if (lane >= off) x += t;
                }
                if (lane == 31) wsum[warp] = x;
            }
            __syncthreads();
            if (threadIdx.x < kRadix) {
                uint32_t pre = x - tot;
                for (int w = 0; w < warp; ++w) pre += wsum[w];
                for (int w = 0; w < 32; ++w) wcnt[w * kRadix + threadIdx.x] += pre;
            }
            __syncthreads();
#pragma unroll
            for (int it = 0; it < ITEMS; ++it)
                if (dig[it] < 0x100u) pairs[wcnt[warp * kRadix + dig[it]] + rk[it]] = el[it];
            __syncthreads();
#pragma unroll
            for (int it = 0; it < ITEMS; ++it)
                if (wbase + 32 * it < n) el[it] = pairs[wbase + 32 * it];
            // (the next pass writes pairs only after a barrier)
        }
        if (nlow > 0 || q.shift == 0) break;   // in order by full pattern
        // runs of equal keys: out of order anywhere, longer than kRunMax anywhere
        bool fix = false, longer = false;
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const int i = wbase + 32 * it;
            if (i >= n || el[it].x == 0) continue;
            if (i > 0 && pairs[i - 1].x == el[it].x &&
                sort_bits(A.in[pairs[i - 1].y]) > sort_bits(A.in[el[it].y])) fix = true;
            if (i + kRunMax < n && pairs[i + kRunMax].x == el[it].x) longer = true;
        }
        ranked = __syncthreads_or(fix);
        if (!__syncthreads_or(longer) || !ranked) break;
        ranked = false;
        nlow = (q.shift + 7) >> 3;
    }
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int i = wbase + 32 * it;
        if (i >= n) continue;
        const uint64_t b = sort_bits(A.in[el[it].y]);
        int pos = i;
        if (ranked && el[it].x != 0) {
            int left = 0, rank = 0;
            for (int k = i - 1; k >= 0 && pairs[k].x == el[it].x; --k, ++left)
                rank += sort_bits(A.in[pairs[k].y]) <= b;
            for (int k = i + 1; k < n && pairs[k].x == el[it].x; ++k) rank += sort_bits(A.in[pairs[k].y]) < b;
            pos = i - left + rank;
        }
        sort_put(A, pos, b, el[it].y);
    }
}

// nrep copies of a plan's sorted arrays, one after the other (derivative plans).
__global__ void k_replicate(SortedView src, SortedView dst, int64_t n, int64_t m, int nrep)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nrep * (n > m ? n : m);
         i += (int64_t)gridDim.x * blockDim.x) {
        if (i < nrep * n) {
            const int64_t k = i % n;
            dst.r[i] = src.r[k];
            dst.r2[i] = src.r2[k];
            dst.pr[i] = src.pr[k];
        }
        if (i < nrep * m) {
            const int64_t k = i % m;
            dst.w[i] = src.w[k];
            dst.w2[i] = src.w2[k];
            dst.pw[i] = src.pw[k];
        }
    }
}

// Bits of the largest input magnitude from k_prepare's CTA maxima; CTA 0
// leaves it for the scatter.  All threads of the CTA.
__device__ __forceinline__ unsigned long long input_max(const unsigned long long* __restrict__ part, int parts,
                                                        unsigned long long* __restrict__ mx)
{
    __shared__ unsigned long long wm[kSortThreads / 32];
    unsigned long long m = 0;
    for (int i = threadIdx.x; i < parts; i += blockDim.x) m = part[i] > m ? part[i] : m;
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, off);
        m = o > m ? o : m;
    }
    if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
    __syncthreads();
    for (int w = 0; w < kSortThreads / 32; ++w) m = wm[w] > m ? wm[w] : m;
    if (blockIdx.x == 0 && threadIdx.x == 0) *mx = m;
    return m;
}

// Components comp .. comp + G - 1 of the input (user order, rows of stride),
// scaled by 2^-E (exact), into sorted order: member v at out + v n (and as
// double-float at out2 + v n).  One thread per point for all members, so that
// a row is read once.  ws (derivative plans): the input weighted by the sorted
// values, n = nrep nb elements, both problems' copies.
__global__ void __launch_bounds__(kSortThreads) k_gather(const double* __restrict__ c,
                                                         const int32_t* __restrict__ perm, int64_t n, int64_t nb,
                                                         const double* __restrict__ ws, int stride, int comp, int G,
                                                         const unsigned long long* __restrict__ part, int parts,
                                                         unsigned long long* __restrict__ mx,
                                                         double* __restrict__ out, float2* __restrict__ out2)
{
    const int e = -input_exponent(input_max(part, parts, mx));
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i0 = i < nb ? i : i - nb;
        const double* row = c + (int64_t)perm[i0] * stride + comp;
        const double wt = ws ? ws[i0] : 1.0;
        for (int v = 0; v < G; ++v) {
            const double x = scale_pow2(ws ? row[v] * wt : row[v], e);
            out[v * n + i] = x;
            if (out2) {
                const df s = df_from(x);
                out2[v * n + i] = make_float2(s.h, s.l);
            }
        }
    }
}

// Members gs + v m back to user order, components comp .. comp + G - 1.
__global__ void __launch_bounds__(kSortThreads) k_scatter(const double* __restrict__ gs,
                                                          const int32_t* __restrict__ perm, int64_t m, int stride,
                                                          int comp, int G,
                                                          const unsigned long long* __restrict__ mx,
                                                          double* __restrict__ g)
{
    const int e = input_exponent(*mx);   // back to the input's scale (exact)
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        double* row = g + (int64_t)perm[i] * stride + comp;
        for (int v = 0; v < G; ++v) row[v] = scale_pow2(gs[v * m + i], e);
    }
}

// out[u] (+)= sum_v y_u (gs[k] + gs[mb + k]) / 2 back at the input's scale, u = perm[k]:
// the two problems' sums (orders nu - 1 and nu + 1, the second negated) give
// J_nu' = (J_{nu-1} - J_{nu+1}) / 2 (DLMF 10.6.1); vectors after the first add on.
// With one problem (nrep = 1) its sums are the derivative.
__global__ void __launch_bounds__(kSortThreads) k_scatter_deriv(const double* __restrict__ gs,
                                                                const int32_t* __restrict__ perm, int64_t mb,
                                                                int nrep, int stride, int comp, int G,
                                                                const unsigned long long* __restrict__ mx,
                                                                const double* __restrict__ y,
                                                                double* __restrict__ out)
{
    const int e = input_exponent(*mx) - (nrep == 2 ? 1 : 0);
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < mb;
         k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = perm[k];
        double sum = comp == 0 ? 0.0 : out[u];
        for (int v = 0; v < G; ++v) {
            const double* gv = gs + v * nrep * mb;
            const double x = scale_pow2(nrep == 2 ? gv[k] + gv[mb + k] : gv[k], e) * y[u * stride + comp + v];
            sum = comp + v == 0 ? x : sum + x;
        }
        out[u] = sum;
    }
}

// First j in [lo, hi) with wk * r_j > z (hi if none); r ascending.
__device__ __forceinline__ int64_t first_above(const double* __restrict__ r, int64_t lo, int64_t hi, double wk,
                                               double z)
{
    while (lo < hi) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        if (wk * r[mid] <= z) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The same by all lanes of a warp: 32 probes a step instead of one.
__device__ __forceinline__ int64_t first_above_warp(const double* __restrict__ r, int64_t lo, int64_t hi, double wk,
                                                    double z)
{
    const int lane = threadIdx.x & 31;
    while (hi - lo > 32) {
        const int64_t step = (hi - lo + 32) / 33, at = lo + (lane + 1) * step;   // lo < at, ascending
        const int in = __popc(__ballot_sync(0xffffffffu, at < hi && wk * r[at < hi ? at : lo] <= z));
        // the first `in` probes are inside: the answer lies after the last of them, up to the next
        const int64_t nlo = in ? lo + in * step + 1 : lo, nhi = lo + (in + 1) * step;
        lo = nlo;
        hi = nhi < hi ? nhi : hi;
    }
    const int64_t at = lo + lane;
    return lo + __popc(__ballot_sync(0xffffffffu, at < hi && wk * r[at < hi ? at : 0] <= z));
}

constexpr int kStairThreads = 256;   // rows per CTA: one each (four, one after the other, took 19 us at m = 1e5)

// s[k] = max{j : omega_k * r_j <= z} (or -1): the boundary of the local region
// in row k of the sorted matrix, a column local to the row's problem (the one
// with w_off <= k < w_off + m).  f(k) = s[k] + 1 is non-increasing in k within
// a problem (the FP64 product is monotone in both factors), so a CTA whose
// rows lie in one problem searches its first and last rows over all of r, a
// warp each, and its other rows only between those two bounds: four steps of
// latency per CTA instead of twenty per row (m = 1e6: 36 -> 14 us; two problems
// of 1e6 each, every row in full: 156 -> 44).  A CTA that spans problems
// searches every row in full.
__global__ void __launch_bounds__(kStairThreads) k_staircase(const double* __restrict__ r,
                                                             const double* __restrict__ w, int64_t m,
                                                             const ProbParams* __restrict__ probs, int nprob,
                                                             int32_t* __restrict__ s)
{
    __shared__ int64_t fb[2];
    __shared__ int pb[2];
    const int64_t span = kStairThreads;
    auto problem_of = [&](int64_t k) {
        int lo = 0, hi = nprob;   // last problem with w_off <= k
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (probs[mid].w_off <= k) lo = mid; else hi = mid;
        }
        return lo;
    };
    for (int64_t base = (int64_t)blockIdx.x * span; base < m; base += (int64_t)gridDim.x * span) {
        const int64_t last = (base + span < m ? base + span : m) - 1;
        const int warp = threadIdx.x >> 5;
        if (warp < 2) {
            const int64_t k = warp == 0 ? base : last;
            const int p = problem_of(k);
            const ProbParams& P = probs[p];
            const int64_t f = first_above_warp(r + P.r_off, 0, P.n, w[k], P.z);
            if ((threadIdx.x & 31) == 0) {
                pb[warp] = p;
                fb[warp] = f;
            }
        }
        __syncthreads();
        if (pb[0] == pb[1]) {
            const double* rp = r + probs[pb[0]].r_off;
            const double z = probs[pb[0]].z;
            const int64_t hi = fb[0], lo = fb[1];   // f(last) <= f(k) <= f(base)
            const int64_t k = base + threadIdx.x;
            if (k <= last) s[k] = (int32_t)(first_above(rp, lo, hi, w[k], z) - 1);
        } else {
            const int64_t k = base + threadIdx.x;
            if (k <= last) {
                const ProbParams& P = probs[problem_of(k)];
                s[k] = (int32_t)(first_above(r + P.r_off, 0, P.n, w[k], P.z) - 1);
            }
        }
        __syncthreads();   // fb and pb are rewritten by the next range
    }
}

inline int grid_for(int64_t n, int threads)
{
    int64_t b = (n + threads - 1) / threads;
    const int64_t cap = (int64_t)device_sm_count() * 32;
    if (b > cap) b = cap;
    return b < 1 ? 1 : (int)b;
}

inline size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

size_t sort_scratch_bytes(int64_t n)
{
    const int64_t ntiles = (n + kSortTile - 1) / kSortTile;
    return 2 * align256(sizeof(uint2) * (size_t)n) +
           align256(sizeof(uint32_t) * (size_t)kRadix * (size_t)(ntiles > 0 ? ntiles : 1)) +
           align256(sizeof(uint32_t) * (size_t)kRadix);
}

namespace {

template <int ITEMS>
cudaError_t sort_small(const SortPair& S, cudaStream_t s)
{
    const size_t smem = sizeof(uint2) * kSmallThreads * ITEMS + sizeof(uint32_t) * 32 * kRadix;
    cudaError_t e = allow_smem(k_sort_small<ITEMS>, smem);
    if (e != cudaSuccess) return e;
    k_sort_small<ITEMS><<<2, kSmallThreads, smem, s>>>(S);
    count_launches(1);
    return cudaGetLastError();
}

template <int KIND>
void sort_pass(const SortPair& S, int from, int shift, bool direct, cudaStream_t s)
{
    const int nt = S.a[0].ntiles + S.a[1].ntiles;
    k_sort_hist<KIND><<<nt, kSortThreads, 0, s>>>(S, from, shift);
    if (direct) {
        k_sort_scatter<KIND, true><<<nt, kSortThreads, 0, s>>>(S, from, shift);
    } else {
        k_sort_colscan<<<dim3(kRadix / 32, 2), 1024, 0, s>>>(S);
        k_sort_scatter<KIND, false><<<nt, kSortThreads, 0, s>>>(S, from, shift);
    }
    count_launches(direct ? 2 : 3);
}

// k_sort_long by the CTAs that are resident together (up to four per SM, and
// kLongMaxCtas), or by one where a cooperative launch is refused.
cudaError_t sort_long(const SortPair& S, cudaStream_t s)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sort_long, kSortThreads, 0) == cudaSuccess && per_sm > 0) {
        void* args[] = {(void*)&S};
        const int all = (per_sm < 4 ? per_sm : 4) * device_sm_count();
        if (cudaLaunchCooperativeKernel((const void*)k_sort_long, dim3(all < kLongMaxCtas ? all : kLongMaxCtas),
                                        dim3(kSortThreads), args, 0, s) == cudaSuccess) {
            count_launches(1);
            return cudaSuccess;
        }
    }
    (void)cudaGetLastError();
    k_sort_long<<<1, kSortThreads, 0, s>>>(S);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace

// Checks and sorts both arrays (out, perm, split); scratch as
// sort_scratch_bytes each, flag, stats[2] and unsorted[2] of each array zeroed.
// With nseg > 1 segments (device offsets off[0..nseg], nseg <= 65536) each
// segment is sorted on its own: the key passes are followed by stable passes
// on the segment number, so the output keeps the segments in order.
cudaError_t launch_sort_pair(SortPair S, char* const scratch[2], cudaStream_t s)
{
    if (S.a[0].n <= 0 && S.a[1].n <= 0) return cudaSuccess;
    const int64_t most = S.a[0].n > S.a[1].n ? S.a[0].n : S.a[1].n;
    if (S.nseg <= 1 && most <= kSmallSort) {
        if (most <= 1 * kSmallThreads) return sort_small<1>(S, s);
        if (most <= 4 * kSmallThreads) return sort_small<4>(S, s);
        return sort_small<kSmallSort / kSmallThreads>(S, s);
    }
    bool direct = true;
    for (int k = 0; k < 2; ++k) {
        SortArray& A = S.a[k];
        char* p = scratch[k];
        A.ntiles = (int)((A.n + kSortTile - 1) / kSortTile);
        A.e[0] = (uint2*)p; p += align256(sizeof(uint2) * (size_t)A.n);
        A.e[1] = (uint2*)p; p += align256(sizeof(uint2) * (size_t)A.n);
        A.hist = (uint32_t*)p; p += align256(sizeof(uint32_t) * (size_t)kRadix * (size_t)(A.ntiles > 0 ? A.ntiles : 1));
        A.tot = (uint32_t*)p;
        direct = direct && A.ntiles <= kSortDirectTiles;
    }
    const dim3 all(grid_for(most, kSortThreads), 2);
    const int64_t few = (most + 8 * kSortThreads - 1) / (8 * kSortThreads), cap = 2 * (int64_t)device_sm_count();
    k_sort_range<<<dim3((unsigned)(few < cap ? few : cap), 2), kSortThreads, 0, s>>>(S);
    sort_pass<SORT_FIRST>(S, 1, 0, direct, s);
    int cur = 0;
    for (int shift = 8; shift < 32; shift += 8, cur ^= 1) sort_pass<SORT_KEY>(S, cur, shift, direct, s);
    for (int shift = 0; S.nseg > 1 && (shift == 0 || (S.nseg - 1) >> shift); shift += 8, cur ^= 1)
        sort_pass<SORT_SEG>(S, cur, shift, direct, s);
    k_sort_finish<<<all, kSortThreads, 0, s>>>(S, cur);
    count_launches(2);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? sort_long(S, s) : e;
}

cudaError_t launch_replicate(const SortedView& src, const SortedView& dst, int64_t n, int64_t m, int nrep,
                             cudaStream_t s)
{
    const int64_t most = nrep * (n > m ? n : m);
    if (most <= 0) return cudaSuccess;
    k_replicate<<<grid_for(most, 256), 256, 0, s>>>(src, dst, n, m, nrep);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_staircase(const double* r, const double* w, int64_t m, const ProbParams* probs, int nprob,
                             int32_t* s_out, cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    k_staircase<<<grid_for(m, kStairThreads), kStairThreads, 0, s>>>(r, w, m, probs, nprob, s_out);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_gather(const double* c, const int32_t* perm, int64_t n, int64_t nb, const double* ws, int stride,
                          int comp, int G, const unsigned long long* part, int parts, unsigned long long* mx,
                          double* out, float2* out2, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    k_gather<<<grid_for(n, kSortThreads), kSortThreads, 0, s>>>(c, perm, n, nb, ws, stride, comp, G, part, parts, mx,
                                                                out, out2);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_scatter_deriv(const double* gs, const int32_t* perm, int64_t mb, int nrep, int stride, int comp, int G,
                                 const unsigned long long* mx, const double* y, double* out, cudaStream_t s)
{
    if (mb <= 0) return cudaSuccess;
    k_scatter_deriv<<<grid_for(mb, kSortThreads), kSortThreads, 0, s>>>(gs, perm, mb, nrep, stride, comp, G, mx, y,
                                                                        out);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_scatter(const double* gs, const int32_t* perm, int64_t m, int stride, int comp, int G,
                           const unsigned long long* mx, double* g, cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    k_scatter<<<grid_for(m, kSortThreads), kSortThreads, 0, s>>>(gs, perm, m, stride, comp, G, mx, g);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace nuht
