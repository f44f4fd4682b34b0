// Algorithm 1 (Subdivide) with SplitIndices (Sec. 4.1) on the device.
//
// The host version (subdivide.cpp) walks a first-in first-out work list.
// Here one CTA processes that list level by level: every mixed block of a
// level is split at once by a group of 16 or 4 lanes (16 candidate rows read
// from the staircase, then a child each), and block-wide prefix sums give each
// child its place in the local / asymptotic / direct lists or in the next
// level.  Bound by the latency of a level (10 at n = m = 1e5, 13 at 1e6): with
// one thread per block its 16 candidates, one after the other, took 16,000
// cycles a level.  n = m = 1e5 84 -> 36 us, 1e6 146 -> 79.
// Children are placed in the order the sequential walk would append them
// (parents in list order, children upper-left, lower-right, upper-right,
// lower-left), so for one problem the lists equal the host's, entry for
// entry.  A batch's roots start together; the host orders the lists by
// problem afterwards (a stable reordering).
//
// The staircase stair[w_off + k] = max{j : omega_k r_j <= z} (problem-local
// column, or -1) is non-increasing in k, so a block is all local iff
// stair[k1] >= j1 and all asymptotic iff stair[k0] < j0.
#include <cooperative_groups.h>
#include <cstdint>

#include "nuht_internal.h"

namespace nuht {

namespace {

constexpr int kSubThreads = 1024;
constexpr int kSubWarps = kSubThreads / 32;

// An asymptotic block too large for one FFT (X S > kAsyMaxXS) is queued like
// a mixed one, flagged in its problem index, and cut into quadrants; the host
// walk does the same in the same order.
constexpr int32_t kQuadFlag = 0x40000000;

__device__ __forceinline__ bool asy_too_big(const double* __restrict__ r, const double* __restrict__ w,
                                            const SubBlk& b)
{
    return 0.5 * (r[b.j1] - r[b.j0]) * 0.5 * (w[b.k1] - w[b.k0]) > kAsyMaxXS;
}

// 0 empty, 1 local, 2 asymptotic, 3 direct, 4 mixed (split further), 5
// asymptotic but too large (cut into quadrants)
__device__ __forceinline__ int classify(const int32_t* __restrict__ st, const SubBlk& b, int64_t min_size)
{
    if (b.k1 < b.k0 || b.j1 < b.j0) return 0;
    if (st[b.k1] >= b.j1) return 1;
    if (st[b.k0] < b.j0) return 2;
    if ((int64_t)(b.k1 - b.k0 + 1) * (int64_t)(b.j1 - b.j0 + 1) <= min_size) return 3;
    return 4;
}

// classify with the staircase values at the block's first and last rows given
__device__ __forceinline__ int classify_v(const SubBlk& b, int s0, int s1, int64_t min_size)
{
    if (b.k1 < b.k0 || b.j1 < b.j0) return 0;
    if (s1 >= b.j1) return 1;
    if (s0 < b.j0) return 2;
    if ((int64_t)(b.k1 - b.k0 + 1) * (int64_t)(b.j1 - b.j0 + 1) <= min_size) return 3;
    return 4;
}

// Exclusive block-wide prefix sum of a 64-bit value (four 16-bit counters
// packed; no carries since a chunk adds at most kSubThreads per field).
__device__ __forceinline__ uint64_t block_scan(uint64_t v, uint64_t* wsum, uint64_t* total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t x = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint64_t s = wsum[lane];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, s, off);
            if (lane >= off) s += y;
        }
        wsum[lane] = s;
    }
    __syncthreads();
    const uint64_t before = (wid > 0 ? wsum[wid - 1] : 0) + x - v;
    *total = wsum[kSubWarps - 1];
    __syncthreads();
    return before;
}

struct SubState {
    int64_t nout[3];   // local, asymptotic, direct blocks written so far
    int64_t nnext;     // blocks of the next level written so far
    int ovf;
    int shared;        // the next level lies in shared memory
};
constexpr int kSubShared = 512;   // levels of up to this many blocks stay in shared memory (at most kSubSolo:
                                  // a level left to the other CTAs lies in a global queue)

__device__ __forceinline__ uint64_t class_count(int cls)
{
    return cls > 0 ? (uint64_t)1 << (16 * ((cls < 4 ? cls : 4) - 1)) : 0ull;
}

// This thread's child (class cls, 0 = none) at its place: pos of its class
// list (out[c * ocap ...]) or of the next level's queue.
__device__ __forceinline__ void place(SubBlk ch, int cls, uint64_t off, const int64_t* base, SubBlk* __restrict__ out,
                                      int64_t ocap, SubBlk* next)
{
    if (cls == 0) return;
    const int f = (cls < 4 ? cls : 4) - 1;
    const int64_t pos = base[f] + (int64_t)((off >> (16 * f)) & 0xffff);
    if (cls >= 4) {
        if (cls == 5) ch.prob |= kQuadFlag;
        next[pos] = ch;
    } else {
        out[f * ocap + pos] = ch;
    }
}

// Places every thread's child in thread order: class lists and the next
// level's queue (next, or, when this is the level's only chunk and its
// children fit, nexts in shared memory).
__device__ __forceinline__ void emit(const SubBlk& ch, int cls, SubState& S, uint64_t* wsum,
                                     SubBlk* __restrict__ out, int64_t ocap, SubBlk* next, int64_t qcap,
                                     SubBlk* nexts, bool only)
{
    uint64_t total;
    const uint64_t off = block_scan(class_count(cls), wsum, &total);
    const int64_t base[4] = {S.nout[0], S.nout[1], S.nout[2], S.nnext};
    bool fits = S.ovf == 0;
    for (int c = 0; c < 3; ++c) fits = fits && base[c] + (int64_t)((total >> (16 * c)) & 0xffff) <= ocap;
    fits = fits && base[3] + (int64_t)(total >> 48) <= qcap;
    const bool sh = only && (int64_t)(total >> 48) <= kSubShared;
    if (fits) place(ch, cls, off, base, out, ocap, sh ? nexts : next);
    __syncthreads();
    if (threadIdx.x == 0) {
        S.shared = sh;
        if (fits) {
            for (int c = 0; c < 3; ++c) S.nout[c] += (int64_t)((total >> (16 * c)) & 0xffff);
            S.nnext += (int64_t)(total >> 48);
        } else {
            S.ovf = 1;   // the counts stay at what was written (within the capacities)
        }
    }
    __syncthreads();
}

// W lanes (16 or 4) share mixed block qa[i]: SplitIndices over up to n_cand
// candidate rows, one lane each at a time (the candidate row minimising the
// mixed area, its column the last local one; ties keep the first), or the
// quadrants of a flagged asymptotic block; then lane c < 4 of the group takes
// child c and its class (0 none / empty, 1..3 a list, 4 the next level, 5
// quadrants next).  Nothing for i >= na.
template <int W>
__device__ __forceinline__ void make_child(int64_t i, int64_t na, const SubBlk* qa, const int32_t* __restrict__ stair,
                                           const double* __restrict__ r_s, const double* __restrict__ w_s,
                                           const ProbParams* __restrict__ probs, int64_t min_size, int n_cand,
                                           bool may_exceed, SubBlk* ch, int* cls)
{
    const int sub = threadIdx.x & (W - 1);
    const bool live = i < na;
    SubBlk b = live ? qa[i] : SubBlk{0, -1, 0, -1, 0};
    const bool quad = (b.prob & kQuadFlag) != 0;
    b.prob &= ~kQuadFlag;
    const ProbParams& P = probs[b.prob];
    const int32_t* st = stair + P.w_off;
    const int rows = b.k1 - b.k0 + 1;
    const int nc = !live || quad ? 0 : (rows <= n_cand ? rows : n_cand);
    // the product fits 32 bits for up to 2^32 / n_cand rows
    const bool narrow = (int64_t)n_cand * rows <= 0xffffffffLL;
    int64_t best = INT64_MAX;
    int bc = 0x7fffffff, bk = b.k0, bj = b.j0 - 1;
    for (int c0 = sub; c0 < nc; c0 += 4 * W) {
        int kv[4], jv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = c0 + u * W;
            kv[u] = b.k0;
            if (c < nc) {
                if (rows <= n_cand) kv[u] += c;
                else if (narrow) kv[u] += (int)((unsigned)c * (unsigned)(rows - 1) / (unsigned)(n_cand - 1));
                else kv[u] += (int)((int64_t)c * (rows - 1) / (n_cand - 1));
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) jv[u] = c0 + u * W < nc ? st[kv[u]] : 0;   // all in flight
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = c0 + u * W, k = kv[u];
            int j = jv[u];
            if (j > b.j1) j = b.j1;
            if (j < b.j0) j = b.j0 - 1;
            const int64_t area = (int64_t)(k - b.k0 + 1) * (b.j1 - j) + (int64_t)(b.k1 - k) * (j - b.j0 + 1);
            if (c < nc && area < best) {
                best = area;
                bc = c;
                bk = k;
                bj = j;
            }
        }
    }
#pragma unroll
    for (int off = W / 2; off > 0; off >>= 1) {
        const int64_t oa = __shfl_xor_sync(0xffffffffu, best, off);
        const int oc = __shfl_xor_sync(0xffffffffu, bc, off);
        const int ok = __shfl_xor_sync(0xffffffffu, bk, off), oj = __shfl_xor_sync(0xffffffffu, bj, off);
        if (oa < best || (oa == best && oc < bc)) {
            best = oa;
            bc = oc;
            bk = ok;
            bj = oj;
        }
    }
    if (quad) {
        bk = (b.k0 + b.k1) >> 1;
        bj = (b.j0 + b.j1) >> 1;
    }
    // 0 upper left (local), 1 lower right (asymptotic), 2 upper right, 3 lower left
    const bool low = sub & 1, right = sub == 1 || sub == 2;
    *ch = SubBlk{low ? bk + 1 : b.k0, low ? b.k1 : bk, right ? bj + 1 : b.j0, right ? b.j1 : bj, b.prob};
    *cls = 0;
    if (!live || sub >= 4 || ch->k1 < ch->k0 || ch->j1 < ch->j0) return;
    if (quad) {
        *cls = 2;
    } else {
        const int s0 = st[ch->k0], s1 = st[ch->k1];
        *cls = classify_v(*ch, s0, s1, min_size);
    }
    if (may_exceed && *cls == 2 && asy_too_big(r_s + P.r_off, w_s + P.w_off, *ch)) *cls = 5;
}

// Whether some problem's whole range exceeds one FFT: only then can a block
// (the test loads its corner values otherwise, one more step of latency for
// every level).
__device__ __forceinline__ bool any_may_exceed(const double* __restrict__ r_s, const double* __restrict__ w_s,
                                               const ProbParams* __restrict__ probs, int nprob)
{
    bool big = false;
    for (int p = threadIdx.x; p < nprob; p += blockDim.x) {
        const ProbParams& P = probs[p];
        if (P.m > 0 && P.n > 0)
            big = big || !(0.5 * (r_s[P.r_off + P.n - 1] - r_s[P.r_off]) * 0.5 *
                               (w_s[P.w_off + P.m - 1] - w_s[P.w_off]) <= kAsyMaxXS);
    }
    return __syncthreads_or(big);
}

// The roots and the levels of up to max_level blocks, by one CTA: levels of up
// to kSubShared blocks stay in shared memory (sq), larger ones in the global
// queues.  Returns the size of the level left over (in qa) and whether the
// global queues were swapped an odd number of times.
__device__ __forceinline__ int64_t solo_walk(const int32_t* __restrict__ stair, const double* __restrict__ r_s,
                                             const double* __restrict__ w_s, const ProbParams* __restrict__ probs,
                                             int nprob, int64_t min_size, int n_cand, bool may_exceed, SubBlk*& qa,
                                             SubBlk*& qb, int64_t qcap, SubBlk* __restrict__ out, int64_t ocap,
                                             int64_t max_level, SubState& S, uint64_t* wsum,
                                             SubBlk (*sq)[kSubShared], int* swapped)
{
    if (threadIdx.x == 0) {
        S.nout[0] = S.nout[1] = S.nout[2] = 0;
        S.nnext = 0;
        S.ovf = 0;
    }
    __syncthreads();
    // the roots, one per problem
    for (int base = 0; base < nprob; base += kSubThreads) {
        const int p = base + threadIdx.x;
        SubBlk ch{0, -1, 0, -1, 0};
        int cls = 0;
        if (p < nprob) {
            const ProbParams& P = probs[p];
            ch = SubBlk{0, (int32_t)P.m - 1, 0, (int32_t)P.n - 1, p};
            cls = classify(stair + P.w_off, ch, min_size);
            if (cls == 2 && asy_too_big(r_s + P.r_off, w_s + P.w_off, ch)) cls = 5;
        }
        emit(ch, cls, S, wsum, out, ocap, qa, qcap, sq[0], nprob <= kSubThreads);
    }
    int64_t na = S.nnext;
    bool sh = S.shared;
    int cur = 0, sw = 0;
    while (na > 0 && na <= max_level && S.ovf == 0) {
        __syncthreads();   // every thread has read S.nnext, S.shared and S.ovf
        if (threadIdx.x == 0) S.nnext = 0;
        __syncthreads();
        const bool wide = na <= kSubThreads / 16;
        const int per = wide ? kSubThreads / 16 : kSubThreads / 4;   // blocks per chunk
        const SubBlk* lv = sh ? sq[cur] : qa;
        for (int64_t base = 0; base < na; base += per) {
            SubBlk ch;
            int cls;
            if (wide)
                make_child<16>(base + threadIdx.x / 16, na, lv, stair, r_s, w_s, probs, min_size, n_cand, may_exceed,
                               &ch, &cls);
            else
                make_child<4>(base + threadIdx.x / 4, na, lv, stair, r_s, w_s, probs, min_size, n_cand, may_exceed,
                              &ch, &cls);
            emit(ch, cls, S, wsum, out, ocap, qb, qcap, sq[cur ^ 1], na <= per);
        }
        na = S.nnext;
        sh = S.shared;
        cur ^= 1;
        SubBlk* tmp = qa;
        qa = qb;
        qb = tmp;
        sw ^= 1;
    }
    *swapped = sw;
    return na;
}

__global__ void __launch_bounds__(kSubThreads) k_subdivide(
    const int32_t* __restrict__ stair, const double* __restrict__ r_s, const double* __restrict__ w_s,
    const ProbParams* __restrict__ probs, int nprob, int64_t min_size,
    int n_cand, SubBlk* qa, SubBlk* qb, int64_t qcap, SubBlk* __restrict__ out, int64_t ocap,
    int64_t* __restrict__ res)
{
    __shared__ uint64_t wsum[kSubWarps];
    __shared__ SubState S;
    __shared__ SubBlk sq[2][kSubShared];
    int swapped;
    const bool big = any_may_exceed(r_s, w_s, probs, nprob);
    solo_walk(stair, r_s, w_s, probs, nprob, min_size, n_cand, big, qa, qb, qcap, out, ocap, (int64_t)1 << 62, S,
              wsum, sq, &swapped);
    if (threadIdx.x == 0) {
        res[0] = S.nout[0];
        res[1] = S.nout[1];
        res[2] = S.nout[2];
        res[3] = S.ovf;
    }
}

// Multi-CTA form of k_subdivide (cooperative launch).  CTA 0 walks the first
// levels alone, as k_subdivide, while a level holds at most kSubSolo blocks;
// from the first larger level on, every CTA takes consecutive chunks of
// kSubThreads / 4 blocks of a level.  After its block-wide scan a CTA publishes
// its four counts (ctot), and after a grid-wide barrier each CTA forms its
// chunk's offsets from the counts of the chunks before it: the offsets of the
// one-CTA walk, so the lists are the same entry for entry.  Every CTA keeps
// the same copy of the list counts (SubState), so all take the same number of
// barriers.  gst carries CTA 0's state to the others.
constexpr int64_t kSubSolo = 512;   // two chunks of 4-lane groups

__global__ void __launch_bounds__(kSubThreads) k_subdivide_grid(
    const int32_t* __restrict__ stair, const double* __restrict__ r_s, const double* __restrict__ w_s,
    const ProbParams* __restrict__ probs, int nprob, int64_t min_size,
    int n_cand, SubBlk* qa, SubBlk* qb, int64_t qcap, SubBlk* __restrict__ out, int64_t ocap,
    int64_t* __restrict__ res, int4* ctot, int64_t* gst)
{
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    __shared__ uint64_t wsum[kSubWarps];
    __shared__ SubState S;
    __shared__ int64_t cpre[4], ctall[4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ SubBlk sq[2][kSubShared];
    const bool big = any_may_exceed(r_s, w_s, probs, nprob);
    if (blockIdx.x == 0) {
        int swapped;
        const int64_t na = solo_walk(stair, r_s, w_s, probs, nprob, min_size, n_cand, big, qa, qb, qcap, out, ocap,
                                     kSubSolo, S, wsum, sq, &swapped);
        if (threadIdx.x == 0) {
            gst[0] = S.nout[0];
            gst[1] = S.nout[1];
            gst[2] = S.nout[2];
            gst[3] = na;
            gst[4] = S.ovf;
            gst[5] = swapped;
        }
    }
    grid.sync();
    if (threadIdx.x == 0) {
        S.nout[0] = gst[0];
        S.nout[1] = gst[1];
        S.nout[2] = gst[2];
        S.nnext = gst[3];
        S.ovf = (int)gst[4];
    }
    __syncthreads();
    if (blockIdx.x != 0 && gst[5]) {
        // the pending level is in the queue CTA 0 last wrote (CTA 0's own
        // pointers were swapped by its walk already)
        SubBlk* tmp = qa;
        qa = qb;
        qb = tmp;
    }
    int64_t na = S.nnext;
    const int64_t per_round = (int64_t)gridDim.x * (kSubThreads / 4);
    while (na > 0 && S.ovf == 0) {
        __syncthreads();   // every thread has read S.nnext and S.ovf
        if (threadIdx.x == 0) S.nnext = 0;
        __syncthreads();
        for (int64_t r0 = 0; r0 < na; r0 += per_round) {
            SubBlk ch;
            int cls;
            make_child<4>(r0 + (int64_t)blockIdx.x * (kSubThreads / 4) + threadIdx.x / 4, na, qa, stair, r_s, w_s,
                          probs, min_size, n_cand, big, &ch, &cls);
            uint64_t total;
            const uint64_t off = block_scan(class_count(cls), wsum, &total);
            if (threadIdx.x == 0)
                ctot[blockIdx.x] = make_int4((int)(total & 0xffff), (int)((total >> 16) & 0xffff),
                                             (int)((total >> 32) & 0xffff), (int)(total >> 48));
            grid.sync();
            if (warp == 0) {
                // counts of the chunks before this CTA's, and of the round
                int64_t a[4] = {0, 0, 0, 0}, tt[4] = {0, 0, 0, 0};
                for (int b = lane; b < (int)gridDim.x; b += 32) {
                    const int4 c = ctot[b];
                    const int64_t v[4] = {c.x, c.y, c.z, c.w};
                    for (int f = 0; f < 4; ++f) {
                        tt[f] += v[f];
                        if (b < (int)blockIdx.x) a[f] += v[f];
                    }
                }
                for (int f = 0; f < 4; ++f) {
                    for (int o = 16; o > 0; o >>= 1) {
                        a[f] += __shfl_xor_sync(0xffffffffu, a[f], o);
                        tt[f] += __shfl_xor_sync(0xffffffffu, tt[f], o);
                    }
                    if (lane == 0) {
                        cpre[f] = a[f];
                        ctall[f] = tt[f];
                    }
                }
            }
            __syncthreads();
            bool fits = S.ovf == 0;
            for (int c = 0; c < 3; ++c) fits = fits && S.nout[c] + ctall[c] <= ocap;
            fits = fits && S.nnext + ctall[3] <= qcap;
            if (fits) {
                const int64_t base[4] = {S.nout[0] + cpre[0], S.nout[1] + cpre[1], S.nout[2] + cpre[2],
                                         S.nnext + cpre[3]};
                place(ch, cls, off, base, out, ocap, qb);
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                if (fits) {
                    for (int c = 0; c < 3; ++c) S.nout[c] += ctall[c];
                    S.nnext += ctall[3];
                } else {
                    S.ovf = 1;
                }
            }
            grid.sync();   // ctot is rewritten by the next round; the next level reads this one's queue
        }
        na = S.nnext;
        SubBlk* tmp = qa;
        qa = qb;
        qb = tmp;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        res[0] = S.nout[0];
        res[1] = S.nout[1];
        res[2] = S.nout[2];
        res[3] = S.ovf;
    }
}

}  // namespace

int subdivide_grid_ctas()
{
    int dev = 0, sms = 0, coop = 0, nb = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_subdivide_grid, kSubThreads, 0) != cudaSuccess ||
        nb < 1)
        return 0;
    return sms < kSubGridMax ? sms : kSubGridMax;
}

cudaError_t launch_subdivide(const int32_t* stair, const double* r_s, const double* w_s, const ProbParams* probs,
                             int nprob, int64_t min_size,
                             int n_cand, SubBlk* qa, SubBlk* qb, int64_t qcap, SubBlk* out, int64_t ocap,
                             int64_t* res, int4* ctot, int64_t* gst, int grid_ctas, cudaStream_t s)
{
    if (grid_ctas > 1 && grid_ctas <= kSubGridMax && ctot && gst) {
        void* args[] = {(void*)&stair, (void*)&r_s, (void*)&w_s, (void*)&probs, (void*)&nprob, (void*)&min_size,
                        (void*)&n_cand, (void*)&qa, (void*)&qb, (void*)&qcap, (void*)&out, (void*)&ocap,
                        (void*)&res, (void*)&ctot, (void*)&gst};
        const cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_subdivide_grid, dim3(grid_ctas),
                                                          dim3(kSubThreads), args, 0, s);
        if (e == cudaSuccess) {
            count_launches(1);
            return cudaSuccess;
        }
        (void)cudaGetLastError();   // not launched: the one-CTA walk below
    }
    k_subdivide<<<1, kSubThreads, 0, s>>>(stair, r_s, w_s, probs, nprob, min_size, n_cand, qa, qb, qcap, out, ocap,
                                          res);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace nuht
