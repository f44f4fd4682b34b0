// Work lists of a plan, built on the device from the block lists of the
// subdivision (Algorithm 1): per-block descriptors (local expansion, Sec. 3.1;
// type-3 geometry of the asymptotic blocks, Sec. 3.2 / 4.2; direct blocks),
// the offsets of their moments and grids, and the tile segments of every
// kernel.  Two kernels: sizes (one thread per block; the CTA that finishes last
// also forms the column-wise prefix over the CTAs' sums) and fill (one thread
// per block).  The block counts are read from device memory, so nothing here
// waits for the host.
#include <cmath>
#include <cstdint>

#include "nuht_internal.h"

namespace nuht {

namespace {

__device__ __forceinline__ int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

__device__ __forceinline__ void atomic_max64(int64_t* p, int64_t v)
{
    atomicMax((unsigned long long*)p, (unsigned long long)v);   // values are non-negative
}

__device__ __forceinline__ int64_t clamp_count(int64_t c, int64_t cap) { return c < cap ? c : cap; }

// Rows of class y (0 local, 1 asymptotic, 2 direct), its counter columns and
// the place of their totals.
__device__ __forceinline__ int64_t class_rows(const BlockBuild& bb, int y) { return clamp_count(bb.res[y], bb.ocap); }
__device__ __forceinline__ int class_cols(int y) { return y == 0 ? kLocalCols : (y == 1 ? kAsyCols : kDirCols); }
__device__ __forceinline__ int class_total(int y) { return y == 0 ? TOT_LOCAL : (y == 1 ? TOT_ASY : TOT_DIR); }

// Descriptor and counters of one block; maxima into smax (shared).
__device__ __forceinline__ void block_size_one(const BlockBuild& bb, int y, int64_t i, unsigned long long* smax)
{
    auto maxv = [&](int k, int64_t v) { atomicMax(&smax[k], (unsigned long long)v); };
    {
        if (y == 0) {
            const SubBlk b = bb.sub[i];
            const ProbParams& P = bb.probs[b.prob];
            LocalBlock lb{};
            lb.prob = b.prob;
            lb.k0 = (int32_t)(b.k0 + P.w_off); lb.k1 = (int32_t)(b.k1 + P.w_off);
            lb.j0 = (int32_t)(b.j0 + P.r_off); lb.j1 = (int32_t)(b.j1 + P.r_off);
            lb.R = bb.r_s[lb.j1];
            lb.R_h = (float)lb.R;
            lb.R_l = (float)(lb.R - (double)lb.R_h);
            const double iR = lb.R > 0.0 ? 1.0 / lb.R : 0.0;
            lb.iR_h = (float)iR;
            lb.iR_l = (float)(iR - (double)lb.iR_h);
            bb.loc[i] = lb;
            const int64_t rows = b.k1 - b.k0 + 1, cols = b.j1 - b.j0 + 1;
            int64_t* c = bb.lcnt + i * kLocalCols;
            c[LC_MOM] = P.L + 1;
            c[LC_TMOM] = ceil_div(cols, bb.mom_tile);
            c[LC_TEVAL] = ceil_div(rows, bb.eval_tile);
            c[LC_RC] = rows + cols;
        } else if (y == 1) {
            const int64_t a = i;
            const SubBlk b = bb.sub[bb.ocap + a];
            const ProbParams& P = bb.probs[b.prob];
            struct { double x, y, z, w; } e;   // r_j0, r_j1, omega_k0, omega_k1
            e.x = bb.r_s[P.r_off + b.j0]; e.y = bb.r_s[P.r_off + b.j1];
            e.z = bb.w_s[P.w_off + b.k0]; e.w = bb.w_s[P.w_off + b.k1];
            const int Q = P.Q;
            AsyBlock ab{};
            ab.prob = b.prob;
            ab.k0 = (int32_t)(b.k0 + P.w_off); ab.k1 = (int32_t)(b.k1 + P.w_off);
            ab.j0 = (int32_t)(b.j0 + P.r_off); ab.j1 = (int32_t)(b.j1 + P.r_off);
            // r_c rounded to a multiple of 2^(10 - fr) (any centre serves the
            // type-3 transform); the fixed-point frame keeps r < 2^(62 - fr)
            int er;
            frexp(e.y, &er);
            ab.fr = 62 - er;
            ab.rc = ldexp(rint(ldexp(0.5 * (e.x + e.y), ab.fr - 10)), 10 - ab.fr);
            ab.Rc_fx = (int64_t)ldexp(ab.rc, ab.fr);
            const double X = 0.5 * (e.y - e.x);
            {
                // w_c rounded to a multiple of 2^(10 - fw), like r_c
                int eo;
                frexp(e.w, &eo);
                ab.fw = 62 - eo;
                ab.wc = ldexp(rint(ldexp(0.5 * (e.z + e.w), ab.fw - 10)), 10 - ab.fw);
                ab.Wc_fx = (int64_t)ldexp(ab.wc, ab.fw);
            }
            const double S = 0.5 * (e.w - e.z);
            // a single frequency (S = 0) takes any spacing: one that puts the
            // block's points within a few cells (scale-free, unlike a constant)
            const double Seff = S > 0.0 ? S : (X > 0.0 ? 1.0 / X : 1.0);
            ab.h = M_PI / (2.0 * Seff);
            ab.inv_h = (2.0 / M_PI) * Seff;
            {
                int eh, ew;
                frexp(ab.inv_h, &eh);
                ab.KH = (int64_t)ldexp(ab.inv_h, 62 - eh);      // exact: 53-bit mantissa
                ab.sA = ab.fr + 62 - eh - 41;
                // w_c / (2 pi) in double-double, then 62 bits of it
                const double c_hi = 0.15915494309189535, c_lo = -9.839338337591243e-18;
                const double p = ab.wc * c_hi;
                const double err = fma(ab.wc, c_hi, -p) + ab.wc * c_lo;
                frexp(p, &ew);
                int64_t kw = llrint(ldexp(p, 62 - ew)) + llrint(ldexp(err, 62 - ew));
                int sw = ab.fr + 62 - ew - 64;
                if (sw > 64) {
                    kw = sw - 64 < 63 ? kw >> (sw - 64) : 0;
                    sw = 64;
                }
                ab.KW = kw;
                ab.sW = sw;
            }
            const bool fx_bad = ab.sA < 1 || ab.sA > 127 || ab.sW < 0;
            const double n1f = ceil(X * ab.inv_h + 0.5 * bb.w) + 1.0;   // one cell of rounding margin
            int64_t* c = bb.acnt + a * kAsyCols;
            for (int k = 0; k < kAsyCols; ++k) c[k] = 0;
            bb.fcls[a] = -1;
            if (fx_bad || !(n1f <= (double)(1 << 22))) {
                maxv(MX_ERR, 1);
                return;
            }
            ab.N1 = (int32_t)n1f;
            const int64_t nf1 = 2 * (int64_t)ab.N1 + 1;
            int lg = 64 - __clzll((long long)(2 * nf1 - 1));   // smallest 2^lg >= 2 nf1
            if (lg < 5) lg = 5;
            if (lg > kFftMaxLog2) {
                maxv(MX_ERR, 1);
                return;
            }
            ab.log2nf2 = lg;
            ab.nf2 = 1 << lg;
            ab.rho = e.x;
            ab.alpha = 0.5 * bb.w * ab.h;
            ab.alpha2 = ldexp(bb.w * M_PI, -lg);
            ab.inv_delta = ab.nf2 * (0.5 / M_PI);
            ab.hd = ab.h * ab.inv_delta;
            ab.alpha_h = (float)ab.alpha;
            ab.alpha_l = (float)(ab.alpha - (double)ab.alpha_h);
            {
                int ed, er2;
                frexp(ab.hd, &ed);
                ab.KD = (int64_t)ldexp(ab.hd, 62 - ed);          // exact: 53-bit mantissa
                ab.sD = ab.fw + 62 - ed - 40;   // 40 fractional bits: |s hd| <= nf2 / 4 <= 2^22
                const double c_hi = 0.15915494309189535, c_lo = -9.839338337591243e-18;
                const double p = ab.rc * c_hi;
                const double err = fma(ab.rc, c_hi, -p) + ab.rc * c_lo;
                frexp(p, &er2);
                int64_t kr = llrint(ldexp(p, 62 - er2)) + llrint(ldexp(err, 62 - er2));
                int sr = ab.fw + 62 - er2 - 64;
                if (sr > 64) {
                    kr = sr - 64 < 63 ? kr >> (sr - 64) : 0;
                    sr = 64;
                }
                ab.KRc = kr;
                ab.sR = sr;
                if (ab.sD < 1 || ab.sD > 127 || sr < 0) {
                    maxv(MX_ERR, 1);
                    return;
                }
            }
            {
                // the largest FFT-grid position of a frequency, and w cells around it
                const double te = ceil(fmax(e.w - ab.wc, ab.wc - e.z) * ab.hd) + bb.w + 2.0;
                ab.tmax = te < (double)ab.nf2 ? (int32_t)te : ab.nf2;
            }
            ab.rho_h = (float)ab.rho;
            ab.rho_l = (float)(ab.rho - (double)ab.rho_h);
            bb.asy[a] = ab;
            const int64_t rows = b.k1 - b.k0 + 1, cols = b.j1 - b.j0 + 1;
            c[AC_GB] = nf1 * Q;
            c[AC_GQ] = (int64_t)ab.nf2 * Q;
            c[AC_TSPREAD] = ceil_div(cols, bb.spread_tile);
            c[AC_TINTERP] = ceil_div(rows, bb.interp_tile);
            maxv(MX_LOG2, lg);
            {
                const int np = fft_split(lg).np;
                c[AC_IP0] = fft_tile(lg, 0, Q).ntiles;
                c[AC_NP1] = np > 1;
                c[AC_NP2] = np > 2;
                if (np > 1) c[AC_IP1] = fft_tile(lg, 1, Q).ntiles;
                if (np > 2) c[AC_IP2] = fft_tile(lg, 2, Q).ntiles;
            }
            if (!bb.lowp) {
                // double-float FFTs only
            } else if ((int64_t)ab.nf2 * Q <= kFftSmemMax) {      // all Q grids in one CTA
                bb.fcls[a] = 0;
                c[AC_NFK] = 1;
                c[AC_IFK] = 1;
                maxv(MX_FBLOCK_PTS, (int64_t)ab.nf2 * Q);
            } else if (ab.nf2 <= kFftSingleMax) {                 // one CTA per grid
                bb.fcls[a] = 1;
                c[AC_NFS] = 1;
                c[AC_IFS] = Q;
                maxv(MX_NF2_SMALL, ab.nf2);
            } else {                                              // two passes, groups of lines
                bb.fcls[a] = 2;
                c[AC_NFL] = 1;
                const int logN2 = (lg + 1) >> 1, logN1 = lg - logN2;
                const int lpcA = (kFftLineBatch >> logN2) > 0 ? (kFftLineBatch >> logN2) : 1;
                const int lpcB = (kFftLineBatch >> logN1) > 0 ? (kFftLineBatch >> logN1) : 1;
                c[AC_IFA] = (int64_t)Q * (((1 << logN1) + lpcA - 1) / lpcA);
                c[AC_IFB] = (int64_t)Q * (((1 << logN2) + lpcB - 1) / lpcB);
            }
            c[AC_RC] = rows + cols;
            c[AC_NF2] = ab.nf2;
        } else {
            const int64_t d = i;
            const SubBlk b = bb.sub[2 * bb.ocap + d];
            const ProbParams& P = bb.probs[b.prob];
            bb.dir[d] = DirectBlock{b.prob, (int32_t)(b.k0 + P.w_off), (int32_t)(b.k1 + P.w_off),
                                    (int32_t)(b.j0 + P.r_off), (int32_t)(b.j1 + P.r_off), 0};
            const int64_t rows = b.k1 - b.k0 + 1, cols = b.j1 - b.j0 + 1;
            bb.dcnt[d] = rows * cols;
            maxv(MX_DIR_ROWS, rows);
            maxv(MX_DIR_COLS, cols);
            maxv(MX_DIR_AREA, rows * cols);
        }
    }
}

// Sizes, descriptors and counters of every block (CTA = kBlockTile rows of
// class blockIdx.y), the CTAs' column sums, and by the CTA that finishes last
// their exclusive prefix and the totals (four launches before: sizes and three
// of scans).  Bound by the latency of each asymptotic row's FP64 geometry, whose
// instructions a warp issues 16 cycles apart: 64 rows per CTA spread it over
// more SMs than 256 did (23 -> 16 us at 700 asymptotic blocks), and the other
// warps help with the prefix.
constexpr int kSizeThreads = 256;
__global__ void __launch_bounds__(kSizeThreads) k_block_sizes(BlockBuild bb)
{
    __shared__ unsigned long long smax[kMaxv], ssum[kAsyCols];
    __shared__ bool is_last;
    const int y = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t rows = class_rows(bb, y);
    if ((int64_t)blockIdx.x * kBlockTile >= rows) return;   // whole CTA
    if (threadIdx.x < kMaxv) smax[threadIdx.x] = 0;
    if (threadIdx.x < kAsyCols) ssum[threadIdx.x] = 0;
    __syncthreads();
    const int64_t i = threadIdx.x < kBlockTile ? (int64_t)blockIdx.x * kBlockTile + threadIdx.x : rows;
    if (i < rows) block_size_one(bb, y, i, smax);
    __syncthreads();
    const int ncol = class_cols(y);
    const int64_t* mat = y == 0 ? bb.lcnt : (y == 1 ? bb.acnt : bb.dcnt);
    for (int c = 0; threadIdx.x < kBlockTile && c < ncol; ++c) {
        int64_t v = i < rows ? mat[i * ncol + c] : 0;   // this thread's own stores
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0 && v) atomicAdd(&ssum[c], (unsigned long long)v);
    }
    __syncthreads();
    if (threadIdx.x < ncol)
        bb.part[((int64_t)y * bb.ptiles + blockIdx.x) * kAsyCols + threadIdx.x] = (int64_t)ssum[threadIdx.x];
    if (threadIdx.x < kMaxv && smax[threadIdx.x]) atomic_max64(&bb.maxv[threadIdx.x], (int64_t)smax[threadIdx.x]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned active = 0;
        for (int k = 0; k < 3; ++k) active += (unsigned)ceil_div(class_rows(bb, k), kBlockTile);
        is_last = atomicAdd(bb.ticket, 1u) + 1 == active;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    // one warp per column, four tiles per lane and step
    for (int col = warp; col < kTotals; col += kSizeThreads / 32) {
        const int k = col >= TOT_DIR ? 2 : (col >= TOT_ASY ? 1 : 0), c = col - class_total(k);
        const int64_t nt = ceil_div(class_rows(bb, k), kBlockTile);
        int64_t* pc = bb.part + (int64_t)k * bb.ptiles * kAsyCols + c;
        int64_t carry = 0;
        for (int64_t t0 = 0; t0 < nt; t0 += 128) {
            const int64_t t = t0 + 4 * lane;
            int64_t v[4], sum = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = t + u < nt ? __ldcg((const long long*)(pc + (t + u) * kAsyCols)) : 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) sum += v[u];
            int64_t x = sum;
            for (int off = 1; off < 32; off <<= 1) {
                const int64_t o = __shfl_up_sync(0xffffffffu, x, off);
                if (lane >= off) x += o;
            }
            int64_t run = carry + x - sum;   // exclusive offset of the lane's first tile
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (t + u < nt) pc[(t + u) * kAsyCols] = run;
                run += v[u];
            }
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) bb.totals[col] = carry;
    }
}

// Exclusive prefix sums of NCOL counters over all rows of a class: c[] of this
// thread's row, the tile's offset from part.
template <int NCOL>
__device__ __forceinline__ void class_prefix(const BlockBuild& bb, int y, const int64_t* row, bool live, int64_t* c,
                                             int64_t (*wsum)[kBlockTile / 32])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NCOL; ++k) {
        const int64_t v = live ? row[k] : 0;
        int64_t x = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int64_t o = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += o;
        }
        if (lane == 31) wsum[k][warp] = x;
        c[k] = x - v;
    }
    __syncthreads();
    const int64_t* part = bb.part + ((int64_t)y * bb.ptiles + blockIdx.x) * kAsyCols;
#pragma unroll
    for (int k = 0; k < NCOL; ++k) {
        int64_t p = part[k];
        for (int w = 0; w < warp; ++w) p += wsum[k][w];
        c[k] += p;
    }
}

__device__ __forceinline__ void put_seg(const BuildLists& L, int list, int64_t idx, int32_t blk, int32_t len,
                                        int64_t first, int64_t last, int64_t prefix)
{
    L.seg[list][idx] = Seg{blk, len, first, last};
    L.pre[list][idx] = (int32_t)prefix;
}

__global__ void __launch_bounds__(kBlockTile) k_block_fill(BlockBuild bb, BuildLists L)
{
    const int64_t nl = clamp_count(bb.res[0], bb.ocap), na = clamp_count(bb.res[1], bb.ocap),
                  nd = clamp_count(bb.res[2], bb.ocap);
    const int64_t* tl = bb.totals + TOT_LOCAL;
    const int64_t* ta = bb.totals + TOT_ASY;
    __shared__ int64_t wsum[kAsyCols][kBlockTile / 32];
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        *L.status = 0;
        // closing entries of the prefix arrays
        L.pre[LIST_MOM][nl] = (int32_t)tl[LC_TMOM];
        L.pre[LIST_EVAL][nl] = (int32_t)tl[LC_TEVAL];
        L.pre[LIST_SPREAD][na] = (int32_t)ta[AC_TSPREAD];
        L.pre[LIST_INTERP][na] = (int32_t)ta[AC_TINTERP];
        L.pre[LIST_FBLOCK][ta[AC_NFK]] = (int32_t)ta[AC_IFK];
        L.pre[LIST_FSMALL][ta[AC_NFS]] = (int32_t)ta[AC_IFS];
        L.pre[LIST_FA][ta[AC_NFL]] = (int32_t)ta[AC_IFA];
        L.pre[LIST_FB][ta[AC_NFL]] = (int32_t)ta[AC_IFB];
        L.pre[LIST_P0][na] = (int32_t)ta[AC_IP0];
        L.pre[LIST_P1][ta[AC_NP1]] = (int32_t)ta[AC_IP1];
        L.pre[LIST_P2][ta[AC_NP2]] = (int32_t)ta[AC_IP2];
    }
    const int y = blockIdx.y;
    const int64_t rows = y == 0 ? nl : (y == 1 ? na : nd), i = (int64_t)blockIdx.x * kBlockTile + threadIdx.x;
    if ((int64_t)blockIdx.x * kBlockTile >= rows) return;   // whole CTA
    const bool live = i < rows;
    {
        if (y == 0) {
            int64_t c[kLocalCols];
            class_prefix<kLocalCols>(bb, y, bb.lcnt + i * kLocalCols, live, c, wsum);
            if (!live) return;
            LocalBlock lb = bb.loc[i];
            lb.mom_off = c[LC_MOM];
            L.loc[i] = lb;
            put_seg(L, LIST_MOM, i, (int32_t)i, bb.mom_tile, lb.j0, lb.j1, c[LC_TMOM]);
            put_seg(L, LIST_EVAL, i, (int32_t)i, bb.eval_tile, lb.k0, lb.k1, c[LC_TEVAL]);
            L.blk[i] = SubBlk{lb.k0, lb.k1, lb.j0, lb.j1, lb.prob};
        } else if (y == 1) {
            const int64_t a = i;
            int64_t c[kAsyCols];
            class_prefix<kAsyCols>(bb, y, bb.acnt + a * kAsyCols, live, c, wsum);
            if (!live) return;
            AsyBlock ab = bb.asy[a];
            ab.b_off = c[AC_GB];
            ab.q_off = c[AC_GQ];
            L.asy[a] = ab;
            put_seg(L, LIST_SPREAD, a, (int32_t)a, bb.spread_tile, ab.j0, ab.j1, c[AC_TSPREAD]);
            put_seg(L, LIST_INTERP, a, (int32_t)a, bb.interp_tile, ab.k0, ab.k1, c[AC_TINTERP]);
            const int Q = bb.probs[ab.prob].Q;
            const int np = fft_split(ab.log2nf2).np;
            put_seg(L, LIST_P0, a, (int32_t)a, 1, 0, fft_tile(ab.log2nf2, 0, Q).ntiles - 1, c[AC_IP0]);
            if (np > 1)
                put_seg(L, LIST_P1, c[AC_NP1], (int32_t)a, 1, 0, fft_tile(ab.log2nf2, 1, Q).ntiles - 1, c[AC_IP1]);
            if (np > 2)
                put_seg(L, LIST_P2, c[AC_NP2], (int32_t)a, 1, 0, fft_tile(ab.log2nf2, 2, Q).ntiles - 1, c[AC_IP2]);
            if (bb.fcls[a] < 0) {
                // no FP32 FFT
            } else if (bb.fcls[a] == 0) {
                put_seg(L, LIST_FBLOCK, c[AC_NFK], (int32_t)a, 1, 0, 0, c[AC_IFK]);
            } else if (bb.fcls[a] == 1) {
                put_seg(L, LIST_FSMALL, c[AC_NFS], (int32_t)a, 1, 0, Q - 1, c[AC_IFS]);
            } else {
                const int lg = ab.log2nf2;
                const int logN2 = (lg + 1) >> 1, logN1 = lg - logN2;
                const int lpcA = (kFftLineBatch >> logN2) > 0 ? (kFftLineBatch >> logN2) : 1;
                const int lpcB = (kFftLineBatch >> logN1) > 0 ? (kFftLineBatch >> logN1) : 1;
                const int64_t ia = (int64_t)Q * (((1 << logN1) + lpcA - 1) / lpcA);
                const int64_t ib = (int64_t)Q * (((1 << logN2) + lpcB - 1) / lpcB);
                put_seg(L, LIST_FA, c[AC_NFL], (int32_t)a, 1, 0, ia - 1, c[AC_IFA]);
                put_seg(L, LIST_FB, c[AC_NFL], (int32_t)a, 1, 0, ib - 1, c[AC_IFB]);
            }
            L.blk[nl + a] = SubBlk{ab.k0, ab.k1, ab.j0, ab.j1, ab.prob};
        } else if (live) {
            const int64_t d = i;
            const DirectBlock db = bb.dir[d];
            L.dir[d] = db;
            L.blk[nl + na + d] = SubBlk{db.k0, db.k1, db.j0, db.j1, db.prob};
        }
    }
}

}  // namespace

static cudaError_t block_grid(int64_t tiles, dim3* grid)
{
    if (tiles < 1 || tiles > 0x7fffffff) return cudaErrorInvalidValue;
    *grid = dim3((unsigned)tiles, 3);
    return cudaSuccess;
}

cudaError_t launch_block_build(const BlockBuild& bb, cudaStream_t s)
{
    dim3 grid;
    const cudaError_t e = block_grid(bb.ptiles, &grid);   // the counts are still on the device
    if (e != cudaSuccess) return e;
    k_block_sizes<<<grid, kSizeThreads, 0, s>>>(bb);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_block_fill(const BlockBuild& bb, const BuildLists& L, int64_t max_rows, cudaStream_t s)
{
    dim3 grid;
    const cudaError_t e = block_grid((max_rows > 0 ? max_rows + kBlockTile - 1 : kBlockTile) / kBlockTile, &grid);
    if (e != cudaSuccess) return e;
    k_block_fill<<<grid, kBlockTile, 0, s>>>(bb, L);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace nuht
