// FFTs of the asymptotic blocks (the inner transform of the type-3 NUFFT, see
// k_asy.cu):  Q_t = sum_l b_l / psi^(alpha2 l) e^{2 pi i l t / nf2} for the 2M
// grids of every block, nf2 a power of two, and the transposed transform of
// the adjoint.
//
// FP64 plans (and every adjoint): k_asy_fft, in double-float.  A block's
// transform runs in one to three passes (fft_split) over lines of 32..512
// points; every CTA takes a tile of up to kFftTileVals values -- some lines,
// each with a run of the block's Hankel terms q, which are adjacent in memory.
// Mixed-precision forward transforms: FP32 butterflies (the _f32 kernels).
#include <algorithm>
#include <cstdint>

#include "asy_dev.cuh"
#include "df64.cuh"
#include "nuht_internal.h"

namespace nuht {

int device_sm_count();

namespace {

// Complex double-float values are float4 (re.h, re.l, im.h, im.l).
__device__ __forceinline__ float4 cdf(df re, df im) { return make_float4(re.h, re.l, im.h, im.l); }

__device__ __forceinline__ float4 cdf_scale(float4 a, df s)
{
    return cdf(df_mul(df{a.x, a.y}, s), df_mul(df{a.z, a.w}, s));
}

// A finite double as double-float from its bits (integer and FP32
// instructions only; FP64 runs at 1/64 of the FP32 rate): the top 24 bits of
// the significand exactly, the next 29 rounded; zero and subnormals give 0.
__device__ __forceinline__ df df_from_bits(double x)
{
    const long long b = __double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return df{0.f, 0.f};
    const long long m = (b & 0xFFFFFFFFFFFFFLL) | (1LL << 52);   // x = +-m 2^(e - 1075)
    float h = ldexpf((float)(int)(m >> 29), e - 1075 + 29);
    float l = ldexpf((float)(int)(m & 0x1FFFFFFF), e - 1075);
    if (b < 0) {
        h = -h;
        l = -l;
    }
    return fast_two_sum(h, l);
}

// FP64 complex as double-float
__device__ __forceinline__ float4 cdf_from(double2 v)
{
    return cdf(df_from_bits(v.x), df_from_bits(v.y));
}

// 1 / psi^(alpha2 l): the correction of mode l of the inner FFT, in
// double-float (|l| <= N1 < 2^24 is exact in FP32).
__device__ __forceinline__ df mode_correction(const AsyBlock& B, const Tables& tab, int l)
{
    const df a2 = df_from_bits(B.alpha2);
    return df_recip(psihat_of(tab, df_mul(a2, df{(float)(l < 0 ? -l : l), 0.f})));
}

// ------------------------------------------------- double-float FFT passes
// Sums and differences with the low parts added but not renormalised: a value
// stays the exact sum of its parts to 2^-47 over the few levels of one
// register butterfly (8 instructions per real sum instead of 11); products
// and the stores between stages renormalise.
__device__ __forceinline__ float4 c_add(float4 a, float4 b)
{
    float s, e, t, f;
    two_sum(a.x, b.x, s, e);
    two_sum(a.z, b.z, t, f);
    return make_float4(s, e + (a.y + b.y), t, f + (a.w + b.w));
}

__device__ __forceinline__ float4 c_sub(float4 a, float4 b)
{
    float s, e, t, f;
    two_sum(a.x, -b.x, s, e);
    two_sum(a.z, -b.z, t, f);
    return make_float4(s, e + (a.y - b.y), t, f + (a.w - b.w));
}

__device__ __forceinline__ float4 c_neg(float4 a) { return make_float4(-a.x, -a.y, -a.z, -a.w); }
__device__ __forceinline__ float4 c_mul_i(float4 a) { return make_float4(-a.z, -a.w, a.x, a.y); }

__device__ __forceinline__ float4 c_norm(float4 a)
{
    return cdf(fast_two_sum(a.x, a.y), fast_two_sum(a.z, a.w));
}

// a b + c d in double-float as one compensated sum of the two products.
__device__ __forceinline__ df df_dot2(df a, df b, df c, df d)
{
    const float p = a.h * b.h, q = c.h * d.h;
    float s, e;
    two_sum(p, q, s, e);
    e += fmaf(a.h, b.h, -p) + fmaf(c.h, d.h, -q);
    e = fmaf(a.h, b.l, e);
    e = fmaf(a.l, b.h, e);
    e = fmaf(c.h, d.l, e);
    e = fmaf(c.l, d.h, e);
    return fast_two_sum(s, e);
}

__device__ __forceinline__ float4 c_mul(float4 a, float4 b)
{
    const df ar{a.x, a.y}, ai{a.z, a.w}, br{b.x, b.y}, bi{b.z, b.w};
    return cdf(df_dot2(ar, br, ai, df{-bi.h, -bi.l}), df_dot2(ar, bi, ai, br));
}

// a e^{i pi / 4}
__device__ __forceinline__ float4 c_mul_w8(float4 a)
{
    const df c{0.707106769084930419921875f, 1.21016175e-8f};   // sqrt(1/2)
    float s, e, t, f;
    two_sum(a.x, -a.z, s, e);
    two_sum(a.x, a.z, t, f);
    return cdf(df_mul(df{s, e + (a.y - a.w)}, c), df_mul(df{t, f + (a.y + a.w)}, c));
}

// y_k = sum_p x_p e^{2 pi i p k / 4}, in place, natural order.
__device__ __forceinline__ void dft4(float4& x0, float4& x1, float4& x2, float4& x3)
{
    const float4 a = c_add(x0, x2), b = c_sub(x0, x2), c = c_add(x1, x3), d = c_mul_i(c_sub(x1, x3));
    x0 = c_add(a, c);
    x1 = c_add(b, d);
    x2 = c_sub(a, c);
    x3 = c_sub(b, d);
}

template <int R>
__device__ __forceinline__ void dft(float4 (&x)[R]);

template <>
__device__ __forceinline__ void dft<4>(float4 (&x)[4])
{
    dft4(x[0], x[1], x[2], x[3]);
}

// The even outputs are the DFT of u_p = x_p + x_{p+4}, the odd ones of
// v_p = (x_p - x_{p+4}) e^{2 pi i p / 8}.
__device__ __forceinline__ void dft8_tail(float4 (&x)[8], float4 u0, float4 u1, float4 u2, float4 u3, float4 v0,
                                          float4 v1, float4 v2, float4 v3)
{
    v1 = c_mul_w8(v1);
    v2 = c_mul_i(v2);
    v3 = c_mul_i(c_mul_w8(v3));
    dft4(u0, u1, u2, u3);
    dft4(v0, v1, v2, v3);
    x[0] = u0; x[2] = u1; x[4] = u2; x[6] = u3;
    x[1] = v0; x[3] = v1; x[5] = v2; x[7] = v3;
}

template <>
__device__ __forceinline__ void dft<8>(float4 (&x)[8])
{
    dft8_tail(x, c_add(x[0], x[4]), c_add(x[1], x[5]), c_add(x[2], x[6]), c_add(x[3], x[7]), c_sub(x[0], x[4]),
              c_sub(x[1], x[5]), c_sub(x[2], x[6]), c_sub(x[3], x[7]));
}

// The same for x_2 = .. = x_5 = 0: the first stage of a forward transform,
// whose input fills a quarter of the points at either end.
__device__ __forceinline__ void dft8_outer(float4 (&x)[8])
{
    dft8_tail(x, x[0], x[1], x[6], x[7], x[0], x[1], c_neg(x[6]), c_neg(x[7]));
}

// e^{2 pi i k / 2^tw_log2}, 0 <= k < 2^tw_log2, from the table of its first half.
__device__ __forceinline__ float4 tw_at(const Tables& tab, int k)
{
    const int half = 1 << (tab.tw_log2 - 1);
    const float4 t = tab.tw2[k & (half - 1)];
    return (k & half) ? c_neg(t) : t;
}

// e^{2 pi i m / N} for 0 <= m < N = 2^logN as double-float: the table entry for
// the top bits of m / N times the rotation by the rest, an angle below
// 2 pi / 2^tw_log2, from its Taylor series (five terms, truncation < 1e-19).
__device__ __forceinline__ float4 cdf_twiddle(const Tables& tab, int logN, long long m)
{
    const int sh = logN - tab.tw_log2;
    const float4 t = tw_at(tab, sh > 0 ? (int)(m >> sh) : (int)(m << -sh));
    const int lo = sh > 0 ? (int)(m & ((1LL << sh) - 1)) : 0;
    if (lo == 0) return t;
    // angle 2 pi lo / N: lo / N is exact in FP32 (lo < 2^sh <= 2^11, N a power of two)
    const df twopi{6.2831854820251465f, -1.7484555314695172e-07f};
    const df a = df_mul(twopi, df{ldexpf((float)lo, -logN), 0.f});
    const df a2 = df_mul(a, a);
    // sin a = a (1 - a^2/6 (1 - a^2/20 (1 - a^2/42))), cos a = 1 - a^2/2 (1 - a^2/12 (1 - a^2/30))
    df sn = df_add(df{1.f, 0.f}, df_negate(df_mul(a2, df{1.f / 42.f, 0.f})));
    sn = df_add(df{1.f, 0.f}, df_negate(df_mul(df_mul(a2, df{0.05f, -7.450580707946131e-10f}), sn)));
    sn = df_add(df{1.f, 0.f}, df_negate(df_mul(df_mul(a2, df{0.1666666716337204f, -4.967053879312289e-09f}), sn)));
    sn = df_mul(a, sn);
    df cs = df_add(df{1.f, 0.f}, df_negate(df_mul(a2, df{0.03333333507180214f, -1.7384682293e-09f})));
    cs = df_add(df{1.f, 0.f}, df_negate(df_mul(df_mul(a2, df{0.0833333358168602f, -2.4835269e-09f}), cs)));
    cs = df_add(df{1.f, 0.f}, df_negate(df_mul(df_mul(a2, df{0.5f, 0.f}), cs)));
    return c_mul(t, cdf(cs, sn));
}

// What a CTA of one pass works on (see k_asy_fft).
struct FftGeom {
    int lg, len;         // line length
    int lgst;            // log2 of the row stride between a line's points
    int lgl, cq;         // log2 lines of the tile, Hankel terms of the tile
    int l0, q0;          // its first line and term
    int Q, N, N1;
    // row of point p of tile line l (in place for all but the last pass)
    __device__ __forceinline__ int row(int l, int p) const
    {
        const int x = l0 + l;
        return (x & ((1 << lgst) - 1)) + ((x >> lgst) << (lgst + lg)) + (p << lgst);
    }
    // shared-memory index of (point, line, term)
    __device__ __forceinline__ int at(int p, int l, int q) const { return ((p << lgl) + l) * cq + q; }
    // signed mode of row t
    __device__ __forceinline__ int mode(int t) const { return t < (N >> 1) ? t : t - N; }
};

// One radix-R stage of every line of the tile: sub-transforms of n = 2^lgn
// points (grp of them per line, one after the other).  Item (grp, m, line, q)
// takes the points m + p n/R, leaves output k of the radix-R DFT, times
// e^{2 pi i m k / n}, at m + k n/R: the next stage's sub-transform grp R + k.
// ld(pos, p, line, q) and st(pos, k, line, q, value): pos = grp n + m + p n/R.
template <int R, bool OUTER, bool TWIDDLE, class Ld, class St>
__device__ __forceinline__ void fft_stage(const FftGeom& G, const Tables& tab, int lgn, Ld&& ld, St&& st)
{
    constexpr int lgR = R == 8 ? 3 : 2;
    const int lgm = lgn - lgR;
    const int nitems = ((G.len >> lgR) << G.lgl) * G.cq;
    for (int i = threadIdx.x; i < nitems; i += blockDim.x) {
        const int rest = i / G.cq, q = i - rest * G.cq;
        const int l = rest & ((1 << G.lgl) - 1), gm = rest >> G.lgl;
        const int m = gm & ((1 << lgm) - 1), grp = gm >> lgm;
        const int pos = (grp << lgn) + m;
        float4 x[R];
#pragma unroll
        for (int p = 0; p < R; ++p) x[p] = (OUTER && p >= 2 && p < 6) ? make_float4(0.f, 0.f, 0.f, 0.f) : ld(pos + (p << lgm), l, q);
        if constexpr (OUTER) dft8_outer(x);
        else dft<R>(x);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            float4 v = x[k];
            if (TWIDDLE && k > 0) v = c_mul(v, tw_at(tab, (m * k) << (tab.tw_log2 - lgn)));
            else v = c_norm(v);
            st(pos + (k << lgm), grp, k, l, q, v);
        }
    }
}

// One pass of the blocks' transforms; work item = tile g * (q chunks) + chunk
// of a block.  N = nf2 points in rows [t][Q].
//   one pass:     the whole line, src -> dst
//   two passes:   N = N1 N2.  Pass 0: for each n1, the FFT over n2 of
//     x[n1 + N1 n2], times e^{2 pi i n1 k2 / N}, at tmp[n1 + N1 k2]; pass 1: for
//     each k2, the FFT over n1 of tmp[n1 + N1 k2], which is X[k2 + N2 k1].
//   three passes: pass 1 splits its lines of N1 = A B points the same way in
//     place (n1 = a + A b), pass 2 writes X[k2 + N2 (kb + B ka)].
// Forward (ADJ = false): pass 0 reads the modes |l| <= N1 of the spread grid
// src (at b_off), corrected by 1/psi^(alpha2 l) -- a quarter of the points at
// either end, since nf2 >= 2 (2 N1 + 1) -- and the last pass stores the rows
// the interpolation can read, |t| <= tmax (about nf2/4), at dst + q_off.
// Transposed (ADJ): those rows of the target grid src (at q_off) are
// transformed (the DFT matrix is symmetric) and only the modes |l| <= N1 are
// kept, corrected, and stored at dst + b_off.
//
// Bound: issue slots of the double-float butterflies.  A line's first stage
// reads global memory and its last stage writes it, radix 8 (or 4) in
// registers between, so a value crosses shared memory two or four times
// instead of once per two levels and once more bit-reversed; lanes run over
// the terms q first, so that a warp moves whole 128-byte rows (2M = 8) and no
// two lanes of a quarter-warp meet in a bank; the mode corrections and the
// twiddles between passes are formed once per point and serve all terms of
// the tile.  Measured against the kernels this replaced (radix-4 stages from
// bit-reversed shared memory, one term per CTA, corrections and twiddles
// formed for each term): 1080 + 580 instructions per value in two passes and
// L1 74-88 % busy; now 413 + 355 + 283 in three.  FFT of 2^23 points x 8 terms
// 4.65 -> 2.61 ms (64 bytes per value and pass: 2.4 TB/s), n = m = 1e6 (3200
// blocks) 0.235 -> 0.105, five launches -> two or three; 2500 x 3000 points
// forward + adjoint FFTs 118 -> 41 us.
template <bool ADJ, bool FIRST>
__global__ void __launch_bounds__(kFftThreads, 5)
k_asy_fft(const ProbParams* __restrict__ probs, const AsyBlock* __restrict__ blks, const Tile* __restrict__ items,
          Tables tab, int pass, const double2* __restrict__ src, float4* tmp, float4* __restrict__ dst,
          int64_t src_stride, int64_t tmp_stride, int64_t dst_stride)
{
    extern __shared__ float4 Xs[];
    const Tile it = items[blockIdx.x];
    const AsyBlock& B = blks[it.blk];
    const int64_t b_off = B.b_off, q_off = B.q_off;
    const int LN = B.log2nf2;
    FftGeom G;
    G.Q = probs[B.prob].Q;
    G.N = 1 << LN;
    G.N1 = B.N1;
    const FftSplit S = fft_split(LN);
    const FftTile T = fft_tile(LN, pass, G.Q);
    const bool last = pass + 1 == S.np;
    G.lg = T.lg;
    G.len = 1 << T.lg;
    G.lgst = S.lgst(pass);
    G.lgl = T.lgl;
    const int g = (int)it.start / T.nqc, ch = (int)it.start - g * T.nqc;
    G.l0 = g << T.lgl;
    G.q0 = ch * T.qc;
    G.cq = G.Q - G.q0 < T.qc ? G.Q - G.q0 : T.qc;
    src += blockIdx.y * src_stride;   // member blockIdx.y of a batch of real components
    tmp += blockIdx.y * tmp_stride + q_off;
    dst += blockIdx.y * dst_stride;
    const int npt = G.len << G.lgl;
    float4* tw = Xs + npt * G.cq;             // twiddles between passes, [point][line]
    float2* corr = (float2*)tw;               // mode corrections (before tw is needed), [point][line]
    // output row of the last pass: lines are (kb, k2), kb fastest, B = 2^lgB
    const int lgB = S.np == 3 ? S.lg1 : 0, lgN2 = S.np > 1 ? S.lg0 : 0;
    auto out_row = [&](int l, int k) {
        const int x = G.l0 + l;
        return (x >> lgB) + ((x & ((1 << lgB) - 1)) << lgN2) + (k << (lgN2 + lgB));
    };
    if ((FIRST && !ADJ) || (ADJ && last)) {
        for (int e = threadIdx.x; e < npt; e += blockDim.x) {
            const int p = e >> G.lgl, l = e & ((1 << G.lgl) - 1);
            const int md = G.mode(ADJ ? out_row(l, p) : G.row(l, p));
            if (md >= -G.N1 && md <= G.N1) {
                const df c = mode_correction(B, tab, md);
                corr[e] = make_float2(c.h, c.l);
            }
        }
        __syncthreads();
    }
    const int zero_lo = B.tmax, zero_hi = G.N - B.tmax;   // rows between are outside the window
    auto ld_first = [&](int p, int l, int q) -> float4 {
        const int t = G.row(l, p);
        if (!FIRST) return tmp[(int64_t)t * G.Q + G.q0 + q];
        if (ADJ) {
            if (t > zero_lo && t < zero_hi) return make_float4(0.f, 0.f, 0.f, 0.f);
            return cdf_from(src[q_off + (int64_t)t * G.Q + G.q0 + q]);
        }
        const int md = G.mode(t);
        if (md < -G.N1 || md > G.N1) return make_float4(0.f, 0.f, 0.f, 0.f);
        const float2 c = corr[(p << G.lgl) + l];
        return cdf_scale(cdf_from(src[b_off + (int64_t)(md + G.N1) * G.Q + G.q0 + q]), df{c.x, c.y});
    };
    auto st_sm = [&](int pos, int, int, int l, int q, float4 v) { Xs[G.at(pos, l, q)] = v; };
    auto ld_sm = [&](int pos, int l, int q) { return Xs[G.at(pos, l, q)]; };
    // stage 0: radix 8, global -> shared
    fft_stage<8, FIRST && !ADJ, true>(G, tab, G.lg, ld_first, st_sm);
    if (!last) {
        __syncthreads();   // corr is no longer read
        const int lgw = G.lg + G.lgst;
        for (int e = threadIdx.x; e < npt; e += blockDim.x) {
            const int k = e >> G.lgl, x = (G.l0 + (e & ((1 << G.lgl) - 1))) & ((1 << G.lgst) - 1);
            tw[e] = cdf_twiddle(tab, lgw, (long long)x * k);
        }
    }
    __syncthreads();
    // a middle stage for lines of more than 64 points
    int lgn = G.lg - 3, lgg = 3, lg2 = 0;   // sub-transform, log2 of the sub-transforms per line, the middle stage's radix
    if (lgn > 3) {
        lg2 = lgn == 4 ? 2 : 3;
        if (lg2 == 3) fft_stage<8, false, true>(G, tab, lgn, ld_sm, st_sm);
        else fft_stage<4, false, true>(G, tab, lgn, ld_sm, st_sm);
        __syncthreads();
        lgn -= lg2;
        lgg += lg2;
    }
    // last stage: shared -> global.  Sub-transform grp holds the outputs
    // k1 + 8 k2 (+ 8 R2 k3 for output k3 of this stage) with grp = k1 R2 + k2
    auto st_out = [&](int, int grp, int k3, int l, int q, float4 v) {
        const int k = (grp >> lg2) + ((grp & ((1 << lg2) - 1)) << 3) + (k3 << lgg);
        if (!last) {
            tmp[(int64_t)G.row(l, k) * G.Q + G.q0 + q] = c_mul(v, tw[(k << G.lgl) + l]);
            return;
        }
        const int t = out_row(l, k);
        if (ADJ) {
            const int md = G.mode(t);
            if (md < -G.N1 || md > G.N1) return;
            const float2 c = corr[(k << G.lgl) + l];
            dst[b_off + (int64_t)(md + G.N1) * G.Q + G.q0 + q] = cdf_scale(v, df{c.x, c.y});
        } else if (t <= zero_lo || t >= zero_hi) {
            dst[q_off + (int64_t)t * G.Q + G.q0 + q] = v;
        }
    };
    if (lgn == 3) fft_stage<8, false, false>(G, tab, lgn, ld_sm, st_out);
    else fft_stage<4, false, false>(G, tab, lgn, ld_sm, st_out);
}

// ------------------------------------------------- mixed precision (FP32)
// nlines independent FFTs (e^{+2 pi i k n / N}) of N = 2^logN FP32 complex
// values (float2: re, im) stored one after the other in shared memory, each in
// bit-reversed order, sharing every butterfly stage; tw2[k] = e^{2 pi i k /
// 2^tw_log2}.  The decimation-in-time stages run two at a time (radix 4); an
// odd stage count starts with one radix-2 stage (twiddle 1).
__device__ __forceinline__ void cf2_bfly(float2& u, float2& v, float4 w)
{
    const float vr = v.x * w.x - v.y * w.z, vi = fmaf(v.x, w.z, v.y * w.x);
    const float ur = u.x, ui = u.y;
    u = make_float2(ur + vr, ui + vi);
    v = make_float2(ur - vr, ui - vi);
}

__device__ void smem_fft_lines_f32(float2* X, int logN, int nlines, const float4* __restrict__ tw2, int tw_log2)
{
    const int N = 1 << logN;
    int st = 0;
    if (logN & 1) {
        const int half = N >> 1;
        for (int b = threadIdx.x; b < nlines * half; b += blockDim.x) {
            const int i0 = 2 * b;
            const float2 u = X[i0], v = X[i0 + 1];
            X[i0] = make_float2(u.x + v.x, u.y + v.y);
            X[i0 + 1] = make_float2(u.x - v.x, u.y - v.y);
        }
        __syncthreads();
        st = 1;
    }
    const int quarter = N >> 2;
    for (; st < logN; st += 2) {
        const int len = 1 << st;
        const int sh1 = tw_log2 - (st + 1), sh2 = tw_log2 - (st + 2);
        for (int b = threadIdx.x; b < nlines * quarter; b += blockDim.x) {
            const int line = b >> (logN - 2);
            const int bb = b & (quarter - 1);
            const int pos = bb & (len - 1);
            const int i0 = line * N + ((bb >> st) << (st + 2)) + pos;
            float2 a = X[i0], c1 = X[i0 + len], c2 = X[i0 + 2 * len], c3 = X[i0 + 3 * len];
            const float4 t1 = tw2[pos << sh1];
            cf2_bfly(a, c1, t1);
            cf2_bfly(c2, c3, t1);
            cf2_bfly(a, c2, tw2[pos << sh2]);
            cf2_bfly(c1, c3, tw2[(pos + len) << sh2]);
            X[i0] = a;
            X[i0 + len] = c1;
            X[i0 + 2 * len] = c2;
            X[i0 + 3 * len] = c3;
        }
        __syncthreads();
    }
}

__device__ __forceinline__ float2 cf2_of(float4 v) { return make_float2(v.x, v.z); }
__device__ __forceinline__ float4 cf4_of(float2 v) { return make_float4(v.x, 0.f, v.y, 0.f); }

// Split of a two-pass FFT of 2^LN points into lines: N2 = 2^ceil(LN/2)
// points per pass-A line, N1 = 2^floor(LN/2) per pass-B line; each CTA takes
// as many lines as fit kFftLineBatch points.
struct FourStep {
    int logN1, logN2, N1, N2, lpcA, lpcB, groupsA, groupsB;
};
__host__ __device__ __forceinline__ FourStep four_step(int LN)
{
    FourStep f;
    f.logN2 = (LN + 1) >> 1;
    f.logN1 = LN - f.logN2;
    f.N1 = 1 << f.logN1;
    f.N2 = 1 << f.logN2;
    f.lpcA = kFftLineBatch >> f.logN2; if (f.lpcA < 1) f.lpcA = 1;
    f.lpcB = kFftLineBatch >> f.logN1; if (f.lpcB < 1) f.lpcB = 1;
    f.groupsA = (f.N1 + f.lpcA - 1) / f.lpcA;
    f.groupsB = (f.N2 + f.lpcB - 1) / f.lpcB;
    return f;
}

// Value tt of a block's FFT input: mode l of the spread grid (|l| <= N1),
// corrected by 1/psi^(alpha2 l), rounded to FP32 complex.
__device__ __forceinline__ float2 fft_in_f32(const AsyBlock& B, const Tables& tab, const double2* __restrict__ src,
                                             int Q, int q, int tt)
{
    const int l = (tt < (B.nf2 >> 1)) ? tt : tt - B.nf2;
    if (l < -B.N1 || l > B.N1) return make_float2(0.f, 0.f);
    return cf2_of(cdf_scale(cdf_from(src[B.b_off + (int64_t)(l + B.N1) * Q + q]), mode_correction(B, tab, l)));
}

__global__ void k_asy_fft_small_f32(const ProbParams* __restrict__ probs, const AsyBlock* __restrict__ blks,
                                    const Tile* __restrict__ items, Tables tab,
                                    const double2* __restrict__ src, float4* __restrict__ dst, int64_t src_stride,
                                    int64_t dst_stride)
{
    extern __shared__ float2 Xf[];
    src += blockIdx.y * src_stride;   // member blockIdx.y of a batch of real components
    dst += blockIdx.y * dst_stride;
    const Tile it = items[blockIdx.x];
    const AsyBlock B = blks[it.blk];
    const int Q = probs[B.prob].Q;
    const int q = (int)it.start;
    const int N = B.nf2, logN = B.log2nf2;
    for (int tt = threadIdx.x; tt < N; tt += blockDim.x)
        Xf[__brev(tt) >> (32 - logN)] = fft_in_f32(B, tab, src, Q, q, tt);
    __syncthreads();
    smem_fft_lines_f32(Xf, logN, 1, tab.tw2, tab.tw_log2);
    for (int tt = threadIdx.x; tt < N; tt += blockDim.x) dst[B.q_off + (int64_t)tt * Q + q] = cf4_of(Xf[tt]);
}

// All Q grids of one small block (nf2 * Q <= kFftSmemMax) by one CTA: the
// deconvolution factor of each mode is computed once and used for every q;
// the Q transforms share every butterfly stage.
__device__ __forceinline__ void fft_whole_f32(const AsyBlock& B, int Q, const Tables& tab,
                                              const double2* __restrict__ src, float4* __restrict__ dst, float2* Xf)
{
    const int N = B.nf2, logN = B.log2nf2, half = N >> 1;
    for (int tt = threadIdx.x; tt < N; tt += blockDim.x) {
        const int l = (tt < half) ? tt : tt - N;
        const int dst_i = __brev(tt) >> (32 - logN);
        if (l < -B.N1 || l > B.N1) {
            for (int q = 0; q < Q; ++q) Xf[q * N + dst_i] = make_float2(0.f, 0.f);
        } else {
            const df sc = mode_correction(B, tab, l);
            const double2* row = src + B.b_off + (int64_t)(l + B.N1) * Q;
            for (int q = 0; q < Q; ++q) Xf[q * N + dst_i] = cf2_of(cdf_scale(cdf_from(row[q]), sc));
        }
    }
    __syncthreads();
    smem_fft_lines_f32(Xf, logN, Q, tab.tw2, tab.tw_log2);
    float4* gq = dst + B.q_off;
    for (int idx = threadIdx.x; idx < N * Q; idx += blockDim.x) {
        const int tt = idx / Q, q = idx - tt * Q;
        gq[idx] = cf4_of(Xf[q * N + tt]);
    }
}

// The blocks with pts_lo < nf2 * Q <= pts_hi.  SCAN = false (the small class,
// nearly all blocks): one CTA per item, the others return at once.  SCAN (the
// few large ones): every thread of a CTA looks at one item, the items a grid
// apart, and the CTA transforms those of the class that it found.  With a CTA
// per item here too, 1.26e5 CTAs of which almost none had work took 0.11 of
// the 0.64 ms of a complex mixed-precision transform's FFTs (n = m = 4e6).
template <bool SCAN>
__global__ void k_asy_fft_block_f32(const ProbParams* __restrict__ probs, const AsyBlock* __restrict__ blks,
                                    const Tile* __restrict__ items, int nitems, Tables tab,
                                    const double2* __restrict__ src, float4* __restrict__ dst, int pts_lo,
                                    int pts_hi, int64_t src_stride, int64_t dst_stride)
{
    extern __shared__ float2 Xf[];   // [Q][N], each grid bit-reversed
    src += blockIdx.y * src_stride;   // member blockIdx.y of a batch of real components
    dst += blockIdx.y * dst_stride;
    if constexpr (!SCAN) {
        const AsyBlock B = blks[items[blockIdx.x].blk];
        const int Q = probs[B.prob].Q, pts = B.nf2 * Q;
        if (pts > pts_lo && pts <= pts_hi) fft_whole_f32(B, Q, tab, src, dst, Xf);
    } else {
        __shared__ int found[256], nfound;
        for (int64_t base = 0; base < nitems; base += (int64_t)blockDim.x * gridDim.x) {
            if (threadIdx.x == 0) nfound = 0;
            __syncthreads();
            const int64_t i = base + (int64_t)threadIdx.x * gridDim.x + blockIdx.x;
            if (i < nitems) {
                const int b = items[i].blk;
                const int pts = blks[b].nf2 * probs[blks[b].prob].Q;
                if (pts > pts_lo && pts <= pts_hi) found[atomicAdd(&nfound, 1)] = b;
            }
            __syncthreads();
            const int nf = nfound;
            for (int f = 0; f < nf; ++f) {
                const AsyBlock B = blks[found[f]];
                fft_whole_f32(B, probs[B.prob].Q, tab, src, dst, Xf);
                __syncthreads();   // Xf is rewritten by the next block, found by the next round
            }
        }
    }
}

// Two-pass (four-step) FFT for nf2 = N1 * N2 > kFftSingleMax.
// Pass A: for each n1, FFT over n2 of x[n1 + N1 n2], times e^{2 pi i n1 k2 / N},
// stored at tmp[n1 + N1 k2].  Pass B: for each k2, FFT over n1 of
// tmp[n1 + N1 k2], which is X[k2 + N2 k1].  Work item ordinal = g * Q + q,
// g a group of lines handled by one CTA: the Q CTAs of a group run side by
// side and read and write the same rows of the [point][Q] grids (one row is
// all Q values of a point), so a row moves through HBM once, not once per q.
__global__ void k_asy_fft_pass_a_f32(const ProbParams* __restrict__ probs, const AsyBlock* __restrict__ blks,
                                     const Tile* __restrict__ items, Tables tab,
                                     const double2* __restrict__ src, float2* __restrict__ tmp)
{
    extern __shared__ float2 Xf[];
    const Tile it = items[blockIdx.x];
    const AsyBlock B = blks[it.blk];
    const int Q = probs[B.prob].Q;
    const int N = B.nf2;
    const FourStep f = four_step(B.log2nf2);
    const int g = (int)(it.start / Q);
    const int iq = (int)(it.start - (int64_t)g * Q);
    const int l0 = g * f.lpcA;
    const int nl = (f.N1 - l0) < f.lpcA ? (f.N1 - l0) : f.lpcA;
    for (int idx = threadIdx.x; idx < nl * f.N2; idx += blockDim.x) {
        const int li = idx >> f.logN2, n2 = idx & (f.N2 - 1);
        Xf[li * f.N2 + (__brev(n2) >> (32 - f.logN2))] = fft_in_f32(B, tab, src, Q, iq, (l0 + li) + f.N1 * n2);
    }
    __syncthreads();
    smem_fft_lines_f32(Xf, f.logN2, nl, tab.tw2, tab.tw_log2);
    for (int idx = threadIdx.x; idx < nl * f.N2; idx += blockDim.x) {
        const int li = idx >> f.logN2, k2 = idx & (f.N2 - 1);
        const int n1 = l0 + li;
        const long long m = ((long long)n1 * k2) & (N - 1);   // e^{2 pi i n1 k2 / N}
        // FP32 twiddle (m / N is exact in FP32, N <= 2^24)
        float sn, cs;
        sincospif(ldexpf(2.f * (float)m, -B.log2nf2), &sn, &cs);
        const float2 x = Xf[idx];
        tmp[B.q_off + (int64_t)(n1 + f.N1 * k2) * Q + iq] =
            make_float2(x.x * cs - x.y * sn, fmaf(x.x, sn, x.y * cs));
    }
}

__global__ void k_asy_fft_pass_b_f32(const ProbParams* __restrict__ probs, const AsyBlock* __restrict__ blks,
                                     const Tile* __restrict__ items, Tables tab,
                                     const float2* __restrict__ tmp, float4* __restrict__ dst)
{
    extern __shared__ float2 Xf[];
    const Tile it = items[blockIdx.x];
    const AsyBlock B = blks[it.blk];
    const int Q = probs[B.prob].Q;
    const FourStep f = four_step(B.log2nf2);
    const int g = (int)(it.start / Q);
    const int iq = (int)(it.start - (int64_t)g * Q);
    const int k20 = g * f.lpcB;
    const int nl = (f.N2 - k20) < f.lpcB ? (f.N2 - k20) : f.lpcB;
    for (int idx = threadIdx.x; idx < nl * f.N1; idx += blockDim.x) {
        const int li = idx >> f.logN1, n1 = idx & (f.N1 - 1);
        const int i = li * f.N1 + (f.logN1 > 0 ? (__brev(n1) >> (32 - f.logN1)) : 0);
        Xf[i] = tmp[B.q_off + (int64_t)(n1 + f.N1 * (k20 + li)) * Q + iq];
    }
    __syncthreads();
    smem_fft_lines_f32(Xf, f.logN1, nl, tab.tw2, tab.tw_log2);
    for (int idx = threadIdx.x; idx < nl * f.N1; idx += blockDim.x) {
        const int li = idx >> f.logN1, k1 = idx & (f.N1 - 1);
        dst[B.q_off + (int64_t)((k20 + li) + f.N2 * k1) * Q + iq] = cf4_of(Xf[idx]);
    }
}

}  // namespace

size_t fft_smem_bytes(int max_log2, int pass, int Q)
{
    size_t most = 0;
    for (int LN = 5; LN <= max_log2; ++LN) {
        const FftSplit S = fft_split(LN);
        if (pass >= S.np) continue;
        const FftTile T = fft_tile(LN, pass, Q);
        const size_t pts = (size_t)1 << (T.lg + T.lgl);
        const size_t b = sizeof(float4) * pts * T.qc + (S.np > 1 ? sizeof(float4) : sizeof(float2)) * pts;
        if (b > most) most = b;
    }
    return most;
}

cudaError_t launch_asy_fft(const ProbParams* probs, const AsyBlock* blks, const Tile* items, int nitems,
                           size_t smem, int pass, Tables tab, const double2* src, float4* tmp, float4* dst,
                           cudaStream_t s, bool adj, int members, int64_t src_stride, int64_t tmp_stride,
                           int64_t dst_stride)
{
    if (nitems <= 0) return cudaSuccess;
    if (members < 1 || members > 65535) return cudaErrorInvalidValue;
    auto kern = pass == 0 ? (adj ? k_asy_fft<true, true> : k_asy_fft<false, true>)
                          : (adj ? k_asy_fft<true, false> : k_asy_fft<false, false>);
    cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(nitems, members), kFftThreads, smem, s>>>(probs, blks, items, tab, pass, src, tmp, dst, src_stride,
                                                          tmp_stride, dst_stride);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_asy_fft_small_f32(const ProbParams* probs, const AsyBlock* blks, const Tile* items,
                                     int nitems, int max_nf2, Tables tab, const double2* src, float4* dst,
                                     cudaStream_t s, int members, int64_t src_stride, int64_t dst_stride)
{
    if (nitems <= 0) return cudaSuccess;
    if (members < 1 || members > 65535) return cudaErrorInvalidValue;
    size_t smem = sizeof(float2) * (size_t)max_nf2;
    cudaError_t e = allow_smem(k_asy_fft_small_f32, smem);
    if (e != cudaSuccess) return e;
    int nt = max_nf2 / 2;
    if (nt > 256) nt = 256;
    if (nt < 32) nt = 32;
    k_asy_fft_small_f32<<<dim3(nitems, members), nt, smem, s>>>(probs, blks, items, tab, src, dst, src_stride,
                                                                dst_stride);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_asy_fft_block_f32(const ProbParams* probs, const AsyBlock* blks, const Tile* items,
                                     int nitems, int max_pts, Tables tab, const double2* src, float4* dst,
                                     cudaStream_t s, int members, int64_t src_stride, int64_t dst_stride)
{
    if (nitems <= 0) return cudaSuccess;
    if (members < 1 || members > 65535) return cudaErrorInvalidValue;
    if (max_pts < 1 || max_pts > kFftSmemMax) max_pts = kFftSmemMax;
    // blocks of up to kFftSmallPts points in small CTAs (8 KiB, many per SM),
    // the larger ones in CTAs sized for the largest
    constexpr int kFftSmallPts = 1024;
    const int scan_ctas = 8 * device_sm_count();   // at least eight CTAs per SM look for the larger ones
    const int ranges[2][2] = {{0, max_pts < kFftSmallPts ? max_pts : kFftSmallPts}, {kFftSmallPts, max_pts}};
    int launched = 0;
    for (int r = 0; r < 2; ++r) {
        const int lo = ranges[r][0], hi = ranges[r][1];
        if (hi <= lo) continue;
        const size_t smem = sizeof(float2) * (size_t)hi;
        int nt = ((hi / 2 + 31) / 32) * 32;
        if (r == 0 && nt > 128) nt = 128;
        if (nt > 256) nt = 256;
        if (nt < 32) nt = 32;
        auto kern = r ? k_asy_fft_block_f32<true> : k_asy_fft_block_f32<false>;
        cudaError_t e = allow_smem(kern, smem);
        if (e != cudaSuccess) return e;
        int gx = nitems;
        if (r) gx = std::min(nitems, std::max((nitems + nt - 1) / nt, scan_ctas));
        kern<<<dim3(gx, members), nt, smem, s>>>(probs, blks, items, nitems, tab, src, dst, lo, hi, src_stride,
                                                 dst_stride);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        ++launched;
    }
    count_launches(launched);
    return cudaSuccess;
}

cudaError_t launch_asy_fft_large_f32(const ProbParams* probs, const AsyBlock* blks, const Tile* items_a,
                                     int nitems_a, const Tile* items_b, int nitems_b, Tables tab,
                                     const double2* src, float2* tmp, float4* dst, cudaStream_t s)
{
    if (nitems_a <= 0) return cudaSuccess;
    size_t smem = sizeof(float2) * (size_t)kFftLineBatch;
    k_asy_fft_pass_a_f32<<<nitems_a, 256, smem, s>>>(probs, blks, items_a, tab, src, tmp);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_asy_fft_pass_b_f32<<<nitems_b, 256, smem, s>>>(probs, blks, items_b, tab, tmp, dst);
    count_launches(2);
    return cudaGetLastError();
}

}  // namespace nuht
