// Per-call input scaling, and the deterministic mode's conversion of the
// exact 128-bit sums (det_acc.cuh) back to FP64.
//
// The execute kernels hold the coefficients as double-float numbers (pairs of
// FP32), whose exponent range is FP32's.  Every call therefore first scales
// its input vector by 2^-E, E the exponent of the largest |x_i|, so that the
// largest magnitude lies in [1, 2), and scales the output back by 2^E: both
// exact in FP64, and the transform is linear, so any finite input range works.
#include <cstdint>
#include <map>
#include <mutex>
#include <utility>

#include "nuht_internal.h"

namespace nuht {

int device_sm_count();

namespace {

constexpr int kDetThreads = 256;

// Clears the accumulators of a call (Z) and writes every CTA's maximum |x_i|
// to part[blockIdx.x], as the bit pattern of a non-negative double (whose
// integer order is the order of the values); the gather kernel reduces the
// CTAs' maxima.  A maximum does not depend on the order, so the scale is the
// same on every run.  x may be absent, or weighted: |x[perm[i]] ws[i]| (i < nb,
// every vector of comps).
__global__ void __launch_bounds__(kDetThreads) k_prepare(ZeroList Z, const double* __restrict__ x, int64_t count,
                                                         const int32_t* __restrict__ perm,
                                                         const double* __restrict__ ws, int comps,
                                                         unsigned long long* __restrict__ part)
{
    __shared__ unsigned long long wmax[kDetThreads / 32];
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int z = 0; z < Z.n; ++z) {
        double2* p = (double2*)Z.p[z];
        const int64_t n2 = Z.bytes[z] / 16;
        for (int64_t i = t0; i < n2; i += step) p[i] = make_double2(0.0, 0.0);
        if (t0 == 0 && (Z.bytes[z] & 8)) ((double*)Z.p[z])[2 * n2] = 0.0;
    }
    if (!x) return;
    unsigned long long m = 0;
    for (int64_t i = t0; i < count; i += step) {
        double v;
        if (perm) {
            const int64_t i0 = i / comps;
            v = x[(int64_t)perm[i0] * comps + (i - i0 * comps)] * ws[i0];
        } else {
            v = x[i];
        }
        const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
        m = b > m ? b : m;
    }
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, off);
        m = o > m ? o : m;
    }
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kDetThreads / 32; ++w) m = wmax[w] > m ? wmax[w] : m;
        part[blockIdx.x] = m;
    }
}

__global__ void __launch_bounds__(kDetThreads) k_fx_decode(const Fx128* __restrict__ src, double* __restrict__ dst,
                                                           int64_t count, const ProbParams* __restrict__ probs)
{
    const int fxs = probs[0].fxs;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = fx_decode(src[i], fxs);
}

// CTAs of k_prepare: four elements a thread, at most kMaxParts
int prepare_parts(int64_t work)
{
    const int64_t need = (work + 4 * kDetThreads - 1) / (4 * kDetThreads);
    return (int)(need < 1 ? 1 : (need < kMaxParts ? need : kMaxParts));
}

int grid_for(int64_t count)
{
    const int64_t need = (count + kDetThreads - 1) / kDetThreads;
    const int64_t cap = (int64_t)device_sm_count() * 8;
    return (int)(need < 1 ? 1 : (need < cap ? need : cap));
}

}  // namespace

int device_sm_count()
{
    static int cache[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    if (dev >= 0 && dev < 64 && cache[dev] > 0) return cache[dev];
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 1;
    if (dev >= 0 && dev < 64) cache[dev] = sms;
    return sms;
}

cudaError_t allow_smem_of(const void* kernel, size_t bytes)
{
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, size_t> allowed;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    size_t& most = allowed[{kernel, dev}];
    if (bytes <= most) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) most = bytes;
    return e;
}

cudaError_t launch_prepare(const ZeroList& Z, const double* x, int64_t count, const int32_t* perm, const double* ws,
                           int comps, unsigned long long* part, int* parts, cudaStream_t s)
{
    if (!x && Z.n == 0) return cudaSuccess;
    int64_t work = x ? count : 0;
    for (int z = 0; z < Z.n; ++z) work = (int64_t)(Z.bytes[z] / 16) > work ? (int64_t)(Z.bytes[z] / 16) : work;
    const int grid = prepare_parts(work);
    if (parts) *parts = grid;
    k_prepare<<<grid, kDetThreads, 0, s>>>(Z, x, count, perm, ws, comps, part);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_fx_decode(const void* src, double* dst, int64_t count, const ProbParams* probs, cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    k_fx_decode<<<grid_for(count), kDetThreads, 0, s>>>((const Fx128*)src, dst, count, probs);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace nuht
