// Rows of the resin and the voxel error rate's bookkeeping, shared by ver.cu and osmo.cu.
//
// The resin of a row y is a run of x (voxel centres within r_inner of the axis): one pair of
// ends per y, decided in FP64 once per handle (resin_span_kernel), replaces an FP64 test and
// two 64-bit divisions per voxel; kernels take a row per warp.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "internal.cuh"

namespace vamrt {
namespace {

constexpr int kBins = kVerBins;
constexpr int kRowThreads = 512;

__device__ __forceinline__ float ldd(const float *p) { return *p; }
__device__ __forceinline__ float ldd(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
__device__ __forceinline__ float ldd(const __half *p) { return __half2float(*p); }
__device__ __forceinline__ void std_(float *p, float x) { *p = x; }
__device__ __forceinline__ void std_(__nv_bfloat16 *p, float x) { *p = __float2bfloat16_rn(x); }
__device__ __forceinline__ void std_(__half *p, float x) { *p = __float2half_rn(x); }
// x as storage type T holds it
template <typename T>
__device__ __forceinline__ float stored(float x)
{
    T t;
    std_(&t, x);
    return ldd(&t);
}

// *out = max(*out, the block's maximum of m); values >= 0 order like their bit patterns
__device__ __forceinline__ void block_max(float m, float *out)
{
    __shared__ int sh[32];
    const int v = __reduce_max_sync(0xffffffffu, __float_as_int(m));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        const int w = __reduce_max_sync(0xffffffffu, threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0);
        if (threadIdx.x == 0 && w) atomicMax(reinterpret_cast<int *>(out), w);
    }
}

// Two 1024-bin histograms in shared memory: sh[0..1023] in-part, sh[1024..2047] out-of-part.
__device__ __forceinline__ void hist_clear(unsigned *sh)
{
    for (int i = threadIdx.x; i < 2 * kBins; i += blockDim.x) sh[i] = 0u;
}
// a voxel of dose x falls in bin min(floor(x * (1024 / max)), 1023) (FP32)
__device__ __forceinline__ void hist_add(unsigned *sh, float x, float scale, bool part)
{
    const int b = min(max((int)floorf(x * scale), 0), kBins - 1);
    atomicAdd(&sh[(part ? 0 : kBins) + b], 1u);
}
__device__ __forceinline__ float hist_scale(float m) { return m > 0.f ? (float)kBins / m : 0.f; }   // all zero: bin 0
__device__ __forceinline__ void hist_flush(const unsigned *sh, unsigned *hist)
{
    for (int i = threadIdx.x; i < 2 * kBins; i += blockDim.x)
        if (sh[i]) atomicAdd(&hist[i], sh[i]);
}

// True in every thread of the block that arrives last (the others' results are then visible).
__device__ __forceinline__ bool last_block(unsigned *counter)
{
    __shared__ unsigned order;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) order = atomicAdd(counter, 1u);
    __syncthreads();
    if (order != gridDim.x - 1) return false;
    __threadfence();
    return true;
}

// By one block of kRowThreads: out[0] = fewest mismatches over the thresholds i = 1..1023 ("x >=
// tau_i" is "bin >= i"), out[1] = the first threshold with that many, out[2] = resin voxels.
__device__ __forceinline__ void ver_scan(const unsigned *hist, long long *out)
{
    static_assert(kBins == 2 * kRowThreads, "two bins per thread");
    __shared__ unsigned wi[kRowThreads / 32], wo[kRowThreads / 32];
    __shared__ unsigned long long wb[kRowThreads / 32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const unsigned i0 = __ldcg(hist + 2 * t), i1 = __ldcg(hist + 2 * t + 1);
    const unsigned o0 = __ldcg(hist + kBins + 2 * t), o1 = __ldcg(hist + kBins + 2 * t + 1);
    // inclusive sums over the threads
    unsigned si = i0 + i1, so = o0 + o1;
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned a = __shfl_up_sync(0xffffffffu, si, d), b = __shfl_up_sync(0xffffffffu, so, d);
        if (lane >= d) {
            si += a;
            so += b;
        }
    }
    if (lane == 31) {
        wi[w] = si;
        wo[w] = so;
    }
    __syncthreads();
    unsigned all_i = 0, all_o = 0;
    for (int k = 0; k < kRowThreads / 32; ++k) {
        if (k == w) {
            si += all_i;
            so += all_o;
        }
        all_i += wi[k];
        all_o += wo[k];
    }
    // thresholds 2 t and 2 t + 1: in-part bins below, out-of-part bins at or above
    const unsigned in0 = si - i0 - i1, out0 = all_o - (so - o0 - o1);
    unsigned long long best = t > 0 ? ((unsigned long long)(in0 + out0) << 32) | (unsigned)(2 * t) : ~0ull;
    const unsigned long long odd = ((unsigned long long)(in0 + i0 + out0 - o0) << 32) | (unsigned)(2 * t + 1);
    best = min(best, odd);
    for (int d = 16; d > 0; d >>= 1) best = min(best, __shfl_down_sync(0xffffffffu, best, d));
    if (lane == 0) wb[w] = best;
    __syncthreads();
    if (t == 0) {
        for (int k = 1; k < kRowThreads / 32; ++k) best = min(best, wb[k]);
        out[0] = (long long)(best >> 32);
        out[1] = (long long)(best & 0xffffffffu);
        out[2] = (long long)all_i + all_o;
    }
}

inline unsigned row_grid(const vamrt_projector *p, int blocks_per_sm)
{
    const int64_t rows = (int64_t)p->g.ny * p->g.nz, warps = kRowThreads / 32;
    const int64_t want = (rows + warps - 1) / warps, cap = (int64_t)p->num_sms * blocks_per_sm;
    return (unsigned)(want < cap ? want : cap);
}

}  // namespace
}  // namespace vamrt
