// What the convolution kernels' epilogues share: bias, ReLU and storage of 16 channels of one
// voxel, and the barriers of an epilogue warp set.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace vamrt {
namespace {

template <typename OT>
__device__ __forceinline__ void store16(OT *dst, const uint32_t *v, const float *bias, int relu)
{
    float r[16];
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
        const float4 b4 = bias ? __ldg((const float4 *)(bias + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
        r[i] = __uint_as_float(v[i]) + b4.x;
        r[i + 1] = __uint_as_float(v[i + 1]) + b4.y;
        r[i + 2] = __uint_as_float(v[i + 2]) + b4.z;
        r[i + 3] = __uint_as_float(v[i + 3]) + b4.w;
    }
    if (relu) {
#pragma unroll
        for (int i = 0; i < 16; ++i) r[i] = fmaxf(r[i], 0.f);
    }
    if constexpr (sizeof(OT) == 2) {
        uint32_t p[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(r[2 * i], r[2 * i + 1]);
            p[i] = *(const uint32_t *)&h;
        }
        uint4 *d = (uint4 *)dst;
        d[0] = make_uint4(p[0], p[1], p[2], p[3]);
        d[1] = make_uint4(p[4], p[5], p[6], p[7]);
    } else {
        float4 *d = (float4 *)dst;
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
    }
}

// the 128 threads of epilogue set `set` (warps 4 set .. 4 set + 3) agree on a flag
// (named barrier 1 + set)
__device__ __forceinline__ bool epi_all(bool v, int set)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, %2, 128, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v), "r"(1 + set)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void epi_sync(int set) { asm volatile("bar.sync %0, 128;" ::"r"(1 + set) : "memory"); }

}  // namespace
}  // namespace vamrt
