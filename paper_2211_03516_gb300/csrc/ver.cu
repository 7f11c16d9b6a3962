// Voxel error rate of a dose against a binary target: the fraction of resin voxels whose
// printed state (dose above a threshold) differs from the target, at the best of 1023
// thresholds tau_i = (i / 1024) max(dose), i = 1..1023, the maximum taken over the resin.  It measures how well a dose
// prints the part independently of the dose's scale, the quantity the optimiser's
// stopping rule is after (Sec. 2.7).
//
// Exact integer bookkeeping: each resin voxel falls in bin b = min(floor(x * (1024/max)),
// 1023) (FP32, the dose's precision), so "x >= tau_i" is "b >= i"; two 1024-bin histograms
// (in-part, out-of-part) give every threshold's mismatch count by prefix sums.  Resin =
// voxel centres within r_inner of the axis (decided in FP64).
//
// Two passes over the resin's rows in 16-byte reads (single ones where rows are not 16-byte
// aligned): the maximum, then the histograms, whose last block also scans them.  384 x 384 x 512, BF16 dose:
// 38 us for the maximum's 119 MB and 87 us for the histograms' 356 MB (4.1 TB/s; the bins'
// shared-memory atomics come next), against 1443, 1455 and 50 us of a pass per voxel with an
// FP64 test and 64-bit divisions and a serial scan.
#include "exact_div.cuh"
#include "resin.cuh"

namespace vamrt {
namespace {

// V consecutive voxels of a row as they are stored: 16 bytes from an aligned address, or one voxel
template <int V, typename T>
struct Group {
    static constexpr int kWords = (V * (int)sizeof(T) + 15) / 16;
    uint4 w[kWords];
    __device__ __forceinline__ void load(const T *p)
    {
#pragma unroll
        for (int k = 0; k < kWords; ++k) w[k] = __ldg(reinterpret_cast<const uint4 *>(p) + k);
    }
    __device__ __forceinline__ float operator[](int i) const
    {
        constexpr int kPer = 16 / (int)sizeof(T);
        const uint4 q = w[i / kPer];
        const int j = i % kPer * (int)sizeof(T) / 4;
        const unsigned u = j == 0 ? q.x : j == 1 ? q.y : j == 2 ? q.z : q.w;
        if constexpr (sizeof(T) == 4) {
            return __uint_as_float(u);
        } else {
            const unsigned short h = (unsigned short)(i & 1 ? u >> 16 : u & 0xffffu);
            return ldd(reinterpret_cast<const T *>(&h));
        }
    }
};
template <typename T>
struct Group<1, T> {
    T v;
    __device__ __forceinline__ void load(const T *p) { v = *p; }
    __device__ __forceinline__ float operator[](int) const { return ldd(&v); }
};

// The groups of V voxels of a volume, and the exact divisions that take a group's index to its row and
// plane (padded voxels, and so the indices, are below 2^31)
struct Groups {
    unsigned per, ny, all;       // groups per row, rows per plane, groups
    ExactDiv by_per, by_ny;
    Groups(int V, int nx, int ny_, int nz)
        : per((unsigned)(nx / V)), ny((unsigned)ny_), all(per * ny * (unsigned)nz), by_per(per), by_ny(ny)
    {
    }
};

// f(dose, target) for every resin voxel (target only when given).  Threads take groups of V voxels,
// kDeep of them in flight each.
template <int V, bool kTarget, typename DT, typename F>
__device__ __forceinline__ void each_resin(const DT *__restrict__ dose, const float *__restrict__ target,
                                           const int2 *__restrict__ span, const Groups &G, F &&f)
{
    constexpr int kDeep = kTarget ? 1 : 2;
    const unsigned per = G.per, all = G.all, nx = per * V, stride = gridDim.x * kRowThreads;
    for (unsigned i0 = blockIdx.x * kRowThreads + threadIdx.x; i0 < all; i0 += kDeep * stride) {
        Group<V, DT> d[kDeep];
        Group<V, float> t[kTarget ? kDeep : 1];
        int lo[kDeep], hi[kDeep];            // the group's resin voxels
#pragma unroll
        for (int k = 0; k < kDeep; ++k) {
            const unsigned i = i0 + k * stride;
            lo[k] = hi[k] = 0;
            if (i < all) {
                const unsigned r = G.by_per(i), z = G.by_ny(r);
                const int x = (int)(i - r * per) * V;
                const int2 sp = span[r - z * G.ny];
                lo[k] = max(sp.x - x, 0);
                hi[k] = min(sp.y - x, V);
                if (lo[k] < hi[k]) {
                    d[k].load(dose + (int64_t)r * nx + x);
                    if (kTarget) t[k].load(target + (int64_t)r * nx + x);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < kDeep; ++k) {
            if (lo[k] == 0 && hi[k] == V) {
#pragma unroll
                for (int c = 0; c < V; ++c) f(d[k][c], kTarget ? t[k][c] : 0.f);
            } else if (lo[k] < hi[k]) {
#pragma unroll
                for (int c = 0; c < V; ++c)
                    if (c >= lo[k] && c < hi[k]) f(d[k][c], kTarget ? t[k][c] : 0.f);
            }
        }
    }
}

constexpr int kMaxBlocks = 4, kHistBlocks = 4;      // per SM (2 and 3: within 5 %)

template <int V, typename DT>
__global__ void __launch_bounds__(kRowThreads, kMaxBlocks)
    dose_max_kernel(const DT *__restrict__ dose, const int2 *__restrict__ span, const Groups G, float *__restrict__ out)
{
    float m = 0.f;
    each_resin<V, false>(dose, nullptr, span, G, [&](float d, float) { m = fmaxf(m, d); });
    block_max(m, out);
}

template <int V, typename DT>
__global__ void __launch_bounds__(kRowThreads, kHistBlocks)
    ver_hist_kernel(const DT *__restrict__ dose, const float *__restrict__ target, const int2 *__restrict__ span,
                    const Groups G, VerState *__restrict__ st, long long *__restrict__ out)
{
    __shared__ unsigned sh[2 * kBins];
    hist_clear(sh);
    __syncthreads();
    const float scale = hist_scale(st->dmax);
    each_resin<V, true>(dose, target, span, G, [&](float d, float t) { hist_add(sh, d, scale, t > 0.5f); });
    __syncthreads();
    hist_flush(sh, st->hist);
    if (last_block(&st->counter)) ver_scan(st->hist, out);
}

__global__ void resin_span_kernel(int2 *__restrict__ span, int nx, int ny, double h, double r2)
{
    const int y = blockIdx.x * blockDim.x + threadIdx.x;
    if (y >= ny) return;
    // no fused multiply-adds: plain FP64 rounding
    const double cy = (y - 0.5 * (ny - 1)) * h;
    int lo = nx, hi = 0;
    for (int x = 0; x < nx; ++x) {
        const double cx = (x - 0.5 * (nx - 1)) * h;
        if (__dadd_rn(__dmul_rn(cx, cx), __dmul_rn(cy, cy)) > r2) continue;
        lo = min(lo, x);
        hi = x + 1;
    }
    span[y] = make_int2(min(lo, hi), hi);
}

template <typename DT>
cudaError_t ver_t(const vamrt_projector *p, const DT *dose, const float *target, long long *out3, cudaStream_t s)
{
    const int nx = p->g.nx, ny = p->g.ny, nz = p->g.nz;
    VerState *st = p->ver;
    cudaError_t e = cudaMemsetAsync(st, 0, sizeof(VerState), s);
    if (e != cudaSuccess) return e;
    constexpr int V = 16 / (int)sizeof(DT);
    const bool wide = nx % V == 0 && (((uintptr_t)dose | (uintptr_t)target) & 15) == 0;
    const Groups G(wide ? V : 1, nx, ny, nz);
    auto blocks = [&](int per_sm) {
        const int64_t want = ((int64_t)G.all + kRowThreads - 1) / kRowThreads, cap = (int64_t)p->num_sms * per_sm;
        return (unsigned)(want < cap ? want : cap);
    };
    const unsigned gm = blocks(kMaxBlocks), gh = blocks(kHistBlocks);
    if (wide) {
        dose_max_kernel<V><<<gm, kRowThreads, 0, s>>>(dose, p->spans, G, &st->dmax);
        ver_hist_kernel<V><<<gh, kRowThreads, 0, s>>>(dose, target, p->spans, G, st, out3);
    } else {
        dose_max_kernel<1><<<gm, kRowThreads, 0, s>>>(dose, p->spans, G, &st->dmax);
        ver_hist_kernel<1><<<gh, kRowThreads, 0, s>>>(dose, target, p->spans, G, st, out3);
    }
    count_launches(2);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_resin_spans(const vamrt_projector *p, cudaStream_t s)
{
    resin_span_kernel<<<(p->g.ny + 127) / 128, 128, 0, s>>>(p->spans, p->g.nx, p->g.ny, p->g.voxel_mm,
                                                         p->g.r_inner_mm * p->g.r_inner_mm);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_ver(const vamrt_projector *p, const void *dose, vamrt_dtype dt, const float *target,
                       long long *out3, cudaStream_t s)
{
    if (dt == VAMRT_F32) return ver_t(p, (const float *)dose, target, out3, s);
    if (dt == VAMRT_F16) return ver_t(p, (const __half *)dose, target, out3, s);
    return ver_t(p, (const __nv_bfloat16 *)dose, target, out3, s);
}

}  // namespace vamrt
