// Dose over groups of S = 4 angles a quarter turn apart: every sample serves the four with one
// position, one cell and one set of weights (ring.cuh: groups, turns, windows).
//
//   * A block adds into a ring of rows in shared memory, [angle][row][x][z], 32-bit fixed point
//     (shared-memory integer atomics are native, 1 per bank and clock; FP32 ones are not).
//   * The weights of a run of samples in one cell are summed, with the Beer-Lambert factor,
//     before they are added: 8 atomics per run and angle instead of 8 per sample (0.53-0.6
//     runs per sample).  Angles whose pixels are all zero in a warp are passed over, rays
//     with no lit pixel in the group are not walked.
//   * Rows that the bundle has left are flushed to rotated FP32 accumulators [turn][y][x][z] with
//     16-byte vector reductions (groups that are zero are skipped) while the next rows are
//     walked; gather_turns_kernel adds the four turns up in the caller's layout.
//
// Bound by the shared-memory pipe (95 % of its active cycles with every pixel lit, 1.71 wavefronts per atomic:
// lanes whose rays are less than a voxel apart meet in a bank; issue 63 %).  Against the per-angle kernel
// (operators.cu), us, a third to a half of the pixels lit: 256^3 with 16 jittered rays, 120 angles 119479 ->
// 99765; tall build, BF16, 48 angles 65628 -> 52401; large print, 16 angles 91306 -> 73370.  Four accumulators
// are cleared and gathered whatever is lit, so a dose of a few pixels takes longer (768 x 768 x 1024 at 16 angles,
// one pixel lit, 3455 -> 5342).  Groups of two and single angles share too little of the walk to pay for the
// run sums (64^3, 90 angles, groups of two: an optimiser iteration 5 % slower; 45 angles: 0.75 -> 1.11 ms): they
// keep the per-angle kernel.
#include <algorithm>
#include <type_traits>

#include "ring.cuh"

namespace vamrt {
namespace {

constexpr int S = 4;
// 12 columns and two blocks per SM, or 8 and two with longer stages: 1 % and 5 % slower.
constexpr int kDoseTU = 8, kDoseThreads = kDoseTU * kRingTV;
constexpr int kDoseBlocks = 3;
constexpr int kDoseTab = 128;           // row table: rows being flushed to rows being entered, < 3 R + 1 <= 94
constexpr int kDoseWords = 17 * 1024;   // 68 KB, three blocks per SM

// i / d through an FP32 reciprocal, exact for 0 <= i < 2^22 (see operators.cu)
__device__ __forceinline__ int fdiv(int i, float inv_d) { return (int)(((float)i + 0.5f) * inv_d); }

__device__ __forceinline__ void red_v4(float *p, float4 v)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

// A run's weights carry 2^-100, an angle's factor 2^-49: the product of two normal numbers is
// share x 2^-149, the subnormal whose bit pattern is the share rounded to an integer (share
// < 2^23).  Warps with a negative pixel take x + 1.5 x 2^23 instead, whose bit pattern is
// round(x) + 0x4B400000 (|x| < 2^22).  Both round once, to nearest even.
constexpr float kRunScale = 0x1p-100f, kNonNegScale = 0x1p-49f, kSignedScale = 0x1p100f;

// f(constant m) for the run-time mask m in 1..M: a walk compiled for the angles that a warp
// feeds spends nothing on the others, not even a branch per run.
template <unsigned M, typename F>
__device__ __forceinline__ void by_mask(unsigned m, F &&f)
{
    if constexpr (M > 0) {
        if (m == M)
            f(std::integral_constant<unsigned, M>());
        else
            by_mask<M - 1>(m, f);
    }
}

template <typename PT>
__global__ void __launch_bounds__(kDoseThreads, kDoseBlocks)
    ring_dose_kernel(const RingParams G, const PT *__restrict__ proj, float *__restrict__ accs)
{
    extern __shared__ __align__(16) int iring[];
    __shared__ int slots[3][kSlots];
    __shared__ int wmax_s[3][S];            // largest |weight| of each angle, rotating like slots
    __shared__ int4 rows_s[kDoseTab];        // per row: offsets of it and the next, its slot, its place in the accumulator
    __shared__ Window sW;
    __shared__ float inv_s[S];
    constexpr int kCap = kDoseWords / S;
    constexpr int kAlign = 4;

    const OpParams &P = G.op;
    const int lane = threadIdx.x, tid = threadIdx.y * kRingTV + lane;
    const int u = blockIdx.x * kDoseTU + threadIdx.y, v = blockIdx.z * kRingTV + lane;
    const bool valid = u < P.nu && v < P.nv;
    if (tid < 3 * kSlots) slot_reset(slots[tid / kSlots], tid % kSlots);
    if (tid < 3 * S) wmax_s[tid / S][tid % S] = 0;

    float g[S];
    bool lit = false, odd = false;       // odd: not finite, which fixed point cannot hold
#pragma unroll
    for (int i = 0; i < S; ++i) {
        g[i] = valid ? to_f(proj[((int64_t)G.members[(int64_t)blockIdx.y * S + i] * P.nv + v) * P.nu + u]) : 0.f;
        lit |= g[i] != 0.f;
        odd |= !(fabsf(g[i]) <= 3.402823466e38f);
    }
    if (!__syncthreads_or(lit)) return;
    // the ring starts empty; every flush leaves its rows empty again
    for (int i = tid; i < kDoseWords / 4; i += kDoseThreads) reinterpret_cast<int4 *>(iring)[i] = make_int4(0, 0, 0, 0);

    for (int a = 0; a < P.M; ++a) {
        RRay R{};
        int turn;
        {
            const bool active = lit && ring_ray(G, ((int64_t)a * P.nv + v) * P.nu + u, G.cs[blockIdx.y], R, false);
            if (!active) R.j = R.jhi = 0;
            // values >= 0 order like their bits
#pragma unroll
            for (int i = 0; i < S; ++i) {
                const int wbits = __reduce_max_sync(kFull, active ? __float_as_int(fabsf(g[i] * R.w)) : 0);
                if (lane == 0 && wbits) atomicMax(&wmax_s[a % 3][i], wbits);
            }
            Window W;
            const bool any = bundle(G, slots[a % 3], active, odd, R, kAlign, 1, kCap, false, turn, W);
            if (tid < kSlots) slot_reset(slots[(a + 2) % 3], tid);      // last read one aperture sample ago
            if (tid < S) wmax_s[(a + 2) % 3][tid] = 0;
            if (!any) continue;
            if (tid == 0) sW = W;
        }
        // component c of the ring: angle (c - shift) mod 4, accumulator turn c
        const int sh = shift_of<S>(turn), ex = P.nx + 2;         // a square grid: the same for every turn
        float gc[S];
#pragma unroll
        for (int c = 0; c < S; ++c) {
            gc[c] = g[c];
#pragma unroll
            for (int k = 1; k < S; ++k)
                if (sh == k) gc[c] = g[(c + S - k) % S];
            gc[c] = R.j < R.jhi ? gc[c] * R.w : 0.f;
        }
        const float ratio = exp2f(R.att);
        __syncthreads();
        if (!sW.ok) {
            // bundles too wide for the ring, values that are not finite: FP32 reductions straight
            // into the accumulators
            while (R.j < R.jhi)
                walk(R, ratio, 1.0f, 16, INT_MAX, G.pzp, [&](int e, int y, const Run &r) {
                    const int64_t o[4] = {0, G.pzp, (int64_t)ex * G.pzp, (int64_t)(ex + 1) * G.pzp};
#pragma unroll
                    for (int c = 0; c < S; ++c) {
                        if (gc[c] == 0.f) continue;
                        float *p = accs + (int64_t)c * G.vol_elems + ((int64_t)y * ex * G.pzp + e);
#pragma unroll
                        for (int k = 0; k < 8; ++k) atomicAdd(p + o[2 * (k >> 2) + (k & 1)] + ((k >> 1) & 1), gc[c] * r.w[k]);
                    }
                });
            continue;
        }
        // fixed point: a voxel takes at most cell_bound samples of each of the block's rays, a run
        // a bounded part of them; sums stay below 2^31, shares below 2^22
        unsigned live = 0;       // angles some lane of the warp feeds
        bool sign = false;       // some with a negative value
#pragma unroll
        for (int c = 0; c < S; ++c) {
            const float wmax = __int_as_float(wmax_s[a % 3][(c + S - sh) & (S - 1)]);
            const float scale = fminf(G.share_scale / wmax, 1e30f);
            if (tid == c) inv_s[c] = 1.0f / scale;
            live |= (__any_sync(kFull, gc[c] != 0.f) ? 1u : 0u) << c;
            sign |= __any_sync(kFull, gc[c] < 0.f);
            gc[c] *= scale;
        }
        // a warp without a negative value may hold -0.0 (a dark pixel, or one below zero that vanishes
        // when it is weighted), as a bit pattern the lowest integer
#pragma unroll
        for (int c = 0; c < S; ++c) gc[c] = sign ? gc[c] * kSignedScale : fabsf(gc[c]) * kNonNegScale;
        const int zpitch = sW.EZ, stages = sW.stages, slab = sW.EX * zpitch, y0 = sW.y0, R_ = sW.R, ring_rows = 2 * R_ + 1;
        auto table = [&](int ya, int yb) {      // warp 0, one lane per row
            for (int y = ya + lane; y <= yb; y += 32) {
                const int slot = (y - y0) % ring_rows, next = slot + 1 == ring_rows ? 0 : slot + 1;
                int xo, zo;
                corner(sW, y, kAlign, xo, zo);
                rows_s[y & (kDoseTab - 1)] = make_int4(row_offset(sW, y, kAlign, slot), row_offset(sW, y + 1, kAlign, next),
                                                      slot * slab, (y * ex + xo) * G.pzp + zo);
            }
        };
        if (threadIdx.y == 0) table(y0, min(y0 + 2 * R_, sW.y1));
        __syncthreads();
        // a lane's place in the columns that its warp flushes together
        const int quads = zpitch >> 2, per = 32 / quads, col = lane / quads, quad = lane - col * quads;
        for (int t = 0; t < stages; ++t) {
            const int lim = y0 + (t + 1) * R_;
            auto add = [&](auto mask_) {
                constexpr unsigned kMask = decltype(mask_)::value;
                walk(R, ratio, kRunScale, INT_MAX, lim, zpitch, [&](int e, int y, const Run &r) {
                    const int4 o = rows_s[y & (kDoseTab - 1)];
                    int *p0 = iring + (o.x + e), *p1 = iring + (o.y + e);
                    int *p[4] = {p0, p0 + zpitch, p1, p1 + zpitch};      // 2 y + x
#pragma unroll
                    for (int c = 0; c < S; ++c)
                        if (kMask >> c & 1) {
#pragma unroll
                            for (int k = 0; k < 8; ++k)                  // 4 y + 2 z + x
                                atomicAdd(p[2 * (k >> 2) + (k & 1)] + c * kCap + (k >> 1 & 1),
                                          __float_as_int(r.w[k] * gc[c]));
                        }
                });
            };
            if (!sign)
                by_mask<(1u << S) - 1>(live, add);
            else
                walk(R, ratio, kRunScale, INT_MAX, lim, zpitch, [&](int e, int y, const Run &r) {
                    const int4 o = rows_s[y & (kDoseTab - 1)];
                    int *p0 = iring + (o.x + e), *p1 = iring + (o.y + e);
                    int *p[4] = {p0, p0 + zpitch, p1, p1 + zpitch};
#pragma unroll
                    for (int c = 0; c < S; ++c) {
                        if (gc[c] == 0.f) continue;
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            atomicAdd(p[2 * (k >> 2) + (k & 1)] + c * kCap + (k >> 1 & 1),
                                      __float_as_int(fmaf(r.w[k], gc[c], 12582912.0f)) - 0x4B400000);
                    }
                });
            __syncthreads();
            // rows below lim are complete (the last stage: all): flush them while the next stage's
            // rows, which lie in other slots, are walked
            if (threadIdx.y == 0) table(y0 + (t + 2) * R_ + 1, min(y0 + (t + 3) * R_, sW.y1));
            const int ya = y0 + t * R_, yb = t + 1 == stages ? sW.y1 : lim - 1, EX = sW.EX;
            const float inv_ex = 1.0f / (float)EX;
            if (col < per)
                for (int i = threadIdx.y * per + col; i < (yb - ya + 1) * EX; i += kDoseTU * per) {
                    const int row = fdiv(i, inv_ex), x = i - row * EX;
                    const int4 o = rows_s[(ya + row) & (kDoseTab - 1)];
                    int *b = iring + (o.z + x * zpitch + 4 * quad);
                    float *q = accs + (o.w + x * G.pzp + 4 * quad);
#pragma unroll
                    for (int c = 0; c < S; ++c) {
                        int4 *b4 = reinterpret_cast<int4 *>(b + c * kCap);
                        const int4 n = *b4;
                        if ((n.x | n.y | n.z | n.w) != 0) {
                            const float inv = inv_s[c];
                            red_v4(q + (int64_t)c * G.vol_elems,
                                   make_float4((float)n.x * inv, (float)n.y * inv, (float)n.z * inv, (float)n.w * inv));
                            *b4 = make_int4(0, 0, 0, 0);
                        }
                    }
                }
        }
    }
}

// out[z][y][x] (+)= sum over the four turns of the rotated accumulators acc[r][y][x][z] at the
// turned voxel, in the order r = 0..3.  `out` has the given row and plane pitch and origin.  A
// block takes 32 x and 32 z of one y: every read and write is a run of 128 bytes.
constexpr int kGatherX = 32, kGatherZ = 32;
template <typename DT>
__global__ void __launch_bounds__(256) gather_turns_kernel(const float *__restrict__ acc, DT *__restrict__ out, int nx,
                                                           int ny, int nz, int pzp, int64_t row, int64_t plane,
                                                           int64_t origin, int accumulate)
{
    __shared__ float tile[kGatherZ][kGatherX + 1];
    const int x0 = blockIdx.x * kGatherX, sy = blockIdx.y, z0 = blockIdx.z * kGatherZ;
    const int64_t vol = (int64_t)(nx + 2) * (ny + 2) * pzp;
    const int a = threadIdx.x & 31, b = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < kGatherX / 8; ++k) {
        const int sx = x0 + b + 8 * k, sz = z0 + a;
        float v = 0.f;
        if (sx < nx && sz < nz) {
            // the padded voxels of the turns that turn to (sx, sy)
            const float *p = acc + (sz + 1);
            v = p[((int64_t)(sy + 1) * (nx + 2) + (sx + 1)) * pzp];
            v += p[vol + ((int64_t)(nx - sx) * (ny + 2) + (sy + 1)) * pzp];
            v += p[2 * vol + ((int64_t)(ny - sy) * (nx + 2) + (nx - sx)) * pzp];
            v += p[3 * vol + ((int64_t)(sx + 1) * (ny + 2) + (ny - sy)) * pzp];
        }
        tile[a][b + 8 * k] = v;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kGatherZ / 8; ++k) {
        const int sx = x0 + a, sz = z0 + b + 8 * k;
        if (sx >= nx || sz >= nz) continue;
        DT *q = out + origin + sz * plane + sy * row + sx;
        float v = tile[b + 8 * k][a];
        if (accumulate) v += to_f(*q);
        st_val(q, v);
    }
}

constexpr size_t kDoseSmem = sizeof(float) * kDoseWords;

}  // namespace

cudaError_t launch_ring_dose(const vamrt_projector *p, const void *proj, vamrt_dtype dt, cudaStream_t s)
{
    const RingParams &G = p->ring;
    cudaError_t e = cudaMemsetAsync(p->ring_vols, 0, sizeof(float) * 4 * (size_t)G.vol_elems, s);
    if (e != cudaSuccess) return e;
    return by_storage(dt, const_cast<void *>(proj), [&](auto *pr) {
        using PT = std::remove_pointer_t<decltype(pr)>;
        cudaError_t f = cudaFuncSetAttribute(ring_dose_kernel<PT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kDoseSmem);
        if (f != cudaSuccess) return f;
        ring_dose_kernel<PT><<<ring_grid(G, kDoseTU), dim3(kRingTV, kDoseTU), kDoseSmem, s>>>(G, pr, p->ring_vols);
        count_launches(1);
        return cudaGetLastError();
    });
}

// out[z][y][x] at the given pitches (elements) and origin
cudaError_t launch_ring_gather(const vamrt_projector *p, void *out, vamrt_dtype dt, int64_t row, int64_t plane,
                               int64_t origin, int accumulate, cudaStream_t s)
{
    const RingParams &G = p->ring;
    const int nx = G.op.nx, ny = G.op.ny, nz = G.op.nz;
    const dim3 grid((unsigned)((nx + kGatherX - 1) / kGatherX), (unsigned)ny, (unsigned)((nz + kGatherZ - 1) / kGatherZ));
    return by_storage(dt, out, [&](auto *d) {
        gather_turns_kernel<<<grid, 256, 0, s>>>(p->ring_vols, d, nx, ny, nz, G.pzp, row, plane, origin, accumulate);
        count_launches(1);
        return cudaGetLastError();
    });
}

}  // namespace vamrt
