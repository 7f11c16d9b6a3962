// 3x3x3 convolution on the 5th-generation tensor cores, marching along z: every plane of the
// input is staged once per block column and feeds three output planes at a time.
//
//   Y[p][co] = act( bias[co] + sum_{t, ci} X[p + off(t)][ci] * Wt[co][t][ci] )
//
// What bounds it.  The kernel of conv3d_halo.cu stages regions of 5 rows with their halo (4.7
// reads of X through L2 at W = 128), reloads the weights with every chunk and reads each A operand
// (32 cycles at 128 bytes a cycle) for N = 48 columns (24 cycles of tensor work).
//
// A block takes TY rows x all W columns (T <= 2 tiles of 128 slots) of one 16-channel slice of Y,
// keeps that slice's weights in shared memory, and walks z.  A stage is cps (1, 2 or 4) 16-channel
// chunks of one plane of X with one halo row on either side: (TY + 2) x W slots of 32, 64 or 128
// bytes in the swizzled K-major layout of that width, one TMA box, zero fill outside the volume
// and past the last channel.  A chunk's A operand for dy is the slot run shifted by whole rows.  N stacks (output plane, dx, co): the plane z' adds to
// the outputs z' - 1, z' and z' + 1, whose accumulators (48 columns each: three dx x 16) stand
// side by side in a ring of kRing planes per tile, so one MMA has N = 144 (two where the ring
// wraps; the first MMA into a new plane overwrites and goes apart).  The epilogue adds the dx
// shifts as conv3d_halo.cu does, Y[m] = D[m - 1][-1] + D[m][0] + D[m + 1][+1], neighbours beyond
// a row's ends left out.  Where W does not divide 128, tiles run through the rows 120 slots
// apart with a margin slot at either end, starting 8 slots ahead of the first row.
//
// Measured (GB300, us, conv3d_halo.cu -> this kernel with 32-byte slots -> with the widest slots): 48 ->
// 16 channels on 184 x 128 x 128 283 -> 160 -> 140 (893 TFLOP/s), 16 -> 48 there 342 -> 244 -> 240, 16 ->
// 16 123 -> 91 -> 89, 96 -> 32 on 92 x 64 x 64 199 -> 81 -> 69, 192 -> 64 on 46 x 32 x 32 121 -> 64 -> 56, 64 ->
// 64 there 50 -> 27 -> 22.  Wide operand rows are read faster and take fewer stages.  What bounds it
// now (48 -> 16): the MMAs (145 us without the epilogue's arithmetic and 160 with it, at 32-byte
// slots); TMA and the stores do not show.
//
// Roles: kMarchSets sets of 4 epilogue warps take (plane, tile) units in turn, one warp issues the
// TMA boxes, and one warp per tile issues its MMAs (one elected lane; the order of the MMAs into
// an accumulator is that of one issuer).  Every wait is bounded as in conv3d_halo.cu.
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>

#include "conv_epilogue.cuh"
#include "internal.cuh"
#include "tcgen05.cuh"

namespace vamrt {
namespace {

using namespace tc;

constexpr int kMarchSets = 4, kMarchLoad = 4 * kMarchSets, kMarchMma = kMarchLoad + 1, kMaxT = 2;
constexpr int kMarchThreads = 32 * (kMarchMma + kMaxT);
constexpr int kRing = 5;                    // output planes per tile in TMEM
constexpr int kMaxStages = 8;
constexpr int kLead = 8;                    // slots ahead of a stage's box
constexpr int kWBytes = 27 * 16 * 32;       // weights of one chunk: [dy][144 rows][16]
constexpr int kMarchSmem = 220 * 1024;

struct MarchArgs {
    const __nv_bfloat16 *Wt;
    const float *bias;
    void *Y;
    int *err;
    ConvMarchPlan p;
    int D, H, W, Cin, Cout, relu;
};

// Pieces of a block's run of (column, z): outputs z0 .. z1 - 1 of one column
struct Piece {
    int y0, z0, z1;
};
__device__ __forceinline__ Piece piece_at(const MarchArgs &a, int l, int l1)
{
    const int col = l / a.D, z0 = l - col * a.D;
    return {col * a.p.TY, z0, min(a.D, z0 + l1 - l)};
}

__device__ __forceinline__ void march_fail(volatile int *abort_flag, int *err)
{
    *abort_flag = 1;
    atomicExch(err, 1);
}

template <typename OT>
__device__ void march_epilogue(const MarchArgs &a, uint32_t tmem, int l0, int l1, int co0, float *s_xch, uint32_t accf,
                               uint32_t acce, volatile int *abort_flag)
{
    const int set = threadIdx.x >> 7, tid = threadIdx.x & 127, warp = tid >> 5, lane = tid & 31;
    const int T = a.p.T, mg = a.p.mg, adv = a.p.adv;
    float *xch = s_xch + set * 256;
    int g = 0, step = 0;                   // output planes so far; this set's units
    for (int l = l0; l < l1;) {
        const Piece pc = piece_at(a, l, l1);
        for (int z = pc.z0; z < pc.z1; ++z, ++g) {
            const int slot = g % kRing;
            for (int t = 0; t < T; ++t) {
                if ((g * T + t) % kMarchSets != set) continue;
                const bool ok = mbar_wait(accf + 8 * slot, (g / kRing) & 1) && !*abort_flag;
                if (!epi_all(ok, set)) {
                    if (tid == 0) march_fail(abort_flag, a.err);
                    return;
                }
                tc_fence_after();
                // slot of the region's rows (mg: one margin slot, the tile starts 8 slots early)
                const int q = adv * t + tid - 8 * mg, oy = q / a.W, x = q - oy * a.W, y = pc.y0 + oy;
                const bool valid = tid >= mg && tid < mg + adv && q >= 0 && oy < a.p.TY && y < a.H;
                const uint32_t col = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)((t * kRing + slot) * 48);
                uint32_t dm[16], v[16], dp[16];
                tmem_ld16_issue(col, dm);
                tmem_ld16_issue(col + 16, v);
                tmem_ld16_issue(col + 32, dp);
                tmem_ld_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acce + 8 * slot);
                // rows 32 w - 1 and 32 w + 32 are the neighbouring warps': each publishes its edges
                uint4 *xm = (uint4 *)(xch + (step & 1) * 128), *xp = xm + 16;   // [warp][4] x 16 B
                ++step;
                if (lane == 31)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        xm[warp * 4 + i] = make_uint4(dm[4 * i], dm[4 * i + 1], dm[4 * i + 2], dm[4 * i + 3]);
                if (lane == 0)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        xp[warp * 4 + i] = make_uint4(dp[4 * i], dp[4 * i + 1], dp[4 * i + 2], dp[4 * i + 3]);
                epi_sync(set);
                uint32_t el[16], er[16];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 l4 = warp > 0 ? xm[(warp - 1) * 4 + i] : make_uint4(0, 0, 0, 0);
                    const uint4 r4 = warp < 3 ? xp[(warp + 1) * 4 + i] : make_uint4(0, 0, 0, 0);
                    el[4 * i] = l4.x; el[4 * i + 1] = l4.y; el[4 * i + 2] = l4.z; el[4 * i + 3] = l4.w;
                    er[4 * i] = r4.x; er[4 * i + 1] = r4.y; er[4 * i + 2] = r4.z; er[4 * i + 3] = r4.w;
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const uint32_t up = __shfl_up_sync(0xffffffffu, dm[i], 1);
                    const uint32_t dn = __shfl_down_sync(0xffffffffu, dp[i], 1);
                    const float left = x == 0 ? 0.f : __uint_as_float(lane == 0 ? el[i] : up);
                    const float right = x == a.W - 1 ? 0.f : __uint_as_float(lane == 31 ? er[i] : dn);
                    v[i] = __float_as_uint(left + __uint_as_float(v[i]) + right);
                }
                if (valid)
                    store16<OT>((OT *)a.Y + ((((int64_t)z * a.H + y) * a.W + x) * a.Cout + co0), v,
                                a.bias ? a.bias + co0 : nullptr, a.relu);
            }
        }
        l += pc.z1 - pc.z0;
    }
}

template <typename OT, int CPS>
__global__ void __launch_bounds__(kMarchThreads, 1)
    conv3d_march_kernel(const __grid_constant__ CUtensorMap xmap, const MarchArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    // full[stages], empty[stages], accumulators full[kRing], empty[kRing]
    __shared__ __align__(8) unsigned long long bars[2 * kMaxStages + 2 * kRing];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(16) float s_xch[256 * kMarchSets];
    __shared__ volatile int s_abort;

    const ConvMarchPlan &p = a.p;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int slice = blockIdx.x % p.nslice, co0 = 16 * slice, nc = a.Cin >> 4;
    constexpr int sb = 32 * CPS;           // bytes of a slot
    const int64_t tot = (int64_t)p.ry * a.D, blk = blockIdx.x / p.nslice;
    const int l0 = (int)(blk * tot / p.nblk), l1 = (int)((blk + 1) * tot / p.nblk);
    const uint32_t sbase = smem_u32(smem), wbase = sbase, xbase = sbase + nc * kWBytes;
    const uint32_t full = smem_u32(&bars[0]), empty = full + 8 * kMaxStages;
    const uint32_t accf = empty + 8 * kMaxStages, acce = accf + 8 * kRing;

    if (tid == 0) {
        for (int s = 0; s < p.ns; ++s) {
            mbar_init(full + 8 * s, 1);
            mbar_init(empty + 8 * s, p.T);
        }
        for (int s = 0; s < kRing; ++s) {
            mbar_init(accf + 8 * s, p.T);
            mbar_init(acce + 8 * s, 4 * p.T);
        }
        mbar_init_fence();
        s_abort = 0;
    }
    if (warp == kMarchMma) tmem_alloc(smem_u32(&s_tmem), (uint32_t)p.ncols);
    // the slice's weights: per chunk and dy, rows n = (output plane z' + b - 1: dz = 1 - b, dx, co)
    for (int i = tid; i < nc * 27 * 32; i += kMarchThreads) {
        const int h = i & 1, n = (i >> 1) % 144, cd = (i >> 1) / 144, dy = cd % 3, c = cd / 3;
        const int b = n / 48, dx = n / 16 % 3, co = n & 15, tap = (2 - b) * 9 + dy * 3 + dx;
        const uint4 w = *(const uint4 *)(a.Wt + ((int64_t)(co0 + co) * 27 + tap) * a.Cin + c * 16 + h * 8);
        *(uint4 *)(smem + c * kWBytes + dy * 144 * 32 + (n >> 3) * 256 + h * 128 + (n & 7) * 16) = w;
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp < kMarchLoad) {
        march_epilogue<OT>(a, tmem, l0, l1, co0, s_xch, accf, acce, &s_abort);
    } else if (warp == kMarchLoad) {
        int i = 0, s = 0, phase = 1;
        bool ok = true;
        for (int l = l0; l < l1 && ok;) {
            const Piece pc = piece_at(a, l, l1);
            for (int z = pc.z0 - 1; z <= pc.z1 && ok; ++z)
                for (int c = 0; c < nc; c += CPS, ++i) {
                    if (i >= p.ns) ok = mbar_wait(empty + 8 * s, phase);
                    ok = __all_sync(0xffffffffu, ok && !s_abort);
                    if (!ok) break;
                    if (lane == 0) {
                        mbar_arrive_expect_tx(full + 8 * s, (uint32_t)p.box_bytes);
                        tma_load_4d(xbase + s * p.stage_bytes + kLead * sb, &xmap, c * 16, 0, pc.y0 - 1, z, full + 8 * s);
                    }
                    __syncwarp();
                    if (++s == p.ns) {
                        s = 0;
                        phase ^= 1;
                    }
                }
            l += pc.z1 - pc.z0;
        }
        if (!ok && lane == 0) march_fail(&s_abort, a.err);
    } else if (warp - kMarchMma < p.T) {
        const int t = warp - kMarchMma;
        const uint32_t dcol = tmem + (uint32_t)(t * kRing * 48);
        const uint64_t sw = (uint64_t)(CPS == 4 ? 2 : CPS == 2 ? 4 : 6) << 61;
        const int row16 = a.W * sb / 16;          // a row, in descriptor units of 16 bytes
        int s = 0, phase = 0, g = 0;
        bool ok = true;
        for (int l = l0; l < l1 && ok;) {
            const Piece pc = piece_at(a, l, l1);
            for (int z = pc.z0 - 1; z <= pc.z1 && ok; ++z) {
                // outputs lo .. hi take this plane; z + 1 for the first time.  b0, n: first weight
                // block and number of outputs; s0: ring slot of lo; n1: outputs before the ring wraps
                const int lo = max(z - 1, pc.z0), hi = min(z + 1, pc.z1 - 1), n = hi - lo + 1, b0 = lo - (z - 1);
                const bool fresh = z + 1 < pc.z1;
                const int s0 = (g + lo - pc.z0) % kRing, n1 = min(n, kRing - s0);
                const bool wrap = n > n1;
                const uint32_t id1 = instr_desc(128, 48 * n1), id2 = instr_desc(128, 48 * (n - n1)), d1 = dcol + s0 * 48;
                if (fresh) {
                    const int u = g + z + 1 - pc.z0;
                    if (u >= kRing) ok = mbar_wait(acce + 8 * (u % kRing), (u / kRing - 1) & 1);
                }
                for (int c = 0; c < nc; c += CPS) {
                    ok = ok && mbar_wait(full + 8 * s, phase);
                    ok = __all_sync(0xffffffffu, ok && !s_abort);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint64_t A0 = smem_desc(xbase + s * p.stage_bytes +
                                                          (kLead + p.adv * t - 8 * p.mg) * sb, 16, 8 * sb) | sw;
                        const uint64_t B0 = smem_desc(wbase + c * kWBytes, 128, 256) + (uint64_t)(b0 * 96);
#pragma unroll
                        for (int k = 0; k < CPS; ++k) {
                            if (k && c + k >= nc) break;
                            const uint64_t A = A0 + (uint64_t)(2 * k), B = B0 + (uint64_t)(k * (kWBytes / 16));
#pragma unroll
                            for (int dy = 0; dy < 3; ++dy) {
                                const uint64_t Ad = A + (uint64_t)(dy * row16), Bd = B + (uint64_t)(dy * 144 * 2);
                                if (k == 0 && dy == 0 && fresh && c == 0) {
                                    // first MMA of a fresh plane overwrites: it goes apart from the others
                                    const int na = n - 1, n1a = min(n1, na);
                                    if (n1a > 0) mma_bf16(d1, Ad, Bd, instr_desc(128, 48 * n1a), 1u);
                                    if (na > n1a)
                                        mma_bf16(dcol, Ad, Bd + (uint64_t)(n1a * 96), instr_desc(128, 48 * (na - n1a)), 1u);
                                    mma_bf16(dcol + (s0 + na) % kRing * 48, Ad, Bd + (uint64_t)(na * 96),
                                             instr_desc(128, 48), 0u);
                                } else {
                                    mma_bf16(d1, Ad, Bd, id1, 1u);
                                    if (wrap) mma_bf16(dcol, Ad, Bd + (uint64_t)(n1 * 96), id2, 1u);
                                }
                            }
                        }
                        mma_commit(empty + 8 * s);
                    }
                    __syncwarp();
                    if (++s == p.ns) {
                        s = 0;
                        phase ^= 1;
                    }
                }
                if (ok && z - 1 >= pc.z0 && elect_one()) mma_commit(accf + 8 * ((g + z - 1 - pc.z0) % kRing));
                __syncwarp();
            }
            g += pc.z1 - pc.z0;
            l += pc.z1 - pc.z0;
        }
        if (!ok && lane == 0) march_fail(&s_abort, a.err);
        // after a timeout the MMAs in flight are left to finish (bounded by the wait below)
        if (!ok && elect_one()) mma_commit(accf);
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (s_abort && tid == 0) {
        const unsigned long long t0 = globaltimer();
        while (globaltimer() - t0 < 1000000ull) {}     // 1 ms: far more than a stage's MMAs take
    }
    __syncthreads();
    if (warp == kMarchMma) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, (uint32_t)p.ncols);
    }
}

}  // namespace

// Plan: two tiles (one where it holds all rows), all SMs as blocks of 16-channel slices.
bool plan_conv3d_march(int D, int H, int W, int Cin, int Cout, int taps, int sms, ConvMarchPlan *pl)
{
    if (taps != 27 || D < 1 || H < 1 || W < 8 || W % 8 || W > 240 || Cin < 16 || Cin % 16 || Cout < 16 || Cout % 16)
        return false;
    ConvMarchPlan p{};
    p.mg = 128 % W ? 1 : 0;
    p.adv = p.mg ? 120 : 128;
    const int one = p.mg ? 113 : 128, two = p.mg ? 233 : 256;     // slots that one and two tiles write
    p.T = (int64_t)H * W <= one ? 1 : 2;
    p.TY = std::min(two / W, H);
    if (p.TY < 1) return false;
    p.ncols = p.T * kRing * 48 <= 256 ? 256 : 512;
    // the widest slots that leave two stages of several chunks, or three of one
    for (p.cps = Cin > 32 ? 4 : Cin / 16; p.cps >= 1; p.cps /= 2) {
        const int sb = 32 * p.cps;
        p.box_bytes = (p.TY + 2) * W * sb;
        // slots read: two rows below the first tile's start to the end of the last tile
        const int reach = kLead + 2 * W + p.adv * (p.T - 1) - 8 * p.mg + 128;
        p.stage_bytes = (std::max(kLead * sb + p.box_bytes, reach * sb) + 1023) / 1024 * 1024;
        p.ns = std::min(kMaxStages, (kMarchSmem - Cin / 16 * kWBytes) / p.stage_bytes);
        if (p.ns >= (p.cps > 1 ? 2 : 3)) break;
    }
    if (!p.cps) return false;
    p.nslice = Cout / 16;
    p.ry = (H + p.TY - 1) / p.TY;
    if (p.nslice > sms || (int64_t)p.ry * D >= (1ll << 31)) return false;
    p.nblk = (int)std::min<int64_t>(sms / p.nslice, (int64_t)p.ry * D);
    *pl = p;
    return true;
}

cudaError_t launch_conv3d_march(const void *X, const void *Wt, const float *bias, void *Y, int out_f32, int D, int H,
                                int W, int Cin, int Cout, int relu, const ConvMarchPlan &pl, int *err, cudaStream_t s)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = tma_encoder();
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap xmap;
    const cuuint64_t dims[4] = {(cuuint64_t)Cin, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)D};
    const cuuint64_t strides[3] = {(cuuint64_t)Cin * 2, (cuuint64_t)W * Cin * 2, (cuuint64_t)H * W * Cin * 2};
    const cuuint32_t box[4] = {(cuuint32_t)(16 * pl.cps), (cuuint32_t)W, (cuuint32_t)(pl.TY + 2), 1};
    const cuuint32_t one[4] = {1, 1, 1, 1};
    if (enc(&xmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(X), dims, strides, box, one,
            CU_TENSOR_MAP_INTERLEAVE_NONE,
            pl.cps == 4 ? CU_TENSOR_MAP_SWIZZLE_128B : pl.cps == 2 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorNotSupported;
    const MarchArgs a{(const __nv_bfloat16 *)Wt, bias, Y, err, pl, D, H, W, Cin, Cout, relu};
    // at least 116 KB of shared memory keeps one block per SM, so TMEM is never oversubscribed
    const int smem = std::max(Cin / 16 * kWBytes + pl.ns * pl.stage_bytes, 116 * 1024);
    auto k = conv3d_march_kernel<float, 1>;
    if (out_f32)
        k = pl.cps == 4 ? conv3d_march_kernel<float, 4> : pl.cps == 2 ? conv3d_march_kernel<float, 2> : k;
    else
        k = pl.cps == 4   ? conv3d_march_kernel<__nv_bfloat16, 4>
            : pl.cps == 2 ? conv3d_march_kernel<__nv_bfloat16, 2>
                          : conv3d_march_kernel<__nv_bfloat16, 1>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k<<<(unsigned)(pl.nslice * pl.nblk), kMarchThreads, smem, s>>>(xmap, a);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace vamrt
