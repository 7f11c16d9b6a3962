// Weight gradient of the 3x3x3 convolution on the 5th-generation tensor cores, every input
// voxel staged once per tile and shared by all 27 taps:
//
//   dW[co][t][ci] += sum_p dY[p][co] X[p + off(t)][ci]      (zero outside the volume)
//
// What bounds it.  The kernel of conv3d_wgrad.cu stages a copy of X per tap, 27 reads of X
// through L2 (2.97 GB for 16 channels on 184 x 128 x 128), and multiplies with N = Cout, where
// a 128 x 16 operand read from shared memory (32 cycles) feeds 8 cycles of tensor work.
//
// Tile.  TZ output planes x TY (1, 2 or 4) output rows x XB columns.  Staged, in slots of 16
// channels (32 bytes, the 32-byte swizzled MN-major operand layout): X's planes with their
// halo, [TZ + 2][chunk of 16 channels][TY + 2 rows][XB], no halo along x (one 5-dimensional
// TMA box), and of dY three copies shifted by dx, [dx][16-channel block][TZ][TY][XB].  TMA's
// zero fill supplies all padding, and channels past the last chunk.
//
// GEMM mapping.  K = positions (a run of 16 slots per MMA), N = 3 Ct: the dx copies of Ct
// output channels.  M = taps x channels: row s of X after the first row that output (oz, oy)
// reaches is (dz, chunk, dy), so eight column blocks of 16 channels one row apart (LBO = one
// row) are one M = 128 operand, and nt of them hold all (dz, chunk, dy) of the block's chunks.
// With TY = 1 every row is used, with TY = 2 three of four are and with TY = 4 half, but X is
// staged 2 or 1.5 times instead of 3.  All starts are whole swizzle atoms, and no data moves between taps.
//
// Blocks own a group of chunks, a slice of output channels and a share of the tiles: every
// nsplit-th (neighbouring blocks work on neighbouring tiles, so the halo's second reads are L2
// hits), or, where `run` is set, a run of that many positions.  They add their sums into dW with FP32 atomics, every `seg` tiles and at the end.  Warp 0 issues the
// tiles' boxes into a ring of slots, warps 2-7 issue the MMAs, one elected lane each; warps 4-7
// drain TMEM between segments and all eight at the end.  Every wait is bounded as in
// conv3d_wgrad.cu.
//
// Measured (GB300, us, the kernel of conv3d_wgrad.cu -> this one): 48 -> 16 channels on 184 x 128 x
// 128 1348 -> 270 (467 TFLOP/s; 190 with tiles of 16 planes, which the rule on long sums beside the
// plan excludes), 16 -> 16 there 455 -> 95, 96 -> 32 on 92 x 64 x 64 263 -> 82, 16 -> 32 there 65 ->
// 33, 48 -> 16 on 100 x 90 x 80 754 -> 57.  What bounds it now: an MMA of 128 x 48 x 16 takes 77
// cycles, of which its operands' reads are most.
//
// Values that are not finite.  Positions outside the volume meet real voxels of X (x = -1 and x = W of
// the shifted copies of dY, rows and planes past the volume of a last tile): dY is zero there, but
// its product with an X that is not finite is not, while a dY that is not finite does not meet the
// zeros beside the volume in x.  Either leaves a sum of its row of M that is not finite, so the rows
// that have one when TMEM is drained are summed again from global memory by the definition (direct_row).
// Nothing else pays for it: 48 -> 16 channels on 184 x 128 x 128 264.0 -> 264.9 us (a warp that looks at every
// tile's faces ahead of its MMAs: 317); with one infinite voxel 5.6 ms, x all NaN 17 ms.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>

#include "internal.cuh"
#include "tcgen05.cuh"

namespace vamrt {
namespace {

using namespace tc;

constexpr int kWgThreads = 256;
constexpr int kIssuer0 = 2, kIssuers = 6;
constexpr int kMaxSlots = 4;
constexpr int kSlotBytes = 32;             // 16 BF16 channels of one voxel
constexpr int kSmem = 220 * 1024;

struct Args {
    float *dW;
    int *err;
    WgradHaloPlan p;
    int Cin, Cout, D, H, W;
    const __nv_bfloat16 *X, *dY;
};

// box at channel 0 of slot (x, y) and the outer coordinates u, v
__device__ __forceinline__ void load_box(uint32_t dst, const CUtensorMap *map, int x, int y, int u, int v, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5, %6}], [%7];" ::"r"(dst),
        "l"((uint64_t)map), "r"(0), "r"(x), "r"(y), "r"(u), "r"(v), "r"(bar)
        : "memory");
}

// The tiles of split b are first, first + step, ... below end
struct TileRange {
    int first, end, step;
};
__device__ __forceinline__ TileRange tiles_of(const WgradHaloPlan &p, int b)
{
    if (!p.run) return {b, p.ntiles, p.nsplit};
    const int64_t last = (int64_t)(b + 1) * p.run * p.ntiles / p.npos;
    return {(int)((int64_t)b * p.run * p.ntiles / p.npos), b == p.nsplit - 1 ? p.ntiles : (int)last, 1};
}

__device__ __forceinline__ bool finite(float x) { return fabsf(x) <= 3.402823466e38f; }

// By a warp, lane l for output channel co0 + l % 16: adds the sums of tap row (dz, dy), channel ci over the
// positions of `tiles`, zero padding and no other, into dW.  Its lanes' halves take alternate rows; sums
// that are all NaN end it.
__device__ __noinline__ void direct_row(const Args &a, const TileRange &tiles, int dz, int dy, int ci, int co0, int lane)
{
    const WgradHaloPlan &p = a.p;
    double total[3] = {0.0, 0.0, 0.0};
    for (int tile = tiles.first; tile < tiles.end; tile += tiles.step) {
        const int tx = tile % p.nx, r = tile / p.nx, ty = r % p.ny, tz = r / p.ny;
        const int q0 = tx * p.XB, q1 = q0 + p.XB;             // columns of X
        for (int row = lane >> 4; row < p.TZ * p.TY; row += 2) {
            const int z = tz * p.TZ + row / p.TY, y = ty * p.TY + row % p.TY, zx = z + dz - 1, yx = y + dy - 1;
            if (z >= a.D || y >= a.H) continue;
            const bool in = zx >= 0 && zx < a.D && yx >= 0 && yx < a.H;
            const __nv_bfloat16 *xr = a.X + ((int64_t)(in ? zx : z) * a.H + (in ? yx : y)) * a.W * a.Cin + ci;
            const __nv_bfloat16 *gr = a.dY + ((int64_t)z * a.H + y) * a.W * a.Cout + co0 + (lane & 15);
            auto x = [&](int q) { return in ? __bfloat162float(xr[(int64_t)q * a.Cin]) : 0.f; };
            auto g = [&](int px) { return __bfloat162float(gr[(int64_t)px * a.Cout]); };
            float sum[3] = {0.f, 0.f, 0.f};                    // of positions q + 1, q, q - 1
            if (q0 == 0) {
                sum[0] = g(1) * x(0) + g(0) * 0.f;
                sum[1] = g(0) * x(0);
            }
            if (q1 == a.W) {
                sum[1] += g(a.W - 1) * x(a.W - 1);
                sum[2] += g(a.W - 2) * x(a.W - 1) + g(a.W - 1) * 0.f;
            }
            const int qa = max(q0, 1), qb = min(q1, a.W - 1);
            float before = g(qa - 1), at = g(qa);
#pragma unroll 8
            for (int q = qa; q < qb; ++q) {
                const float after = g(q + 1), v = x(q);
                sum[0] = fmaf(after, v, sum[0]);
                sum[1] = fmaf(at, v, sum[1]);
                sum[2] = fmaf(before, v, sum[2]);
                before = at;
                at = after;
            }
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) total[dx] += sum[dx];
        }
        const int nan = isnan(total[0]) && isnan(total[1]) && isnan(total[2]);
        if (__all_sync(0xffffffffu, __shfl_xor_sync(0xffffffffu, nan, 16) | nan)) break;
    }
#pragma unroll
    for (int dx = 0; dx < 3; ++dx) {
        const double s = total[dx] + __shfl_xor_sync(0xffffffffu, total[dx], 16);
        if (lane < 16) atomicAdd(a.dW + ((int64_t)(co0 + lane) * 27 + dz * 9 + dy * 3 + dx) * a.Cin + ci, (float)s);
    }
}

// Add accumulators tile0, tile0 + step, ... of this warp's 32 TMEM lanes, the sums of `tiles`, into dW: lane
// 32 q + l is row 16 s + ci of M, s = 8 tile + 2 q + l / 16
__device__ __forceinline__ void drain(const Args &a, const TileRange &tiles, uint32_t tmem, int q, int lane, int tile0,
                                      int step, int chunk0, int co0)
{
    const WgradHaloPlan &p = a.p;
    const int N = 3 * p.Ct, RY = p.TY + 2, ncg = min(p.cg, a.Cin / 16 - chunk0);
    for (int m = tile0; m < p.nt; m += step) {
        const int s = 8 * m + 2 * q + (lane >> 4), dy = s % RY, ch = s / RY % p.cg, dz = s / RY / p.cg;
        const bool use = dy < 3 && dz < 3 && ch < ncg;
        const int ci = 16 * (chunk0 + ch) + (lane & 15);
        for (int co = 0; co < p.Ct; co += 16) {
            float sum[3][16];
            bool whole = true;
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                const int n0 = dx * p.Ct + co;
                tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(m * N + n0), sum[dx]);
                for (int part = 1; part < p.kp; ++part) {
                    float v[16];
                    tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)((part * p.nt + m) * N + n0), v);
#pragma unroll
                    for (int j = 0; j < 16; ++j) sum[dx][j] += v[j];
                }
#pragma unroll
                for (int j = 0; j < 16; ++j) whole &= finite(sum[dx][j]);
            }
            if (use && whole) {
                float *dst = a.dW + ((int64_t)(co0 + co) * 27 + dz * 9 + dy * 3) * a.Cin + ci;
#pragma unroll
                for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                    for (int j = 0; j < 16; ++j) atomicAdd(dst + ((int64_t)j * 27 + dx) * a.Cin, sum[dx][j]);
            }
            for (unsigned again = __ballot_sync(0xffffffffu, use && !whole); again; again &= again - 1) {
                const int l = __ffs(again) - 1;
                direct_row(a, tiles, __shfl_sync(0xffffffffu, dz, l), __shfl_sync(0xffffffffu, dy, l),
                           __shfl_sync(0xffffffffu, ci, l), co0 + co, lane);
            }
        }
    }
}

__global__ void __launch_bounds__(kWgThreads, 1)
    conv3d_wgrad_halo_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap ymap,
                             const __grid_constant__ Args a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // full[slots], empty[slots], then: segment's MMAs done, segment drained, all MMAs done
    __shared__ __align__(8) unsigned long long bars[2 * kMaxSlots + 3];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    __shared__ int s_fin;

    const WgradHaloPlan &p = a.p;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int chunk0 = (blockIdx.x % p.ngroups) * p.cg, co0 = (blockIdx.x / p.ngroups) * p.Ct;
    const int nb = p.Ct / 16, N = 3 * p.Ct, nacc = p.nt * p.kp, nis = min(kIssuers, nacc);
    const TileRange tiles = tiles_of(p, blockIdx.y);
    const int ybytes = p.TZ * p.TY * p.XB * kSlotBytes;              // a block of dY
    const uint32_t base = smem_u32(smem_raw);
    const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[kMaxSlots]);
    const uint32_t seg_done = smem_u32(&bars[2 * kMaxSlots]), drained = seg_done + 8, done = seg_done + 16;

    if (tid == 0) {
        for (int s = 0; s < p.slots; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, nis);
        }
        mbar_init(seg_done, nis);
        mbar_init(drained, 4);
        mbar_init(done, nis);
        mbar_init_fence();
        s_abort = 0;
        s_fin = 0;
    }
    if (warp == kIssuer0) tmem_alloc(smem_u32(&s_tmem), p.ncols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp == 0) {
        // ---- producer: lane 0 X's box, lanes 1-3 dY's for each dx ----
        int c = 0;
        for (int tile = tiles.first; tile < tiles.end; tile += tiles.step, ++c) {
            const int slot = c % p.slots;
            bool ok = true;
            if (c >= p.slots) ok = mbar_wait(empty0 + 8 * slot, (c / p.slots - 1) & 1);
            if (!__all_sync(0xffffffffu, ok) || __any_sync(0xffffffffu, s_abort)) {
                if (lane == 0) {
                    s_abort = 1;
                    atomicExch(a.err, 1);
                }
                break;
            }
            const uint32_t sb = base + slot * p.slot_bytes, bar = full0 + 8 * slot;
            if (lane == 0) mbar_arrive_expect_tx(bar, (uint32_t)(p.x_bytes + 3 * nb * ybytes));
            __syncwarp();
            const int tx = tile % p.nx, r = tile / p.nx, ty = r % p.ny, tz = r / p.ny;
            if (lane == 0)
                load_box(sb, &xmap, tx * p.XB, ty * p.TY - 1, chunk0, tz * p.TZ - 1, bar);
            else if (lane < 4)
                load_box(sb + p.x_bytes + (lane - 1) * nb * ybytes, &ymap, tx * p.XB - (lane - 2), ty * p.TY, tz * p.TZ,
                         co0 / 16, bar);
        }
    } else if (warp >= kIssuer0) {
        // ---- issuers: accumulator acc = (part, m), MMAs part, part + kp, ... of a plane ----
        const bool issuer = warp - kIssuer0 < nis;
        const int nrow = p.TY * p.XB / 16;                      // MMAs per plane
        const uint32_t idesc = instr_desc(128, N) | (1u << 15) | (1u << 16);   // A, B MN-major
        const uint64_t sw = (uint64_t)6 << 61;                  // 32-byte swizzle
        const int row16 = p.XB * kSlotBytes / 16;               // a row, in descriptor units of 16 bytes
        const int planeA = (p.TY + 2) * p.cg * row16, planeB = p.TY * row16;
        int c = 0, k = 0;                                       // tile of the segment, segment
        int slot = 0, phase = 0;
        for (int tile = tiles.first; tile < tiles.end; tile += tiles.step, ++c) {
            bool ok = true;
            if (c == p.seg) {
                if (issuer && elect_one()) mma_commit(seg_done);
                __syncwarp();
                if (warp >= 4) {
                    ok = mbar_wait(seg_done, k & 1);
                    if (__all_sync(0xffffffffu, ok)) {
                        tc_fence_after();
                        drain(a, {tile - c * tiles.step, tile, tiles.step}, tmem, warp & 3, lane, 0, 1, chunk0, co0);
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(drained);
                    }
                }
                ok = ok && mbar_wait(drained, k & 1);
                tc_fence_after();
                c = 0;
                ++k;
            }
            if (issuer) ok = ok && mbar_wait(full0 + 8 * slot, phase);
            if (!__all_sync(0xffffffffu, ok && !s_abort)) {
                s_abort = 1;
                atomicExch(a.err, 1);
                break;
            }
            tc_fence_after();
            const uint32_t sb = base + slot * p.slot_bytes;
            if (issuer && elect_one()) {
                const uint64_t A0 = smem_desc(sb, p.XB * kSlotBytes, 8 * kSlotBytes) | sw;
                const uint64_t B0 = smem_desc(sb + p.x_bytes, ybytes, 8 * kSlotBytes) | sw;
                for (int acc = warp - kIssuer0; acc < nacc; acc += nis) {
                    const int part = acc / p.nt, m = acc - part * p.nt;
                    const uint32_t d = tmem + (uint32_t)(acc * N);
                    for (int oz = 0; oz < p.TZ; ++oz) {
                        const uint64_t A = A0 + (uint64_t)(8 * m * row16 + oz * planeA), B = B0 + (uint64_t)(oz * planeB);
#pragma unroll 4
                        for (int i = part; i < nrow; i += p.kp)
                            mma_bf16(d, A + (uint64_t)(32 * i), B + (uint64_t)(32 * i), idesc,
                                     (c > 0 || oz > 0 || i != part) ? 1u : 0u);
                    }
                }
                mma_commit(empty0 + 8 * slot);
            }
            __syncwarp();
            if (++slot == p.slots) {
                slot = 0;
                phase ^= 1;
            }
        }
        if (issuer && elect_one()) mma_commit(done);
        __syncwarp();
    }
    __syncthreads();
    if (tid == 0) {
        s_fin = mbar_wait(done, 0) ? 1 : 0;     // every MMA issued has completed
        if (!s_fin) atomicExch(a.err, 1);
    }
    __syncthreads();
    tc_fence_after();
    if (s_fin && !s_abort && tiles.first < tiles.end) {
        const int segs = ((tiles.end - tiles.first - 1) / tiles.step) / p.seg;        // added already
        drain(a, {tiles.first + segs * p.seg * tiles.step, tiles.end, tiles.step}, tmem, warp & 3, lane, warp >> 2,
              kWgThreads / 128, chunk0, co0);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kIssuer0) tmem_dealloc(tmem, p.ncols);
}

}  // namespace

// Plan: the output channels in the fewest equal slices of at most 80 (N = 3 Ct <= 240), and the
// tile and chunk group that a model of the block's cycles takes for fastest, subject to two
// slots in shared memory and 512 TMEM columns.  The model, fitted to timed layers: an MMA takes
// 48 + 0.6 N cycles (77 at N = 48 and 105 at N = 96: the MN-major operands of 32-byte rows are
// read at half the shared-memory rate), TMA boxes 40 bytes a cycle, a tile 400 cycles of hand-over,
// and an addition into dW between segments 80 N cycles (4 to 8 us).
//
// The tensor cores' FP32 sums drift with their length (8e-10 to 1e-9 of the result per
// position), so a segment's sums are no longer than those of the kernel of conv3d_wgrad.cu.  It
// keeps the shapes where even one tile is longer, and those of more than 32 output channels
// that would need segments: its operands are wide rows there and its M tiles fill all of TMEM
// (64 -> 128 on 23 x 16 x 16: 19 us against 33 here with three segments, 192 -> 64 on 46 x 32 x
// 32: 76 against 68).  Sums of more than 16384 positions drift by more than 1.6e-5, which two
// ways of splitting the same volume would show as a difference between their results; they
// take the positions in that kernel's runs and order (TZ = 1, the same number of partial sums).
bool plan_wgrad_halo(int D, int H, int W, int Cin, int Cout, int taps, int sms, WgradHaloPlan *pl)
{
    WgradPlan other;
    if (taps != 27 || D < 1 || H < 1 || !plan_wgrad_tma(D, H, W, Cin, Cout, taps, sms, &other)) return false;
    const int longest = other.spb * other.KS / other.kp;         // positions per accumulator
    const int nc = Cin / 16, nb = Cout / 16;
    int nslices = 1;
    while (nb % nslices || nb / nslices > 5) ++nslices;
    const int Ct = Cout / nslices, N = 3 * Ct;
    const double mma = 48 + 0.6 * N;
    const int64_t P = (int64_t)D * H * W;
    const bool runs = longest > 16384;
    double best = 0;
    bool found = false;
    for (int ngroups = 1; ngroups <= nc; ++ngroups) {
        const int cg = (nc + ngroups - 1) / ngroups;
        if (runs && ngroups * nslices * other.nsplit > sms) continue;
        if ((nc + cg - 1) / cg != ngroups || ngroups * nslices > sms) continue;
        for (int TY = 1; TY <= 4; TY *= 2) {
            const int RY = TY + 2, nt = ((3 * cg - 1) * RY + 3 + 7) / 8;
            if (nt * N > 512) continue;
            for (int XB = 16; XB <= 128 && W % XB == 0; XB *= 2)
                for (int TZ = runs ? 1 : 2; TZ <= (runs ? 1 : 16); TZ *= 2) {
                    const int row = XB * kSlotBytes, xb = (TZ + 2) * RY * cg * row, yb = 3 * (Ct / 16) * TZ * TY * row;
                    const int slots = std::min(kMaxSlots, kSmem / (xb + yb));
                    const int64_t ntiles = (int64_t)((D + TZ - 1) / TZ) * ((H + TY - 1) / TY) * (W / XB);
                    const int nsplit = runs ? other.nsplit : (int)std::min<int64_t>(sms / (ngroups * nslices), ntiles);
                    const int64_t share = (ntiles + nsplit - 1) / nsplit;
                    // four chains of MMAs in flight, more where that spares additions into dW
                    int kp = 1;
                    while (2 * kp <= TY * XB / 16 && 2 * kp * nt * N <= 512 &&
                           (runs ? 2 * kp <= other.kp : kp * nt < 4 || share * (TZ * TY * XB / kp) > longest))
                        kp *= 2;
                    if (runs && kp != other.kp) continue;
                    const int seg = runs ? (int)ntiles : longest / (TZ * TY * XB / kp);
                    // rows past X's that unused rows of M read lie in dY's blocks
                    if (slots < 2 || seg < 1 || ntiles >= (1ll << 31) || (8 * nt + TY - 1 - 3 * RY * cg) * row > yb) continue;
                    const int64_t nseg = (share + seg - 1) / seg;
                    const double work = nt * mma * (TZ * TY * XB / 16), load = (xb + yb) / 40.0;
                    if (nseg > 1 && Cout > 32) continue;
                    const double cost = (double)share * (std::max(work, load) + 0.15 * std::min(work, load) + 400) +
                                        (double)(nseg - 1) * 80 * N;
                    if (found && cost >= best) continue;
                    found = true;
                    best = cost;
                    int ncols = 32;
                    while (ncols < nt * kp * N) ncols <<= 1;
                    *pl = WgradHaloPlan{TZ, TY, XB, cg, ngroups, Ct, nslices, nt, kp, slots, xb + yb, xb, ncols, nsplit,
                                        W / XB, (H + TY - 1) / TY, (int)ntiles,
                                        runs ? (int)ntiles : (int)((share + nseg - 1) / nseg),
                                        runs ? other.spb * other.KS : 0, (int)P};
                }
        }
    }
    return found;
}

cudaError_t launch_wgrad_halo(const void *X, const void *dY, float *dW, int D, int H, int W, int Cin, int Cout,
                              const WgradHaloPlan &pl, int *err, cudaStream_t s)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = tma_encoder();
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap maps[2];
    for (int k = 0; k < 2; ++k) {
        // [16 channels][x][y][chunk][z] of X, [16 channels][x][y][z][chunk] of dY
        const cuuint64_t C = (cuuint64_t)(k ? Cout : Cin), pl_ = C * 2 * W * H;
        const cuuint64_t d3 = (cuuint64_t)D, c3 = C / 16;
        const cuuint64_t dims[5] = {16, (cuuint64_t)W, (cuuint64_t)H, k ? d3 : c3, k ? c3 : d3};
        const cuuint64_t str[4] = {C * 2, C * 2 * W, k ? pl_ : 32, k ? 32 : pl_};
        const cuuint32_t nz = (cuuint32_t)(k ? pl.TZ : pl.TZ + 2), ncb = (cuuint32_t)(k ? pl.Ct / 16 : pl.cg);
        const cuuint32_t box[5] = {16, (cuuint32_t)pl.XB, (cuuint32_t)(k ? pl.TY : pl.TY + 2), k ? nz : ncb, k ? ncb : nz};
        const cuuint32_t one[5] = {1, 1, 1, 1, 1};
        if (enc(&maps[k], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(k ? dY : X), dims, str, box, one,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorNotSupported;
    }
    // at least 116 KB of shared memory keeps one block per SM, so TMEM is never oversubscribed
    const int smem = std::max(pl.slots * pl.slot_bytes, 116 * 1024);
    cudaError_t e = cudaFuncSetAttribute(conv3d_wgrad_halo_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const Args a{dW, err, pl, Cin, Cout, D, H, W, (const __nv_bfloat16 *)X, (const __nv_bfloat16 *)dY};
    conv3d_wgrad_halo_kernel<<<dim3(pl.ngroups * pl.nslices, pl.nsplit), kWgThreads, smem, s>>>(maps[0], maps[1], a);
    return cudaGetLastError();
}

}  // namespace vamrt
