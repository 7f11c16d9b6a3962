// Projection over groups of angles: every sample serves the group's S angles with one position,
// one cell and one set of weights (ring.cuh: groups, turns, windows).
//
//   * spread_kernel writes the rotated copies of the volume, z innermost, the S components of a
//     voxel side by side, and which 8 x 8 x 8 bricks hold anything.
//   * A block takes the rows of its bundle in stages of R.  Stages whose window touches only
//     empty bricks add exactly nothing: no row of them is fetched and no sample walked.  (The
//     optimiser's models are zero outside the part: of the samples of the workloads' targets
//     between 12 % (64^3) and 92 % lie in empty windows, 73 % on the large print.)
//   * The rows of the next stage to walk are fetched by one TMA tile load each (zero fill
//     outside the grid) while the current stage is walked; two buffers of R + 1 rows.
//   * Two samples per voxel: about every second sample lies in the cell of the one before.  The
//     walk sums the trilinear weights, with the Beer-Lambert factor, of a run of samples in
//     one cell and reads its 8 corners once per run, one 16-byte read (S = 4) per corner
//     for the four angles.  z innermost makes the bank of a voxel its z modulo 8: lanes one
//     plane apart read distinct banks whatever their x and y.
#include <cuda.h>
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "ring.cuh"
#include "tcgen05.cuh"

namespace vamrt {
namespace {

// A block's pixel columns.  Measured (large print's 16-angle crop, sparse / the tall build's
// signed dense volume): 8 columns 22.1 / 50.3 ms, 12 columns 26.0 / 50.5, 4 columns 91 / 60
// (before empty stages were passed over, 8 columns then 79 / 51).
constexpr int kProjTU = 8, kProjThreads = kProjTU * kRingTV;

// Blocks per SM and ring words.  Four components (113 registers) take two blocks with 104 KB
// each, longer stages; two components three with 68 KB (64^3, 90 angles: 83 us against 94).
template <int S>
constexpr int kProjBlocks = S == 4 ? 2 : 3;
template <int S>
constexpr int kProjWords = S == 4 ? 26 * 1024 : 17 * 1024;
constexpr int kBrick = 8;               // occupancy is kept per 8 x 8 x 8 voxels
constexpr int kMaskWords = 64;          // stages whose occupancy a block keeps: 2048

// ---------------------------------------------------------------------------------
// rotated copies of the volume, z innermost:  out[vol][y][x][z][comp]
// ---------------------------------------------------------------------------------
// Source voxel (unpadded) of rotated voxel (X, Y) of copy r.
__device__ __forceinline__ void unrotate(int r, int X, int Y, int nx, int ny, int &sx, int &sy)
{
    sx = r == 0 ? X : r == 1 ? nx - 1 - Y : r == 2 ? nx - 1 - X : Y;
    sy = r == 0 ? Y : r == 1 ? X : r == 2 ? ny - 1 - Y : ny - 1 - X;
}

constexpr int kTileX = 32, kTileY = 8, kTileZ = 8;   // voxels per block of the layout kernels
static_assert(kTileY == kBrick && kTileZ == kBrick, "one brick high and deep");

// One block turns a 32 x 8 x 8 tile of every component of one rotated volume from the
// caller's x-fastest layout into the z-fastest, component-interleaved one.  Reads are
// contiguous along x (r even) or 8 voxels = one 32-byte sector along y (r odd); writes are
// runs of 8 z x S components.
//
// bricks[vol][y / 8][x / 8][z / 8]: whether any component of the 8 x 8 x 8 brick is nonzero.
template <int S, typename VT>
__global__ void __launch_bounds__(256) spread_kernel(const VT *__restrict__ vol, float *__restrict__ out,
                                                     unsigned char *__restrict__ bricks, int nx, int ny, int nz, int pzp,
                                                     int bzp, int64_t brick_stride)
{
    __shared__ float tile[S][kTileZ][kTileY][kTileX + 1];
    __shared__ int lit[kTileX / kBrick];
    const int tz = blockIdx.z % ((pzp + kTileZ - 1) / kTileZ), w = blockIdx.z / ((pzp + kTileZ - 1) / kTileZ);
    const int odd = S == 4 ? 0 : (w & 1);                    // orientation of this volume
    const int ex = (odd ? ny : nx) + 2, ey = (odd ? nx : ny) + 2;
    const int x0 = blockIdx.x * kTileX, y0 = blockIdx.y * kTileY, z0 = tz * kTileZ;
    if (x0 >= ex || y0 >= ey) return;
    const int t = threadIdx.x;
    if (t < kTileX / kBrick) lit[t] = 0;
#pragma unroll
    for (int c = 0; c < S; ++c) {
        const int r = S == 4 ? c : 2 * c + w;
#pragma unroll 4
        for (int i = t; i < kTileX * kTileY * kTileZ; i += 256) {
            const int zz = i >> 8, k = i & 255;
            // lanes along the source's contiguous axis: x for even turns, y for odd ones
            const int xx = (r & 1) ? k >> 3 : k & 31, yy = (r & 1) ? k & 7 : k >> 5;
            const int X = x0 + xx - 1, Y = y0 + yy - 1, Z = z0 + zz - 1;
            float v = 0.f;
            if (X >= 0 && X < ex - 2 && Y >= 0 && Y < ey - 2 && Z >= 0 && Z < nz) {
                int sx, sy;
                unrotate(r, X, Y, nx, ny, sx, sy);
                v = to_f(vol[((int64_t)Z * ny + sy) * nx + sx]);
            }
            tile[c][zz][yy][xx] = v;
        }
    }
    __syncthreads();
    float *base = out + (int64_t)w * S * pzp * ex * ey;
    bool any = false;            // of this thread's voxels, all in brick (t >> 6)
#pragma unroll 4
    for (int i = t; i < kTileX * kTileY * kTileZ; i += 256) {
        const int zz = i & 7, xx = (i >> 3) & 31, yy = i >> 8;
        const int X = x0 + xx, Y = y0 + yy, Z = z0 + zz;
#pragma unroll
        for (int c = 0; c < S; ++c) any |= tile[c][zz][yy][xx] != 0.f;
        if (X >= ex || Y >= ey || Z >= pzp) continue;
        float *p = base + (((int64_t)Y * ex + X) * pzp + Z) * S;
        if (S == 4)
            *reinterpret_cast<float4 *>(p) =
                make_float4(tile[0][zz][yy][xx], tile[1 % S][zz][yy][xx], tile[2 % S][zz][yy][xx], tile[3 % S][zz][yy][xx]);
        else
            *reinterpret_cast<float2 *>(p) = make_float2(tile[0][zz][yy][xx], tile[1][zz][yy][xx]);
    }
    if (__any_sync(kFull, any) && (t & 31) == 0) lit[t >> 6] = 1;      // two warps store the same value
    __syncthreads();
    if (t < kTileX / kBrick && x0 + t * kBrick < ex)
        bricks[w * brick_stride + ((int64_t)(y0 / kBrick) * ((ex + kBrick - 1) / kBrick) + x0 / kBrick + t) * bzp +
               z0 / kBrick] = (unsigned char)lit[t];
}

// Whether stage t's window holds a nonzero voxel, by the bricks it touches (ex: x extent of the
// rotated volume; nothing lies outside the grid).
__device__ __forceinline__ bool stage_lit(const RingParams &G, const unsigned char *bricks, const Window &W, int t, int align,
                                          int ex, int ey)
{
    const int ya = W.y0 + t * W.R, yb = min(ya + W.R, W.y1);
    int xa, za, xb, zb;
    corner(W, ya, align, xa, za);
    corner(W, yb, align, xb, zb);
    const int bx0 = max(min(xa, xb), 0) / kBrick, bx1 = min(max(xa, xb) + W.EX, ex) - 1;
    const int bz0 = max(min(za, zb), 0) / kBrick, bz1 = min(max(za, zb) + W.EZ, G.pzp) - 1;
    const int by0 = max(ya, 0) / kBrick, by1 = min(yb, ey - 1);
    const int nbx = (ex + kBrick - 1) / kBrick;
    unsigned long long any = 0;
    for (int by = by0; by * kBrick <= by1; ++by)
        for (int bx = bx0; bx * kBrick <= bx1; ++bx) {
            const unsigned char *row = bricks + ((int64_t)by * nbx + bx) * G.bzp;
            for (int z = bz0 & ~7; z * kBrick <= bz1; z += 8) {
                unsigned long long w = __ldg(reinterpret_cast<const unsigned long long *>(row + z));
                if (z < bz0) w &= ~0ull << (8 * (bz0 - z));
                const int over = z + 7 - bz1 / kBrick;
                if (over > 0) w &= ~0ull >> (8 * over);
                any |= w;
            }
        }
    return any != 0;
}

template <int S>
__device__ __forceinline__ void ld_shared(float (&v)[S], uint32_t p)
{
    if constexpr (S == 4)
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(p));
    else
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(p));
}
template <int S>
__device__ __forceinline__ void ld_global(float (&v)[S], const float *p)
{
    if constexpr (S == 4) {
        const float4 q = __ldg(reinterpret_cast<const float4 *>(p));
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
        const float2 q = __ldg(reinterpret_cast<const float2 *>(p));
        v[0] = q.x; v[1] = q.y;
    }
}

// acc += the run's weights times its cell's corners; p0, p1: shared addresses of element
// (x, z) of rows y and y + 1, xs: bytes from x to x + 1
template <int S>
__device__ __forceinline__ void gather_shared(float (&acc)[S], const Run &r, uint32_t p0, uint32_t p1, uint32_t xs)
{
    const uint32_t p[4] = {p0, p0 + xs, p1, p1 + xs};        // 2 y + x
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        float v[S];
        ld_shared<S>(v, p[2 * (k >> 2) + (k & 1)] + ((k >> 1) & 1) * S * 4);
#pragma unroll
        for (int c = 0; c < S; ++c) acc[c] = fmaf(r.w[k], v[c], acc[c]);
    }
}
template <int S>
__device__ __forceinline__ void gather_global(float (&acc)[S], const Run &r, const float *p0, const float *p1, int64_t xs)
{
    const float *p[4] = {p0, p0 + xs, p1, p1 + xs};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        float v[S];
        ld_global<S>(v, p[2 * (k >> 2) + (k & 1)] + ((k >> 1) & 1) * S);
#pragma unroll
        for (int c = 0; c < S; ++c) acc[c] = fmaf(r.w[k], v[c], acc[c]);
    }
}

__device__ __forceinline__ void tma_row(uint32_t dst, const CUtensorMap *map, int z, int x, int y, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(z), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// Bounded wait for an mbarrier phase (inlined: a call would cost the walk its registers).
__device__ __forceinline__ bool wait_rows(uint32_t bar, uint32_t parity)
{
    if (tc::mbar_try(bar, parity)) return true;
    const unsigned long long t0 = tc::globaltimer();
    while (!tc::mbar_try(bar, parity))
        if (tc::globaltimer() - t0 > tc::kWaitNs) return false;
    return true;
}

// ---------------------------------------------------------------------------------
// projection
// ---------------------------------------------------------------------------------
// The walk's registers decide how many warps an SM holds: what it does not need (the pixel
// sums, the window, the angle) waits in shared memory.
template <int S, typename PT>
__global__ void __launch_bounds__(kProjThreads, kProjBlocks<S>)
    ring_project_kernel(const RingParams G, const float *__restrict__ vols, PT *__restrict__ proj, uint32_t flags)
{
    extern __shared__ __align__(1024) float ring[];
    __shared__ int slots[3][kSlots];
    __shared__ int2 rowoff[2][kRowTab / 2];      // per buffer: a cell row's offset and the next row's
    __shared__ __align__(8) unsigned long long bars[2];
    __shared__ float pix[S][kProjThreads];
    __shared__ Window sW;
    __shared__ unsigned mask[kMaskWords];
    __shared__ double2 scs;
    constexpr int kAlign = 4 / S, kExq = 4 / S;

    const OpParams &P = G.op;
    const int lane = threadIdx.x, tid = threadIdx.y * kRingTV + lane;
    const uint32_t bar0 = tc::smem_u32(&bars[0]), ring0 = tc::smem_u32(ring);
    if (tid < 3 * kSlots) slot_reset(slots[tid / kSlots], tid % kSlots);
    if (tid == 0) {
        scs = G.cs[blockIdx.y];
        tc::mbar_init(bar0, 1);
        tc::mbar_init(bar0 + 8, 1);
        tc::mbar_init_fence();
    }
#pragma unroll
    for (int i = 0; i < S; ++i) pix[i][tid] = 0.f;
    __syncthreads();

    unsigned parity = 0;         // bit b: parity of the next wait on barrier b
    bool fine = true;            // no wait has run out
    bool wide = false;           // some bundle does not fit the ring
    // one aperture sample's ray, turned, and its block's window (left in sW)
    auto begin = [&](int a, RRay &R, int &turn) {
        const int u = blockIdx.x * kProjTU + threadIdx.y, v = blockIdx.z * kRingTV + lane;
        const bool active = u < P.nu && v < P.nv &&
                            ring_ray(G, ((int64_t)(a % P.M) * P.nv + v) * P.nu + u, scs, R, flags & VAMRT_UNATTENUATED);
        if (!active) R.jhi = R.j = 0;
        Window W;
        const bool any = bundle(G, slots[a % 3], active, false, R, kAlign, kExq, kProjWords<S> / S, true, turn, W);
        if (tid < kSlots) slot_reset(slots[(a + 2) % 3], tid);      // last read one aperture sample ago
        if (tid == 0) sW = W;
        __syncthreads();
        wide |= any && !W.ok;
        return any && W.ok;
    };
    // angle i's sum is component (i + shift) mod S
    auto add_pix = [&](const float(&o)[S], float w, int sh) {
#pragma unroll
        for (int c = 0; c < S; ++c) {
            float *q = &pix[(c + S - sh) & (S - 1)][tid];
            *q = fmaf(w, o[c], *q);
        }
    };
    for (int a = 0; a < P.M; ++a) {
        RRay R{};                    // all zero: nothing to walk, weight 0
        int turn;
        if (!begin(a, R, turn)) continue;
        const float ratio = exp2f(R.att);
        // which stages hold anything: the others add exactly nothing and are passed over
        const int stages = sW.stages, zpitch = sW.EZ;
        const bool known = stages <= 32 * kMaskWords;
        if (known) {
            const unsigned char *bricks = G.bricks + volume_of<S>(turn) * G.brick_stride;
            const int ex = ((turn & 1) ? P.ny : P.nx) + 2, ey = ((turn & 1) ? P.nx : P.ny) + 2;
            for (int t = tid; t < (stages + 31 & ~31); t += kProjThreads) {
                const unsigned m = __ballot_sync(kFull, t < stages && stage_lit(G, bricks, sW, t, kAlign, ex, ey));
                if (lane == 0) mask[t >> 5] = m;
            }
        }
        __syncthreads();
        auto next = [&](int t) {         // first stage >= t to walk
            if (!known) return min(t, stages);
            for (int w = t >> 5; 32 * w < stages; ++w) {
                const unsigned m = mask[w] & (32 * w < t ? ~0u << (t & 31) : ~0u);
                if (m) return 32 * w + __ffs(m) - 1;
            }
            return stages;
        };
        // fetch the rows of stage t into buffer b (warp 0, one lane per row)
        auto issue = [&](int t, int b) {
            const int R_ = sW.R, slab = sW.EX * sW.EZ, first = b * (R_ + 1);
            const CUtensorMap *map =
                G.maps + ((volume_of<S>(turn) * G.n_ex + (sW.EX - kMinEX) / kExq) * (kMaxEZ / kStepEZ) + sW.EZ / kStepEZ - 1);
            const int ya = sW.y0 + t * R_, n = min(R_, sW.y1 - ya) + 1;
            const uint32_t bar = bar0 + 8 * b;
            if (lane == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(n * slab * S * 4)
                             : "memory");
            __syncwarp();
            for (int i = lane; i < n; i += 32) {
                const int y = ya + i;
                int xo, zo;
                corner(sW, y, kAlign, xo, zo);
                // a cell's row and the next, in bytes (the walk adds its element's offset); the
                // shared last row belongs to the next stage's cells
                if (i < R_)
                    rowoff[b][i] = make_int2(row_offset(sW, y, kAlign, first + i) * S * 4,
                                                          row_offset(sW, y + 1, kAlign, first + i + 1) * S * 4);
                tma_row(ring0 + (uint32_t)((first + i) * slab * S * 4), map, zo * S, xo, y, bar);
            }
        };
        int cur = next(0), then = next(cur + 1), passed = 0;
        if (threadIdx.y == 0) {
            if (cur < stages) issue(cur, 0);
            if (then < stages) issue(then, 1);
        }
        __syncthreads();
        for (int b = 0; cur < stages; b ^= 1) {
            if (fine) fine = wait_rows(bar0 + 8 * b, (parity >> b) & 1);
            parity ^= 1u << b;
            if (cur != passed && R.j < R.jhi) {
                const int n = samples_below(R, sW.y0 + cur * sW.R);
                R.j += n;
                R.qx += n * R.sx;
                R.qy += n * R.sy;
                R.qz += n * R.sz;
            }
            float o[S] = {};
            const int ya = sW.y0 + cur * sW.R;
            walk(R, ratio, 1.0f, INT_MAX, ya + sW.R, zpitch, [&](int e, int y, const Run &r) {
                const int2 off = rowoff[b][y - ya];
                const uint32_t at = ring0 + (uint32_t)(e * S * 4);
                gather_shared<S>(o, r, at + off.x, at + off.y, zpitch * S * 4);
            });
            add_pix(o, R.w, shift_of<S>(turn));
            passed = cur + 1;
            cur = then;
            then = next(then + 1);
            __syncthreads();
            if (threadIdx.y == 0 && then < stages) issue(then, b);
        }
    }
    // Bundles too wide for the ring: the same walk on the rotated volume itself, in a loop of
    // its own (its 64-bit addresses would cost the common walk 30 registers).
    if (wide) {
        __syncthreads();
        for (int a = 0; a < P.M; ++a) {
            RRay R{};
            int turn;
            if (begin(P.M + a, R, turn)) continue;
            const float ratio = exp2f(R.att);
            const float *vol = vols + (int64_t)volume_of<S>(turn) * G.vol_elems * S;
            const int64_t row = (int64_t)(((turn & 1) ? P.ny : P.nx) + 2) * G.pzp;
            while (R.j < R.jhi) {
                float o[S] = {};
                walk(R, ratio, 1.0f, 16, INT_MAX, G.pzp, [&](int e, int y, const Run &r) {
                    const float *p = vol + (y * row + e) * S;
                    gather_global<S>(o, r, p, p + row * S, (int64_t)G.pzp * S);
                });
                add_pix(o, R.w, shift_of<S>(turn));
            }
        }
    }
    if (!fine) {
        // a copy did not arrive in time: give what is in flight one more bounded wait, and
        // make the result visibly wrong
        wait_rows(bar0, parity & 1);
        wait_rows(bar0 + 8, (parity >> 1) & 1);
    }
    const int u = blockIdx.x * kProjTU + threadIdx.y, v = blockIdx.z * kRingTV + lane;
    if (u < P.nu && v < P.nv) {
#pragma unroll
        for (int i = 0; i < S; ++i) {
            PT *out = proj + (((int64_t)G.members[(int64_t)blockIdx.y * S + i] * P.nv + v) * P.nu + u);
            float x = fine ? pix[i][tid] : __int_as_float(0x7fffffff);
            if (flags & VAMRT_ACCUMULATE) x += to_f(*out);
            if ((flags & VAMRT_CLAMP_NONNEG) && fine) x = fmaxf(x, 0.f);
            st_val(out, x);
        }
    }
}

}  // namespace

// Partition angles into groups theta0 + i 2 pi / S, S the largest of `max_s` and 2 for which every
// angle has its partners (to 1e-12 rad); 0 without partners.  members: S angle indices per group.
int plan_ring_groups(const double *theta, int n, int max_s, std::vector<int> &members, std::vector<double> &base)
{
    for (int S = max_s; S >= 2; S >>= 1) {
        const double turn = 2.0 * M_PI / S;
        if (n % S) continue;
        struct Item {
            double rest;
            int quad, k;
        };
        std::vector<Item> it((size_t)n);
        for (int k = 0; k < n; ++k) {
            double q = floor(theta[k] / turn + 1e-9);
            double rest = theta[k] - q * turn;
            it[(size_t)k] = {rest, (int)((long long)fmod(q, (double)S) + S) % S, k};
        }
        std::stable_sort(it.begin(), it.end(), [](const Item &a, const Item &b) { return a.rest < b.rest; });
        bool good = true;
        members.assign((size_t)n, -1);
        base.assign((size_t)(n / S), 0.0);
        for (int g = 0; g < n / S && good; ++g) {
            unsigned seen = 0;
            for (int i = 0; i < S; ++i) {
                const Item &x = it[(size_t)(g * S + i)];
                if (fabs(x.rest - it[(size_t)(g * S)].rest) > 1e-12 || (seen >> x.quad & 1)) { good = false; break; }
                seen |= 1u << x.quad;
                members[(size_t)(g * S + x.quad)] = x.k;
            }
            // the first member's own angle: exact for it, turned for its partners
            if (good) base[(size_t)g] = theta[members[(size_t)(g * S)]];
        }
        if (good) return S;
    }
    return 0;
}

int ring_ex_classes(int S) { return (kMaxEX - kMinEX) / (4 / S) + 1; }
size_t ring_map_count(int S) { return (size_t)(4 / S) * ring_ex_classes(S) * (kMaxEZ / kStepEZ); }

// Tensor maps of the rotated volumes for every window class, in the kernel's order.
cudaError_t ring_maps(const RingParams &G, int S, const float *vols, std::vector<CUtensorMap> &maps)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = tma_encoder();
    if (!enc) return cudaErrorNotSupported;
    const int exq = 4 / S, n_ex = ring_ex_classes(S), n_ez = kMaxEZ / kStepEZ;
    maps.resize(ring_map_count(S));
    for (int w = 0; w < 4 / S; ++w) {
        const int odd = S == 4 ? 0 : (w & 1);
        const cuuint64_t ex = (cuuint64_t)(odd ? G.op.ny : G.op.nx) + 2, ey = (cuuint64_t)(odd ? G.op.nx : G.op.ny) + 2;
        const cuuint64_t dims[3] = {(cuuint64_t)G.pzp * S, ex, ey};
        const cuuint64_t str[2] = {(cuuint64_t)G.pzp * S * 4, (cuuint64_t)G.pzp * S * 4 * ex};
        const cuuint32_t one[3] = {1, 1, 1};
        for (int i = 0; i < n_ex; ++i)
            for (int k = 0; k < n_ez; ++k) {
                const cuuint32_t box[3] = {(cuuint32_t)((k + 1) * kStepEZ * S), (cuuint32_t)(kMinEX + i * exq), 1};
                if (enc(&maps[((size_t)w * n_ex + i) * n_ez + k], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
                        const_cast<float *>(vols) + (size_t)w * S * G.vol_elems, dims, str, box, one,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                    return cudaErrorInvalidValue;
            }
    }
    return cudaSuccess;
}

cudaError_t launch_ring_spread(const vamrt_projector *p, const void *vol, vamrt_dtype dt, cudaStream_t s)
{
    const RingParams &G = p->ring;
    const int nx = G.op.nx, ny = G.op.ny, m = std::max(nx, ny) + 2;
    const int zt = (G.pzp + kTileZ - 1) / kTileZ;
    return by_group(p->ring_s, [&](auto s_) {
        constexpr int S = decltype(s_)::value;
        const dim3 grid((unsigned)((m + kTileX - 1) / kTileX), (unsigned)((m + kTileY - 1) / kTileY),
                        (unsigned)(zt * (4 / S)));
        return by_storage(dt, const_cast<void *>(vol), [&](auto *v) {
            spread_kernel<S><<<grid, 256, 0, s>>>(v, p->ring_vols, p->ring_bricks, nx, ny, G.op.nz, G.pzp, G.bzp,
                                                  G.brick_stride);
            count_launches(1);
            return cudaGetLastError();
        });
    });
}

cudaError_t launch_ring_project(const vamrt_projector *p, void *proj, vamrt_dtype dt, uint32_t flags, cudaStream_t s)
{
    const RingParams &G = p->ring;
    return by_group(p->ring_s, [&](auto s_) {
        constexpr int S = decltype(s_)::value;
        constexpr size_t kSmem = sizeof(float) * kProjWords<S>;
        return by_storage(dt, proj, [&](auto *pr) {
            using PT = std::remove_pointer_t<decltype(pr)>;
            cudaError_t e = cudaFuncSetAttribute(ring_project_kernel<S, PT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)kSmem);
            if (e != cudaSuccess) return e;
            ring_project_kernel<S, PT><<<ring_grid(G, kProjTU), dim3(kRingTV, kProjTU), kSmem, s>>>(G, p->ring_vols, pr, flags);
            count_launches(1);
            return cudaGetLastError();
        });
    });
}

}  // namespace vamrt
