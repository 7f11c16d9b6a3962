// What the two hot operators share (ring_project.cu, ring_dose.cu): rays of a group of angles,
// a block's bundle and the window that follows it through the rows of the grid.
//
// Symmetry.  A scan over a full turn in N equal steps holds, with every angle theta, also
// theta + 180 degrees (N even) and theta + 90, 270 (N a multiple of 4, square grids).  A
// quarter turn maps the voxel lattice onto itself, so ray r at theta + 90 i samples the
// volume turned back by 90 i degrees at exactly the positions it samples the volume itself
// at theta.  All S angles of such a group (S = 4 or 2) are walked at once: one ray set-up in FP64, one position, one cell and one set of
// trilinear weights per sample serve S angles.  The projection reads the S rotated volumes
// interleaved, one 16-byte (8) shared-memory read per corner; the dose (S = 4 only) adds into
// rotated accumulators.  Positions are those of the group's first angle: cos and sin of
// the partners would differ from its turned ones by FP64 rounding only (1e-16 rad).
//
// Direction.  The rotated copies W_0 .. W_3 of the volume (W_r(p) = v(p turned by 90 r))
// also let every block walk its rays along +y: it turns its rays by the quarter turn that
// brings their mean direction within 45 degrees of +y and starts from copy r.
//
// Rows and windows.  A block owns a few pixel columns x 32 pixel rows of one group; lanes run
// down a column, so a warp's samples are stacked along z.  Its rays pass through the grid's y
// rows in order.  Per row the block holds a window of EX voxels along x and EZ along z in
// shared memory, z innermost; the window follows the bundle (its corner is a linear function
// of y: the lower envelope of straight lines is concave, so the chord between its values at
// the first and the last row bounds it).  At the 0.05 mm large print a window is 9-16 x 40
// voxels; a box that is aligned with the axes and deep enough to be worth a stage holds
// twice as many voxels per sample where the rays run diagonally.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <limits.h>

#include "internal.cuh"

namespace vamrt {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr double kFix = 4294967296.0;   // 2^32

constexpr int kRingTV = 32;             // pixel rows of a block: a warp's lanes
constexpr int kRowTab = 64;             // rows resident at a time stay below this
constexpr int kMaxEX = 32, kMaxEZ = 64, kMinEX = 8;
constexpr int kStepEZ = 8;              // EZ granularity: whole 128-byte shared-memory slots

__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ float to_f(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ float to_f(__half x) { return __half2float(x); }
__device__ __forceinline__ void st_val(float *p, float x) { *p = x; }
__device__ __forceinline__ void st_val(__nv_bfloat16 *p, float x) { *p = __float2bfloat16_rn(x); }
__device__ __forceinline__ void st_val(__half *p, float x) { *p = __float2half_rn(x); }

// ---------------------------------------------------------------------------------
// rays
// ---------------------------------------------------------------------------------
struct RRay {
    long long qx, qy, qz;   // Q32.32 position of the current sample (turned, padded index coordinates)
    long long sx, sy, sz;   // Q32.32 advance per sample
    float att;              // log2 of the Beer-Lambert factor per sample
    float w;                // T1 T2 delta_mm / M
    int j, jhi;             // current sample, end
};

// Ray r at the group's first angle, relative to the axis (the turn and the grid centre are
// applied by place()).
__device__ __forceinline__ bool ring_ray(const RingParams &G, int64_t r, double2 cs, RRay &R, bool unattenuated)
{
    const int2 J = G.op.J[r];
    if (J.x >= J.y) return false;
    const double4_32a A = G.op.A[r], B = G.op.B[r];
    const double c = cs.x, s = cs.y, dl = A.w;
    const double stx = (c * B.x - s * B.y) * dl;
    const double sty = (s * B.x + c * B.y) * dl;
    const double stz = B.z * dl;
    // sample 0 sits half a step inside the entry point
    R.qx = __double2ll_rn(((c * A.x - s * A.y) + 0.5 * stx) * kFix);
    R.qy = __double2ll_rn(((s * A.x + c * A.y) + 0.5 * sty) * kFix);
    R.qz = __double2ll_rn((G.op.cz + A.z + 0.5 * stz) * kFix);
    R.sx = __double2ll_rn(stx * kFix);
    R.sy = __double2ll_rn(sty * kFix);
    R.sz = __double2ll_rn(stz * kFix);
    R.att = unattenuated ? 0.f : G.op.neg_mu_vox_log2e * (float)A.w;
    R.w = unattenuated ? (float)A.w * G.op.h_over_m : (float)B.w;
    // every sample's cell and the cell above it must lie in the padded grid in z: drop end
    // samples that the rounding carries a hair outside (their in-grid weight is nil)
    int jlo = J.x, jhi = J.y;
    const long long top = (long long)(G.op.pz - 1) << 32;
    auto inside = [&](int j) {
        const long long q = R.qz + (long long)j * R.sz;
        return q >= 0 && q < top;
    };
    for (int t = 0; t < 4 && jlo < jhi && !inside(jlo); ++t) ++jlo;
    for (int t = 0; t < 4 && jlo < jhi && !inside(jhi - 1); ++t) --jhi;
    if (jlo < jhi && !(inside(jlo) && inside(jhi - 1))) jhi = jlo;
    R.j = jlo;
    R.jhi = jhi;
    return jlo < jhi;
}

// Turn a ray by -90 r degrees about the axis and move it to sample R.j in padded indices.
__device__ __forceinline__ void place(const RingParams &G, int r, RRay &R)
{
    if (r & 1) {
        const long long qx = R.qx, sx = R.sx;
        R.qx = R.qy; R.qy = -qx;
        R.sx = R.sy; R.sy = -sx;
    }
    if (r & 2) {
        R.qx = -R.qx; R.qy = -R.qy;
        R.sx = -R.sx; R.sy = -R.sy;
    }
    // centres are multiples of one half: exact in Q32.32
    const long long cx = (long long)(((r & 1) ? G.op.cy : G.op.cx) * 2.0) << 31;
    const long long cy = (long long)(((r & 1) ? G.op.cx : G.op.cy) * 2.0) << 31;
    R.qx += cx + (long long)R.j * R.sx;
    R.qy += cy + (long long)R.j * R.sy;
    R.qz += (long long)R.j * R.sz;
}

// ---------------------------------------------------------------------------------
// a block's bundle: turn, rows, window
// ---------------------------------------------------------------------------------
struct Window {
    int y0, y1;              // rows y0..y1 are touched
    float lx, lsx, lz, lsz;  // lower corner at row y: l + (y - y0) ls, minus |ls|, floored
    int EX, EZ, R, stages;
    bool ok;
};

// fields of the block's reduction slots
enum { kDirX, kDirY, kYMin, kYMax, kBad, kX0Lo, kX0Hi, kX1Lo, kX1Hi, kZ0Lo, kZ0Hi, kZ1Lo, kZ1Hi, kSlots };

__device__ __forceinline__ void slot_reset(int *s, int k)
{
    const bool lo = k == kYMin || k == kX0Lo || k == kX1Lo || k == kZ0Lo || k == kZ1Lo;
    const bool hi = k == kYMax || k == kX0Hi || k == kX1Hi || k == kZ0Hi || k == kZ1Hi;
    s[k] = lo ? INT_MAX : hi ? INT_MIN : 0;
}

__device__ __forceinline__ int fix8(long long q) { return (int)(q >> 24); }   // Q32.32 -> 1/256 voxel, floored

// Block-uniform; every thread calls it with its ray (placed rays when it returns).  `align`:
// z alignment of the window's corner; `exq`: EX granularity; bad_ray:
// the ray wants the walk on global memory.  Returns false when the block has no active ray.
__device__ __forceinline__ bool bundle(const RingParams &G, int *s, bool active, bool bad_ray, RRay &R, int align,
                                       int exq, int cap, bool split, int &turn, Window &W)
{
    const bool lead = threadIdx.x == 0;
    // mean direction -> quarter turn
    int dx = active ? (int)(R.sx >> 16) : 0, dy = active ? (int)(R.sy >> 16) : 0;
    dx = __reduce_add_sync(kFull, dx);
    dy = __reduce_add_sync(kFull, dy);
    if (lead && (dx | dy)) {
        atomicAdd(&s[kDirX], dx);
        atomicAdd(&s[kDirY], dy);
    }
    __syncthreads();
    dx = s[kDirX];
    dy = s[kDirY];
    turn = abs(dy) >= abs(dx) ? (dy > 0 ? 0 : 2) : (dx < 0 ? 1 : 3);
    int ylo = INT_MAX, yhi = INT_MIN, bad = 0;
    if (active) {
        place(G, turn, R);
        const long long m = max(llabs(R.sx), llabs(R.sz));
        bad = 4 * R.sy >= m && R.sy > 0 && !bad_ray ? 0 : 1;
        const int yf = (int)(R.qy >> 32), yl = (int)((R.qy + (long long)(R.jhi - 1 - R.j) * R.sy) >> 32);
        ylo = min(yf, yl);
        yhi = max(yf, yl) + 1;
    }
    ylo = __reduce_min_sync(kFull, ylo);
    yhi = __reduce_max_sync(kFull, yhi);
    bad = __reduce_max_sync(kFull, bad);
    if (lead && ylo <= yhi) {
        atomicMin(&s[kYMin], ylo);
        atomicMax(&s[kYMax], yhi);
    }
    if (lead && bad) atomicMax(&s[kBad], 1);
    __syncthreads();
    W.y0 = s[kYMin];
    W.y1 = s[kYMax];
    if (W.y0 > W.y1) return false;
    W.ok = s[kBad] == 0;
    if (!W.ok) return true;                       // block-uniform
    // x and z of the rays' lines at rows y0 and y1, in 1/256 voxel, 1/64 voxel to spare
    int x0 = INT_MAX, x0h = INT_MIN, x1 = INT_MAX, x1h = INT_MIN, z0 = INT_MAX, z0h = INT_MIN, z1 = INT_MAX, z1h = INT_MIN;
    if (active) {
        const float inv = 1.0f / (float)R.sy;
        const float gx = (float)R.sx * inv, gz = (float)R.sz * inv;
        const float t0 = (float)(((long long)W.y0 << 32) - R.qy) * (256.0f / 4294967296.0f);
        const float t1 = (float)(((long long)W.y1 << 32) - R.qy) * (256.0f / 4294967296.0f);
        const int xi = fix8(R.qx), zi = fix8(R.qz);
        const int ax = xi + (int)floorf(t0 * gx), bx = xi + (int)floorf(t1 * gx);
        const int az = zi + (int)floorf(t0 * gz), bz = zi + (int)floorf(t1 * gz);
        x0 = ax - 4; x0h = ax + 6; x1 = bx - 4; x1h = bx + 6;
        z0 = az - 4; z0h = az + 6; z1 = bz - 4; z1h = bz + 6;
    }
    x0 = __reduce_min_sync(kFull, x0); x0h = __reduce_max_sync(kFull, x0h);
    x1 = __reduce_min_sync(kFull, x1); x1h = __reduce_max_sync(kFull, x1h);
    z0 = __reduce_min_sync(kFull, z0); z0h = __reduce_max_sync(kFull, z0h);
    z1 = __reduce_min_sync(kFull, z1); z1h = __reduce_max_sync(kFull, z1h);
    if (lead && x0 != INT_MAX) {
        atomicMin(&s[kX0Lo], x0); atomicMax(&s[kX0Hi], x0h);
        atomicMin(&s[kX1Lo], x1); atomicMax(&s[kX1Hi], x1h);
        atomicMin(&s[kZ0Lo], z0); atomicMax(&s[kZ0Hi], z0h);
        atomicMin(&s[kZ1Lo], z1); atomicMax(&s[kZ1Hi], z1h);
    }
    __syncthreads();
    const float k = 1.0f / 256.0f, inv_n = 1.0f / (float)(W.y1 - W.y0);     // y1 > y0 always
    W.lx = (float)s[kX0Lo] * k;
    W.lz = (float)s[kZ0Lo] * k;
    W.lsx = (float)(s[kX1Lo] - s[kX0Lo]) * k * inv_n;
    W.lsz = (float)(s[kZ1Lo] - s[kZ0Lo]) * k * inv_n;
    const float usx = (float)(s[kX1Hi] - s[kX0Hi]) * k * inv_n, usz = (float)(s[kZ1Hi] - s[kZ0Hi]) * k * inv_n;
    const float wx = (float)max(s[kX0Hi] - s[kX0Lo], s[kX1Hi] - s[kX1Lo]) * k + fabsf(W.lsx) + fabsf(usx);
    const float wz = (float)max(s[kZ0Hi] - s[kZ0Lo], s[kZ1Hi] - s[kZ1Lo]) * k + fabsf(W.lsz) + fabsf(usz);
    if (!(wx < (float)kMaxEX && wz < (float)kMaxEZ)) {
        W.ok = false;
        return true;
    }
    W.EX = ((max((int)floorf(wx + 0.01f) + 3, kMinEX) + exq - 1) / exq) * exq;
    W.EZ = (((int)floorf(wz + 0.01f) + 3 + align - 1 + kStepEZ - 1) / kStepEZ) * kStepEZ;
    if (W.EX > kMaxEX || W.EZ > kMaxEZ) {
        W.ok = false;
        return true;
    }
    // rows per stage: two stages fit, each with its own copy of the row it shares with the next
    // (split), or one ring of 2 R + 1 rows
    const int rows = min(cap / (W.EX * W.EZ), kRowTab - 2);
    W.R = split ? (rows >> 1) - 1 : (rows - 1) >> 1;
    if (W.R < 1) {
        W.ok = false;
        return true;
    }
    W.stages = (W.y1 - W.y0 + W.R - 1) / W.R;
    return true;
}

// Window corner of row y.
__device__ __forceinline__ void corner(const Window &W, int y, int align, int &xo, int &zo)
{
    const float t = (float)(y - W.y0);
    xo = (int)floorf(fmaf(t, W.lsx, W.lx) - fabsf(W.lsx));
    zo = (int)floorf(fmaf(t, W.lsz, W.lz) - fabsf(W.lsz)) & ~(align - 1);
}

// Ring offset of row y in slot `slot`: element (x, z) of the row sits at offset + x EZ + z.
__device__ __forceinline__ int row_offset(const Window &W, int y, int align, int slot)
{
    int xo, zo;
    corner(W, y, align, xo, zo);
    return slot * (W.EX * W.EZ) - xo * W.EZ - zo;
}

__device__ __forceinline__ float frac_one(unsigned lo)
{
    // 1 + the fraction's top 23 bits, exactly: the funnel shift brings in the exponent of 1.0
    return __uint_as_float(__funnelshift_r(lo, 0x7fu, 9));
}

// Trilinear weights of a run of samples in one cell, corner (x, y, z) at 4 y + 2 z + x.
struct Run {
    float w[8];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k] = 0.f;
    }
    // one more sample of weight att; F = 1 + fraction
    __device__ __forceinline__ void add(float Fx, float Fy, float Fz, float att)
    {
        const float fx = Fx - 1.0f, gx = 2.0f - Fx;
        const float z1 = fmaf(att, Fz, -att), z0 = att - z1;            // att (F - 1), rounded once
        const float y01 = fmaf(z0, Fy, -z0), y00 = z0 - y01, y11 = fmaf(z1, Fy, -z1), y10 = z1 - y11;   // y[z][y]
        const float t[4] = {y00, y10, y01, y11};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            w[2 * k] = fmaf(t[k], gx, w[2 * k]);
            w[2 * k + 1] = fmaf(t[k], fx, w[2 * k + 1]);
        }
    }
};

// Number of the ray's remaining samples with row < lim (its advance along y is positive).
__device__ __forceinline__ int samples_below(const RRay &R, int lim)
{
    const long long L = ((long long)lim << 32) - R.qy;
    if (L <= 0) return 0;
    // the float quotient is within one of the exact one: start below it and count up
    int k = max((int)((float)L / (float)R.sy) - 1, 0);
#pragma unroll
    for (int t = 0; t < 3; ++t) k += (long long)k * R.sy < L ? 1 : 0;
    return min(k, R.jhi - R.j);
}

// Walks the ray's samples with row < lim, at most n of them: flush(e, y, run) is called
// once per run of samples in one cell, at x zpitch + z = e of row y.  Weights carry `unit`
// (a power of two).
template <typename F>
__device__ __forceinline__ void walk(RRay &R, float ratio, float unit, int n, int lim, int zpitch, F &&flush)
{
    int y = (int)(R.qy >> 32);
    n = min(n, R.jhi - R.j);
    if (n <= 0 || y >= lim) return;
    float att = unit * exp2f(R.att * ((float)R.j + 0.5f));   // exact at each stage, then one product per sample
    const int last = R.j + n;
    Run r;
    r.clear();
    int ce = (int)(R.qx >> 32) * zpitch + (int)(R.qz >> 32), cy = y, e = ce;
    do {
        if (e != ce || y != cy) {
            flush(ce, cy, r);
            r.clear();
            ce = e;
            cy = y;
        }
        r.add(frac_one((unsigned)R.qx), frac_one((unsigned)R.qy), frac_one((unsigned)R.qz), att);
        att *= ratio;
        R.qx += R.sx;
        R.qy += R.sy;
        R.qz += R.sz;
        ++R.j;
        y = (int)(R.qy >> 32);
        e = (int)(R.qx >> 32) * zpitch + (int)(R.qz >> 32);
    } while (R.j < last && y < lim);
    flush(ce, cy, r);
}

// component of angle i of a group when the block's turn is r, and the volume it lies in
template <int S>
__device__ __forceinline__ int volume_of(int r) { return S == 4 ? 0 : (r & 1); }
template <int S>
__device__ __forceinline__ int shift_of(int r) { return S == 4 ? r : (r >> 1); }

inline dim3 ring_grid(const RingParams &G, int columns)
{
    return dim3((G.op.nu + columns - 1) / columns, G.n_groups, (G.op.nv + kRingTV - 1) / kRingTV);
}

template <typename F>
cudaError_t by_storage(vamrt_dtype dt, void *ptr, F &&f)
{
    if (dt == VAMRT_F32) return f((float *)ptr);
    if (dt == VAMRT_BF16) return f((__nv_bfloat16 *)ptr);
    return f((__half *)ptr);
}

template <typename F>
cudaError_t by_group(int S, F &&f)
{
    return S == 4 ? f(std::integral_constant<int, 4>()) : f(std::integral_constant<int, 2>());
}

}  // namespace
}  // namespace vamrt
