// Internal declarations shared by the vamrt CUDA translation units.
#pragma once

#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <stdint.h>

#include <vector>

#include "../../include/vamrt.h"

namespace vamrt {

// Largest optimiser run whose error history the handle keeps on the device.
constexpr int kMaxHistory = 4096;
// Partial-sum slots for the deterministic two-pass reductions.
constexpr int kRedBlocks = 1024;

// Operator tiling: a block owns kTileU x kTileV pixels of one angle and walks their rays
// chunk by chunk along the projection axis (kChunkVox voxels of the theta = 0 frame's y
// per chunk).  Each chunk's voxel footprint is staged in a shared-memory box of at most
// kBoxFloats floats; a chunk whose box would not fit runs straight on global memory.
constexpr int kTileU = 8;
constexpr int kTileV = 32;
constexpr int kThreads = kTileU * kTileV;
constexpr int kChunkVox = 20;
constexpr int kBoxFloats = 18 * 1024;
constexpr int kBlocksPerSm = 3;

// Per-launch constants of the two operators.  Positions are in padded index
// coordinates: the scratch volume has a zero halo of one voxel on every face (and its
// rows are padded to a multiple of 4 floats), so voxel (i,j,k) of the caller's grid
// sits at (i+1, j+1, k+1).
struct OpParams {
    const double4_32a *A; // (e_x, e_y, e_z, delta) in voxels, theta = 0 frame, relative to the axis
    const double4_32a *B; // (d_x, d_y, d_z, T1 T2 delta_mm / M)
    const int2 *J;        // [j_lo, j_hi) samples whose footprint reaches the grid
    const double2 *cs;    // (cos theta_k, sin theta_k), FP64
    int nu, nv, M, n_angles;
    int nx, ny, nz;       // caller's grid
    int px, py, pz;       // padded extents (px a multiple of 4)
    double cx, cy, cz;    // axis position in padded index coordinates
    float neg_mu_vox_log2e;  // -mu h log2(e): attenuation = exp2(this * s_vox)
    float y0;             // start of chunk 0 on the theta = 0 frame's y axis, voxels
    float cell_bound;     // most samples of one ray whose footprint holds a given voxel
    float h_over_m;       // voxel pitch (mm) / rays per pixel: delta_mm / M = delta_vox * h_over_m
};

// The voxel error rate's device state, cleared before each use: histograms of the in-part and
// the out-of-part resin voxels, the dose's maximum over the resin, and blocks done.
constexpr int kVerBins = 1024;
struct VerState {
    unsigned hist[2 * kVerBins];
    float dmax;
    unsigned counter;
};

// Per-launch constants of the grouped operators (ring.cuh).  Groups of S angles a quarter,
// half or whole turn apart are walked together on rotated copies of the volume.
struct RingParams {
    OpParams op;
    int n_groups;
    const double2 *cs;     // (cos, sin) of each group's first angle, FP64
    const int *members;    // S angle indices per group, 2 pi / S apart
    int pzp;               // z extent of the rotated copies: nz + 2 rounded up to 4
    int64_t vol_elems;     // voxels of one copy: (nx + 2) (ny + 2) pzp
    const unsigned char *bricks;   // occupancy of the rotated copies, 8^3 voxels a byte
    int bzp;               // bricks along z, rounded up to 8
    int64_t brick_stride;  // bricks of one copy
    const CUtensorMap *maps;   // device: [copy][EX class][EZ class]
    int n_ex;              // EX classes
    float share_scale;     // fixed-point units of the largest ray weight (dose)
};

// Per-ray constants of the FP64 tracer.
struct TraceParams {
    const double *pupil_xy;   // device, M pairs (aperture = VAMRT_APERTURE_LIST)
    int aperture;             // VAMRT_APERTURE_*
    int per_pixel;            // jitter drawn per pixel
    unsigned long long seed;
    int strat_n;              // strata per side (stratified aperture)
    int nu, nv, M, nz;
    double pu, pv;
    double pupil_mm, f_number;
    int telecentric, chief_only;
    double r_in, r_out, n_out, n_glass, n_resin;
    double h, ds;
    const double *surf;       // device, n_surf x (y, radius, n_after, clear, stop flag); n_surf = 0: pupil model
    int n_surf;
    double obj_y, mag, aim, stop_r;
};

}  // namespace vamrt

struct vamrt_projector {
    vamrt_geometry g;          // copy; host pointers cleared
    int device;
    int num_sms;
    int64_t n_rays;
    int64_t rays_in_resin;
    uint64_t samples_per_angle;
    uint64_t device_bytes;
    double4_32a *tabA;         // FP64: a large grid's positions need more than FP32's 24 bits
    double4_32a *tabB;
    int2 *tabJ;
    double2 *cs;
    float *scratch;            // padded FP32 volume, pad_elems floats
    int64_t pad_elems;
    unsigned char *pad_bricks; // which 8^3 bricks of the padded volume hold anything
    double *red;               // kRedBlocks partials + scalars
    double *hist;              // kMaxHistory errors
    vamrt::VerState *ver;
    int2 *spans;               // per y: [first, end) resin voxel of the row
    double *host_err;          // pinned, 4 doubles: the optimiser's E and VER counts
    vamrt::OpParams op;
    int ring_s;                // angles per group of the grouped projection; 0: not set up
    int ring_dose;             // the dose is grouped too
    float *ring_vols;          // 4 rotated copies of the volume, or dose accumulators; the others lie behind them
    unsigned char *ring_bricks;
    double2 *ring_cs;
    int *ring_members;
    CUtensorMap *ring_maps;
    vamrt::RingParams ring;
};

namespace vamrt {

// Count of kernel launches issued by the library (vamrt_launch_count).
void count_launches(unsigned n);
// Set the calling thread's vamrt_last_error() text.
void set_error(const char *msg);

// raytable.cu
cudaError_t launch_raytable(const TraceParams &T, double4_32a *A, double4_32a *B, int2 *J,
                            unsigned long long *counters, cudaStream_t s);

// static_dose.cu: device address of the allocation-free dose entry point's static
// accumulator on the current device `dev` (loads its module on first use)
cudaError_t static_acc_address(int dev, float **out);

// operators.cu
cudaError_t operators_init();
cudaError_t launch_pad(const vamrt_projector *p, const void *vol, vamrt_dtype dt, cudaStream_t s);
cudaError_t launch_adjoint(const vamrt_projector *p, vamrt_dtype vol_dt, void *proj, vamrt_dtype proj_dt,
                           uint32_t flags, cudaStream_t s);
cudaError_t launch_forward(const vamrt_projector *p, const void *proj, vamrt_dtype proj_dt, cudaStream_t s);
cudaError_t launch_unpad(const vamrt_projector *p, void *dose, vamrt_dtype dt, uint32_t flags, cudaStream_t s);
// The same two steps on a caller-chosen FP32 accumulator of p->pad_elems floats (the
// caller zeroes it first).
cudaError_t launch_forward_acc(const vamrt_projector *p, const void *proj, vamrt_dtype proj_dt, float *acc,
                               cudaStream_t s);
cudaError_t launch_unpad_acc(const vamrt_projector *p, const float *acc, void *dose, vamrt_dtype dt, uint32_t flags,
                             cudaStream_t s);

// ring_project.cu: the projection over groups of angles.  Partition the angles (plan), tensor
// maps of the rotated copies, and the launches: spread = caller's volume -> rotated copies.
int plan_ring_groups(const double *theta, int n, int max_s, std::vector<int> &members, std::vector<double> &base);
int ring_ex_classes(int S);
size_t ring_map_count(int S);
cudaError_t ring_maps(const RingParams &G, int S, const float *vols, std::vector<CUtensorMap> &maps);
cudaError_t launch_ring_spread(const vamrt_projector *p, const void *vol, vamrt_dtype dt, cudaStream_t s);
cudaError_t launch_ring_project(const vamrt_projector *p, void *proj, vamrt_dtype dt, uint32_t flags, cudaStream_t s);

// ring_dose.cu: the dose over groups of angles into four rotated accumulators, and their sum
// -> out at the given pitches (elements).
cudaError_t launch_ring_dose(const vamrt_projector *p, const void *proj, vamrt_dtype dt, cudaStream_t s);
cudaError_t launch_ring_gather(const vamrt_projector *p, void *out, vamrt_dtype dt, int64_t row, int64_t plane,
                               int64_t origin, int accumulate, cudaStream_t s);

// loss.cu: loss3 = device doubles {L, 1/|P|, 1/|Q|}; grad may be NULL
cudaError_t launch_threshold_loss(const vamrt_projector *p, const void *dose, vamrt_dtype dose_dt,
                                  const float *target, float d_l, float d_h, double *loss3, void *grad,
                                  vamrt_dtype grad_dt, cudaStream_t s);

// loss.cu: out2 = device {count, sum} of x over target > 1/2 (target given) or over x > 0
// (target NULL), summed in a fixed order
cudaError_t launch_masked_sum(const vamrt_projector *p, const void *x, vamrt_dtype dt, const float *target,
                              int64_t n, double *out2, cudaStream_t s);
// loss.cu: master = sc * x in FP32; x (in dt) rewritten from master when it is not master itself
cudaError_t launch_scale_master(const vamrt_projector *p, void *x, vamrt_dtype dt, float *master, int64_t n, float sc,
                                cudaStream_t s);

// ver.cu: the resin rows' ends (once per handle); out3 = device {best mismatch count, best
// threshold index, resin voxels}
cudaError_t launch_resin_spans(const vamrt_projector *p, cudaStream_t s);
cudaError_t launch_ver(const vamrt_projector *p, const void *dose, vamrt_dtype dt, const float *target,
                       long long *out3, cudaStream_t s);

// ramlak.cu (Radon-method baseline): rows x nu floats, in place allowed
cudaError_t launch_ramlak(const float *in, float *out, int64_t rows, int nu, double pixel_mm, int clamp,
                          cudaStream_t s);

// conv3d_tc.cu (tensor-core convolution of the warm-start network)
cudaError_t launch_conv3d_tc(const void *X, const void *Wt, const float *bias, void *Y, int out_f32, int D, int H,
                             int W, int Cin, int Cout, int taps, int relu, int *err, cudaStream_t s);

// conv3d_wgrad.cu: plan of the TMA-fed weight gradient (host only; false for shapes it
// cannot take)
struct WgradPlan {
    int Mtot, nmt, tpg, kp, KS, BX, nstage, cwA, cwB, slots, slot_bytes, per_sm, ncols, ngroups, nsplit, spb;
};
bool plan_wgrad_tma(int D, int H, int W, int Cin, int Cout, int taps, int sms, WgradPlan *pl);

// conv3d_wgrad_halo.cu: plan and launch of the weight gradient that stages each tile of X once
// for all 27 taps (host only; false for shapes it cannot take)
struct WgradHaloPlan {
    int TZ, TY, XB, cg, ngroups, Ct, nslices, nt, kp, slots, slot_bytes, x_bytes, ncols, nsplit, nx, ny, ntiles, seg, run,
        npos;
};
bool plan_wgrad_halo(int D, int H, int W, int Cin, int Cout, int taps, int sms, WgradHaloPlan *pl);
cudaError_t launch_wgrad_halo(const void *X, const void *dY, float *dW, int D, int H, int W, int Cin, int Cout,
                              const WgradHaloPlan &pl, int *err, cudaStream_t s);

// conv3d_wgrad.cu: the driver's tensor-map encoder (cuTensorMapEncodeTiled, through the
// runtime's driver entry point); NULL when the driver does not provide it
PFN_cuTensorMapEncodeTiled_v12000 tma_encoder();

// conv3d_march.cu (blocks walk along z; 3x3x3): plan (false for shapes it does not take), launch
struct ConvMarchPlan {
    int T, TY, mg, adv, ncols, cps, box_bytes, stage_bytes, ns, nslice, ry, nblk;
};
bool plan_conv3d_march(int D, int H, int W, int Cin, int Cout, int taps, int sms, ConvMarchPlan *pl);
cudaError_t launch_conv3d_march(const void *X, const void *Wt, const float *bias, void *Y, int out_f32, int D, int H,
                                int W, int Cin, int Cout, int relu, const ConvMarchPlan &pl, int *err, cudaStream_t s);

// conv3d_halo.cu (persistent halo-tile variant; W % 8 == 0).  launch returns
// cudaErrorNotSupported for shapes it does not take.
struct ConvHaloPlan {
    int TZ, TY, Nt, T, WP, PT, NX, rowtile, mg, adv, a_bytes, box_bytes, stage_bytes, ncols, ry, nslice, nitems;
};
bool plan_conv3d_halo(int D, int H, int W, int Cin, int Cout, int taps, int sms, ConvHaloPlan *pl);
cudaError_t launch_conv3d_halo(const void *X, const void *Wt, const float *bias, void *Y, int out_f32, int D, int H,
                               int W, int Cin, int Cout, int taps, int relu, int *err, cudaStream_t s);

cudaError_t launch_conv3d_wgrad_tc(const void *X, const void *dY, float *dW, int D, int H, int W, int Cin, int Cout,
                                   int taps, int *err, cudaStream_t s);

// nn_ops.cu
cudaError_t nn_resample(int op, const void *in, void *out, int D, int H, int W, int C, cudaStream_t s);
cudaError_t nn_concat(const void *a, int ca, const void *b, int cb, void *out, int64_t npos, int backward,
                      cudaStream_t s);
cudaError_t nn_relu_bwd(const void *y, void *dy, int64_t n, cudaStream_t s);
cudaError_t nn_bias_grad(const void *dy, float *db, int64_t npos, int C, cudaStream_t s);
cudaError_t nn_flip_weights(const void *w, void *wt, int cout, int taps, int cin, cudaStream_t s);
cudaError_t nn_adam(float *p, const float *g, float *m, float *v, void *pb, int64_t n, float lr, float b1, float b2,
                    float eps, int step, bool nonneg, cudaStream_t s);
cudaError_t nn_prepare_input(const float *proj, void *x, int A, int V, int U, int Dp, float scale, cudaStream_t s);
cudaError_t nn_head_mse(const float *z, int cz, const float *base, float in_scale, const float *target,
                        float target_scale, float *out, float out_scale, void *dz, int A, int V, int U, int Dp,
                        double *loss, cudaStream_t s);
cudaError_t nn_add(const void *x, void *y, int64_t n, cudaStream_t s);
cudaError_t nn_projected_step(float *g, const float *grad, float eta, int64_t n, cudaStream_t s);
cudaError_t nn_absmax(const float *x, int64_t n, float *out, cudaStream_t s);

// export.cu (8-bit export of projections, Sec. 2.7)
cudaError_t launch_export_u8(const vamrt_projector *p, const void *proj, vamrt_dtype dt, unsigned char *codes,
                             float *dequant, double *clip, cudaStream_t s);

// osmo.cu; ver3 (NULL: not wanted): the voxel error rate of the dose written, as launch_ver's out3
cudaError_t launch_sum(const vamrt_projector *p, const float *x, double *out, cudaStream_t s);
cudaError_t launch_osmo_step(const vamrt_projector *p, const float *target, float *model, void *dose,
                             vamrt_dtype dose_dt, const double *fsum, double *err_out, int residual, float alpha,
                             float mu, float *prev, long long *ver3, cudaStream_t s);

}  // namespace vamrt
