// ct_launch.h -- internal kernel launchers, one per projector.
// dir: 0 = forward (volume -> sinogram), 1 = back (sinogram -> volume).
// in_t / out_t: 0 f32, 1 f16, 2 bf16.  All launches are asynchronous on st.
#pragma once
#include <cuda_runtime.h>

#include "ct_types.h"

namespace ctp {

// Blocks of a cluster (at most 8, the portable size) that share a back's views:
// as many as give the chip two waves of resident warps, while every block keeps
// at least two of the npass rounds of views.  Depends on the geometry only.
inline int view_split(long long warps, int npass) {
    int s = 1;
    while (s < 8 && warps * s < 2LL * 152 * 32 && npass >= 4 * s) s *= 2;
    return s;
}

cudaError_t launch_sf(int dir, const CtGrid &g, const CtView *views, int in_t, const void *in,
                      int out_t, void *out, int batch, cudaStream_t st);
cudaError_t launch_dd(int dir, const CtGrid &g, const CtView *views, int in_t, const void *in,
                      int out_t, void *out, int batch, cudaStream_t st);
cudaError_t launch_dd_nc(int dir, const CtGrid &g, const CtView *views, int in_t, const void *in,
                         int out_t, void *out, int batch, cudaStream_t st);
// SF-TR (kind 0), DD (1) or SF-TT (2) with per-voxel footprints (any flat
// detector) of at most 8 cells by 4 rows (nc_footprint_fits); the DD and
// SF-TT back directions take the sinogram already scaled by each cell's
// factor (launch_sftt does that for SF-TT).
bool nc_footprint_fits(const CtGrid &g, int kind);
cudaError_t launch_sftt(int dir, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                        void *out, int batch, cudaStream_t st);
// SF-TT in circular flat 3D geometry on the streaming forward and the
// column-walk back (k_sf.cu), for transaxial footprints of at most 8 cells and
// axial ones of at most 4 rows; the back direction takes the FP32 sinogram
// already scaled by the per-cell amplitude (in_t ignored).
bool sftt_circ_fits(const CtGrid &g);
cudaError_t launch_sftt_circ(int dir, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                             void *out, int batch, cudaStream_t st);
cudaError_t launch_nc(int kind, int dir, const CtGrid &g, const CtView *views, int in_t, const void *in,
                      int out_t, void *out, int batch, cudaStream_t st);
// 2D fan beam (k_fan.cu): every projector, dir 0 forward, 1 back (DD and SF-TT
// take the sinogram already scaled by each cell's factor), 2 the recon-mode
// back of SF, DD and voxel-driven.  fan_fits: 2D, and forward footprints of at
// most 8 cells (wider ones take the general forward of k_sf.cu).
enum FanKind { FAN_SF = 0, FAN_DD = 1, FAN_TT = 2, FAN_VOX = 3, FAN_RAY = 4 };
bool fan_fits(const CtGrid &g, int kind, int dir);
cudaError_t launch_fan(int kind, int dir, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                       void *out, int batch, cudaStream_t st);
// circular cone-beam back (k_circ_back.cuh) of SF-TR, DD (from the scaled FP32
// sinogram) and voxel-driven, recon: in recon mode; for footprints of at most
// 8 cells and voxels shorter than 8 rows on a detector of at least 8 cells
enum BackKind { BK_SF = 0, BK_DD = 1, BK_VOX = 2 };
bool circ_back_fits(const CtGrid &g, int kind);
cudaError_t launch_circ_back(int kind, bool recon, const CtGrid &g, const CtView *views, int in_t, const void *in,
                             int out_t, void *out, int batch, cudaStream_t st);
// circular cone-beam forward (k_circ_fwd.cuh) of SF-TR, DD and voxel-driven
// (kind: BackKind) for footprints of at most 8 cells
size_t circ_fwd_workspace(const CtGrid &g, int batch, int elem_bytes);
bool circ_fwd_fits(const CtGrid &g, int kind, int batch);
cudaError_t launch_circ_fwd(int kind, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                            void *out, int batch, cudaStream_t st);
// voxel-driven forward in circular geometry (that kernel, or k_sf.cu without the copy)
cudaError_t launch_vx_fwd_circ(const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                               void *out, int batch, cudaStream_t st);
// recon mode (FBP): the pre-weighted ramp filter of each detector row, and the
// depth-weighted voxel-driven backprojection of the filtered projections
cudaError_t launch_ramp_filter(const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                               void *out, int batch, cudaStream_t st);
// recon mode with the normalised DD (dd = 1) or SF-TR (dd = 0) footprints;
// non-circular footprints beyond 8 x 4 give cudaErrorNotSupported
cudaError_t launch_recon_fp(int dd, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                            void *out, int batch, cudaStream_t st);
cudaError_t launch_nc_recon(int dd, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                            void *out, int batch, cudaStream_t st);
cudaError_t launch_voxel_recon(const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                               void *out, int batch, cudaStream_t st);
cudaError_t launch_voxel(int dir, const CtGrid &g, const CtView *views, int in_t, const void *in,
                         int out_t, void *out, int batch, cudaStream_t st);
cudaError_t launch_ray(int dir, const CtGrid &g, const CtView *views, int in_t, const void *in,
                       int out_t, void *out, int batch, cudaStream_t st);

cudaError_t launch_dd_back_scratch(const CtGrid &g, const CtView *views, int in_t, const void *in,
                                   int out_t, void *out, int batch, float *scratch, cudaStream_t st);

// xZ[b][j][i][k] = x[b][k][j][i] for elements of elem_bytes (2 or 4) bytes,
// columns nzp elements apart, zero from nz on
cudaError_t zmajor_copy(int elem_bytes, const void *x, void *xZ, int nx, int ny, int nz, int nzp, int batch,
                        cudaStream_t st);
// slices of the circular forwards' copies of the volume: nz rounded up to four,
// or 0: no copy (fan beam, non-circular, and volumes of fewer than four slices,
// which the padding would double and more)
inline int zmajor_pitch(const CtGrid &g) {
    return g.is2d || g.variant == GEO_NONCIRC_FLAT || g.nz < 4 ? 0 : (g.nz + 3) & ~3;
}
// Volumes of at most this many voxels (32^3) go without reordered copies, which would
// cost the smallest calls an allocation and a launch
constexpr long long kCopyVoxels = 32768;
inline bool copies_pay(const CtGrid &g, int batch) { return (long long)g.nx * g.ny * g.nz * batch > kCopyVoxels; }
// the ray-driven forward's copy
inline bool ray_copies(const CtGrid &g, int batch) { return g.ray_x && copies_pay(g, batch); }
// the copy's grid (rows and batch items are its y and z)
inline bool zmajor_copy_fits(const CtGrid &g, int batch) { return copies_pay(g, batch) && batch <= 65535 && g.ny <= 65535; }

// Stream-ordered scratch from a library-owned pool on the current device
// (memory is kept in the pool between calls, so steady-state calls do not
// reach the driver's allocator).
cudaError_t workspace_alloc(void **p, size_t bytes, cudaStream_t st);
// the same for a reordered copy of the volume, which a forward can do without
inline cudaError_t workspace_alloc_copy(void **p, size_t bytes, const CtGrid &g, cudaStream_t st) {
    return bytes > g.copy_max ? cudaErrorMemoryAllocation : workspace_alloc(p, bytes, st);
}
cudaError_t workspace_free(void *p, cudaStream_t st);
// release threshold of the current device's pool (and a trim to it)
cudaError_t workspace_set_limit(size_t bytes);
// bytes the pool holds from the device now, and the high-water mark of the
// bytes in use (reset to zero when reset_high is set)
cudaError_t workspace_usage(size_t *reserved, size_t *used_high, int reset_high);

}  // namespace ctp
