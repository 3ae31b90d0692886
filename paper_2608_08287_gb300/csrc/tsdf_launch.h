// Internal interface between the host runtime (tsdf_api.cu) and the kernels
// (tsdf_kernels.cu). Not part of the C ABI.
#pragma once

#include <cuda_runtime.h>

#include "tsdf_device.cuh"

namespace tsdf {

// Launch accounting: every kernel launch the library enqueues is counted.
void note_launch();

// Stage A: mode 0 = the paper's protocol, 1 = tile kernel, 2 = warp kernel.
cudaError_t launch_allocate(const FrameArgs& f, const VolumeArgs& vol, int probe_load, int mode,
                            cudaStream_t s);
// Stage B: mode 0 = per-thread lookups, 1 = warp kernel, 2 = tile kernel with
// one thread a point, or two for threads_per_point above 1.
cudaError_t launch_integrate(const FrameArgs& f, const VolumeArgs& vol, int mode,
                             int threads_per_point, cudaStream_t s);
// Stage B's mode where none has been set.
constexpr int kIntegrateAuto = -1;
// The mode of launch_integrate for a set (or unset) integrate mode: one that
// was set is taken as it is; unset, the paper's update beside the paper's
// protocol (allocate mode 0), and the tile kernel otherwise. The tile kernel
// looks a tile's blocks up once and adds its sums in bursts. Stage B of a mapped
// 640x480 frame at 5 mm, us by per-thread lookups and by the tile kernel at table
// loads 0.5 / 0.6 / 0.75 / 0.88: 47.5 and 40.6 / 57 and 41 / 88 and 41 / 655 and
// 42; 1280x720 73 and 78 / 86 and 78 / 154 and 79 / 1,517 and 80. Below a load of
// a half per-thread lookups are faster by up to 15 % for coarse voxels and narrow
// bands, which is not worth what they lose above it.
inline int stage_b_kernel(int allocate_mode, int integrate_mode) {
  if (integrate_mode != kIntegrateAuto) return integrate_mode;
  return allocate_mode == 0 ? 0 : 2;
}
// The fused path. threads_per_point > 1 (2, 4 or 8) takes the fused tile
// kernel with each point's walk split over that many threads; it exists for
// fuse mode 2 and the default probe load (cudaErrorInvalidValue otherwise).
cudaError_t launch_fused(const FrameArgs& f, const VolumeArgs& vol, int probe_load, int mode,
                         int threads_per_point, cudaStream_t s);
// Stage B, tile strategy (integrate mode 2): the fused tile kernel's steps
// with step 2 looking the tile's blocks up instead of inserting them.
cudaError_t launch_integrate_tile(const FrameArgs& f, const VolumeArgs& vol,
                                  int threads_per_point, cudaStream_t s);
// The split-walk fused tile kernels (their own translation unit).
cudaError_t launch_fused_split(const FrameArgs& f, const VolumeArgs& vol, int threads_per_point,
                               cudaStream_t s);
// Batched launches (all frames of a session table): allocate + integrate, or
// the fused kernel. factor caps the resident CTAs per SM (0 = as many as fit).
// grid_limit > 0 caps the grid (e.g. at the batch's tile count). all_m4: every
// frame has half band 4 or less (selects the tile kernel whose walk is one
// round).
// stages (fuse mode 0): 1 = stage A only, 2 = stage B only, 3 = both.
cudaError_t launch_batch(const BatchHeader* table, int probe_load, int allocate_mode,
                         int integrate_mode, int fuse_mode, int factor, int grid_limit,
                         bool all_m4, int stages, cudaStream_t s);
cudaError_t launch_batch_status(const BatchHeader* table, unsigned* out, cudaStream_t s);
// Means of n blocks into out (n x 5 x 512); block j is pool block list[j], or
// j when list is null.
cudaError_t launch_export(const VolumeArgs& vol, float* out, unsigned int n,
                          const unsigned int* list, cudaStream_t s);
// Slot-index volumes: occupied slots in slot order (list) and their block
// coordinates, at most cap of them; *found = occupied slots.
cudaError_t launch_slot_list(const VolumeArgs& vol, unsigned int* list, int32_t* coords,
                             unsigned int cap, unsigned int* found, cudaStream_t s);
// Zero the used pool blocks (before the table is cleared).
cudaError_t launch_clear_used(const VolumeArgs& vol, int sm_count, cudaStream_t s);
// Marching-tetrahedra surface of the volume: triangles (9 floats each) and
// cell records (4 int32 each), either may be null; writes at most capacity of
// them and adds the total to *counter (which the caller zeroes first).
cudaError_t launch_extract(const VolumeArgs& vol, float v, float* tris, int32_t* cells,
                           unsigned int capacity, unsigned int* counter, int sm_count,
                           cudaStream_t s);
// Accumulate table occupancy, probe lengths and the pool's total weight into
// *out (which the caller zeroes first).
cudaError_t launch_table_stats(const VolumeArgs& vol, TableStatsDev* out, int sm_count,
                               cudaStream_t s);

}  // namespace tsdf
