// The fused tile kernel with each point's band walk split over 2, 4 or 8
// threads (tile_body, TPP > 1), for the default probe load, and stage B's tile
// kernel (Op = kOpIntegrate). A translation unit of its own so that it
// compiles in parallel with the other kernels.
#include "tsdf_device.cuh"
#include "tsdf_launch.h"
#include "tsdf_tile.cuh"

namespace tsdf {

cudaError_t launch_integrate_tile(const FrameArgs& f, const VolumeArgs& vol,
                                  int threads_per_point, cudaStream_t s) {
  if (threads_per_point > 1) return launch_tile<kOpIntegrate, kLoadCached, 2>(f, vol, s);
  return launch_tile<kOpIntegrate, kLoadCached, 1>(f, vol, s);
}

cudaError_t launch_fused_split(const FrameArgs& f, const VolumeArgs& vol, int threads_per_point,
                               cudaStream_t s) {
  cudaError_t e;
  switch (threads_per_point) {
    case 2: e = launch_tile<kOpFused, kLoadCached, 2>(f, vol, s); break;
    case 4: e = launch_tile<kOpFused, kLoadCached, 4>(f, vol, s); break;
    case 8: e = launch_tile<kOpFused, kLoadCached, 8>(f, vol, s); break;
    default: return cudaErrorInvalidValue;
  }
  if (e == cudaSuccess) note_launch();
  return e;
}

}  // namespace tsdf
