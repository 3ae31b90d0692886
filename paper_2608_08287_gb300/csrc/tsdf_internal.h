// Internal host-side definitions shared by the host runtime files
// (tsdf_api.cu, tsdf_batch.cu). Not part of the C ABI.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

#include "tsdf.h"
#include "tsdf_device.cuh"
#include "tsdf_launch.h"

namespace tsdf {

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

// Byte offsets of a volume's sections inside its one allocation.
struct Offsets {
  size_t table, coords, twrg, blue, total;
};

inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }

tsdf_status from_cuda(cudaError_t e);
tsdf_status decode_err(uint32_t err);

// Threads per point of the fused tile kernel chosen for work of `tiles`
// 16 x 16 pixel tiles running alone on the GPU (one frame, or all frames of a
// batch launched together), where the split walk exists (fuse mode 2, the
// default probe load): 4 up to one tile per SM, 2 up to eight (two rounds of
// resident CTAs at one thread per point), else 1. A split walk gives a small
// frame more warps and shorter ones; a frame of several rounds has warps enough
// and only pays for the second ray per point. One frame into a mapped volume at
// 5 mm, L2 cold, us at 1 / 2 / 4 threads a point, half band 4 and then 8:
//   100x75   18.4 / 12.3 / 10.9   35.2 / 16.4 / 12.7
//   160x120  16.4 / 12.3 / 12.3   28.7 / 16.4 / 16.1
//   240x180  17.7 / 14.4 / 14.3   30.3 / 22.5 / 20.5
//   320x240  18.6 / 18.4 / 18.4   30.7 / 28.7 / 26.6
//   480x360  30.0 / 27.8 / 30.0   51.2 / 45.3 / 45.1
//   640x480  41.0 / 41.0 / 47.1   72.2 / 66.4 / 71.7
//   960x720  75.9 / 84.0 / 98.3   138 / 133 / 150
//   1280x720 106 / 115 / 133      183 / 188 / 201
// The lines lie where half band 4 changes hands; at half band 2 one thread is
// already as fast at 480x360 (20.5 and 20.5) and faster at 640x480 (26.8 and
// 28.7).
int auto_threads_per_point(int fuse_mode, int probe_load, int sm_count, long long tiles);
// The same for stage B's tile kernel: one above four tiles per SM at half bands
// 1 and 2, where a second ray a point costs more than the shorter walks give.
// Both stages of a mapped frame, one of many, us with 1 / 2 threads in stage B:
// 640x480 at 5 mm, half band 1 38.3 / 44.6, 2 48.2 / 52.1, 3 61.7 / 60.1, 4 70.3 /
// 67.7; at 10 mm 30.8 / 41.4, 36.0 / 43.7, 45.2 / 49.1, 50.6 / 52.9; 480x360 at 5
// mm 28.7 / 31.7, 37.0 / 38.0, 48.4 / 46.0, 55.9 / 52.2.
int auto_threads_stage_b(int half_band, int sm_count, long long tiles);
inline long long tiles_of_frame(int width, int height) {
  return static_cast<long long>((width + 15) / 16) * ((height + 15) / 16);
}

}  // namespace tsdf

struct tsdf_volume {
  int device = 0;
  int sm_count = 0;
  float voxel = 0.0f, trunc = 0.0f;
  int half_band = 0;
  uint32_t slots = 0, pool = 0;
  void* mem = nullptr;
  size_t bytes = 0;
  bool owns = false;
  tsdf::Offsets off{};
  tsdf::VolumeArgs va{};
  bool poisoned = false;
  bool dirty = false;          // something was fused since creation or the last reset
  uint32_t* pinned = nullptr;  // {count, err}
  int probe_load = tsdf::kLoadCached;
  int allocate_mode = 1;
  int integrate_mode = tsdf::kIntegrateAuto;
  int fuse_mode = 2;
  int threads_per_point = 0;  // of the fused tile kernel (0: chosen per frame)
  int threads = 256;
  void* stage = nullptr;
  size_t stage_bytes = 0;
  // streaming host input (tsdf_fuse_frames_host), made on first use: two
  // staging slots, a copy stream, slot filled / slot free events, and pinned
  // per-frame error words
  void* stream_stage = nullptr;
  size_t stream_slot_bytes = 0;
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t ev_copied[2] = {nullptr, nullptr};
  cudaEvent_t ev_free[2] = {nullptr, nullptr};
  uint32_t* err_words = nullptr;      // pinned, one word per frame of a call
  uint32_t* err_gathered = nullptr;   // pinned, the words gathered on the device
  uint32_t* err_dev = nullptr;        // device, where they are gathered
  int err_capacity = 0;
};

namespace tsdf {
// Validate a frame and build its kernel arguments (no CUDA call).
tsdf_status make_frame(const tsdf_volume* v, const float* depth, int w, int h,
                       const tsdf_intrinsics* intr, const tsdf_pose* pose, const uint8_t* rgb,
                       FrameArgs* f);

// Stage B's mode of a batch as at its creation (no option value names it).
void unset_integrate_mode(tsdf_batch* batch);
}  // namespace tsdf
