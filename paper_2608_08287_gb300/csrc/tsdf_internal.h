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
// default probe load): 4 up to one tile per SM (where a wide band's walk is
// the frame's time: 100x75 at half band 8 takes 17.7 us against 26.9 with 2),
// 2 up to eight (two rounds of resident CTAs
// at one thread per point), else 1. A split walk gives a small frame more
// warps and shorter ones; a frame of several rounds has warps enough and only
// pays for the second ray per point. One frame into a mapped volume, half band
// 4, us at 1 / 2 / 4 threads a point: 160x120 with its status 33.3 / 27.3 /
// 27.2, 240x180 15.7 / 12.2 / 13.6, 320x240 30.9 / 27.9 / 26.2, 480x360 23.1 /
// 21.9 / 28.1, 640x480 (1,200 tiles) 52.1 / 49.3 / 54.1, 960x720 72.8 / 73.0 /
// 94.3, 1280x720 85.2 / 90.1 / 128.7.
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
