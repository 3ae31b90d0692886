// The tile machinery shared by the kernel translation units: launch shape
// constants, the block directory of a pixel tile, the point walk that fills
// it, the resolution of its blocks in the volume's table, and the tile kernel
// of stage A, stage B and the fused path (paper Section 2.2; its phases are
// described at tile_body).
#pragma once

#include <cstdint>

#include "tsdf_device.cuh"

namespace tsdf {

constexpr int kThreads = 256;
constexpr int kTile = 16;
constexpr int kSetSlots = 2048;    // allocate_kernel: per-CTA key set (16 KB)

// Pixel of this thread in tile (tx, ty): a tile is 16 pixels wide and
// blockDim.x / 16 rows high; warp w covers the 8x4 patch (w & 1, w >> 1).
__device__ __forceinline__ void tile_pixel_at(int tx, int ty, int& u, int& v) {
  const int w = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  u = tx * kTile + (w & 1) * 8 + (lane & 7);
  v = ty * static_cast<int>(blockDim.x >> 4) + (w >> 1) * 4 + (lane >> 3);
}

__device__ __forceinline__ void tile_pixel(int tile, int tiles_x, int& u, int& v) {
  tile_pixel_at(tile % tiles_x, tile / tiles_x, u, v);
}

// Insert into the CTA's shared-memory key set; false if the set is full.
__device__ __forceinline__ bool set_insert(unsigned long long* set, unsigned long long key,
                                           unsigned int h) {
  for (int i = 0; i < kSetSlots; ++i) {
    const unsigned int s = (h + i) & (kSetSlots - 1);
    const unsigned long long prev = atomicCAS(&set[s], kEmptyKey, key);
    if (prev == kEmptyKey || prev == key) return true;
  }
  return false;
}

// Walk state of one point for the generic loop: the last two in-range voxels.
struct WalkDedupe {
  int ax = INT_MIN, ay = 0, az = 0, bx = INT_MIN, by = 0, bz = 0;
  __device__ __forceinline__ bool seen_then_push(int x, int y, int z) {
    if ((x == ax && y == ay && z == az) || (x == bx && y == by && z == bz)) return true;
    bx = ax; by = ay; bz = az;
    ax = x; ay = y; az = z;
    return false;
  }
};

__device__ __forceinline__ unsigned long long block_key_of(int gx, int gy, int gz) {
  return pack_key(gx >> 3, gy >> 3, gz >> 3);
}

// ----------------------------------------------------------------------------
// stage A, the paper's protocol (Listing 1 per sample, waits for publication)
// ----------------------------------------------------------------------------
template <int P>
__global__ void __launch_bounds__(kThreads)
    allocate_kernel(const __grid_constant__ FrameArgs f, const __grid_constant__ VolumeArgs vol,
                    int tiles_x) {
  __shared__ unsigned long long s_set[kSetSlots];
  __shared__ unsigned int s_err;
  if (threadIdx.x == 0) s_err = load_err_volatile(vol.hdr);
  for (int i = threadIdx.x; i < kSetSlots; i += kThreads) s_set[i] = kEmptyKey;
  __syncthreads();
  if (s_err) return;  // poisoned volume: do nothing

  int u, v;
  tile_pixel(blockIdx.x, tiles_x, u, v);
  Ray r;
  bool valid = false;
  if (u < f.W && v < f.H)
    valid = make_ray(f, u, v, load_depth(f, static_cast<long long>(v) * f.W + u), r);
  const int lane = threadIdx.x & 31;
  unsigned long long last_key = kEmptyKey;
  WalkDedupe walk;
  for (int k = 0; k <= 2 * f.M; ++k) {
    bool cand = false;
    unsigned long long key = kEmptyKey;
    int bx = 0, by = 0, bz = 0;
    if (valid) {
      int gx, gy, gz;
      float zc;
      if (sample_voxel(f, r, k, gx, gy, gz) && !walk.seen_then_push(gx, gy, gz) &&
          voxel_test(f, gx, gy, gz, zc)) {
        bx = gx >> 3;
        by = gy >> 3;
        bz = gz >> 3;
        key = pack_key(bx, by, bz);
        if (key != last_key) {
          cand = true;
          last_key = key;
        }
      }
    }
    // warp-level dedupe before any compare-exchange
    const unsigned int m = __ballot_sync(0xffffffffu, cand);
    if (cand) {
      const unsigned int peers = __match_any_sync(m, key);
      if (lane == __ffs(peers) - 1) {
        if (!set_insert(s_set, key, hash_block(bx, by, bz))) insert_block<P>(vol, key, bx, by, bz);
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kSetSlots; i += kThreads) {
    const unsigned long long key = s_set[i];
    if (key != kEmptyKey) {
      int bx, by, bz;
      unpack_key(key, bx, by, bz);
      insert_block<P>(vol, key, bx, by, bz);
    }
  }
}

// One-entry cache of a resolved block.
struct BlockCacheT {
  unsigned long long key = kEmptyKey;
  int idx = -1;
};

enum TileOp { kOpAllocate = 0, kOpIntegrate = 1, kOpFused = 2 };

// Resolve one key on its own (paths that could not use a tile's directory or a
// warp's list: rare, so kept out of line to keep the kernels' hot code small).
template <int Op, int P>
__device__ __noinline__ int resolve_single(const VolumeArgs& vol, unsigned long long key) {
  int bx, by, bz;
  unpack_key(key, bx, by, bz);
  if (Op == kOpAllocate) return insert_block<P, false>(vol, key, bx, by, bz);
  if (Op == kOpFused) return insert_block<P, true>(vol, key, bx, by, bz);
  return resolve_for_update(vol, lookup_block(vol, key, bx, by, bz));
}

// Five sums of one accepted voxel, added straight to the pool.
__device__ __forceinline__ void add_voxel_direct(const VolumeArgs& vol, int idx, int l, float t,
                                                 bool colour, float cr, float cg, float cb) {
  if (idx < 0) return;
  add_contribution(vol, static_cast<size_t>(idx) * kBlockVoxels + l, t, colour,
                   cr, cg, cb);
}

// Pixel of this thread when TPP consecutive threads share one point: a tile
// is 16 pixels wide and 8 / TPP high, and each of its four warps covers a
// patch of 4 pixels' width and that height.
template <int TPP>
__device__ __forceinline__ void tile_pixel_shared(int tx, int ty, int& u, int& v) {
  constexpr int rows = 8 / TPP;
  static_assert(kThreads / 2 == kTile * rows * TPP, "four warps of 32 / TPP points");
  const int w = static_cast<int>(threadIdx.x >> 5), p = static_cast<int>(threadIdx.x & 31u) / TPP;
  u = tx * kTile + w * 4 + (p & 3);
  v = ty * rows + (p >> 2);
}

// Threads of a tile kernel's CTA. With one thread a point 128 and 256 measured
// alike when they were chosen (640x480: 51.6 and 52.1 us; 1280x720 at half band
// 8: 125 and 120 us); a split walk was faster with the smaller CTA (640x480: 49.3
// against 50.0 us, 1280x720: 90 against 96 us), whose barriers hold fewer warps
// back.
template <int TPP>
__host__ __device__ constexpr int tile_threads() {
  return TPP == 1 ? kThreads : kThreads / 2;
}

// Pixel rows of one tile of a kernel whose points have TPP threads each.
template <int TPP>
constexpr int tile_rows() {
  return tile_threads<TPP>() / (kTile * TPP);
}

// ----------------------------------------------------------------------------
// the tile kernel: stage A, stage B or both for one tile of pixels
// ----------------------------------------------------------------------------
// The distinct blocks of a tile live in a small shared-memory directory, an
// open-addressed set of 32-bit tags (a block's offset from the tile's base
// block); the first thread to add a block appends its slot to a list.
template <int D>
struct TileShared {
  static constexpr int kSlots = D;
  alignas(16) unsigned dir[D];         // tags
  alignas(16) int idx[D];              // their pool indices
  alignas(16) unsigned short list[D];  // occupied slots in order of arrival
  alignas(8) unsigned long long base;  // key of the tile's base block
  alignas(16) unsigned short todo[D];  // slots whose blocks were claimed, or are waited for
  int n, n_open;                       // occupied slots; new blocks that their home slots did not settle
  int won, pending;                    // blocks claimed in this round, and waited for
  unsigned first;                      // pool index of the first of the claimed
  unsigned err;
};

// Directory slots, four or more a point: a 256-point tile of a 640x480 frame at
// 5 mm has 24 blocks, at most 62, but where the voxels are finer than the
// pixels nearly every sample has a block of its own (160x120 at 5 mm: up to 300
// at half band 4, more for wider bands). Points whose blocks find no room are
// resolved on their own, one by one, which is slow: when these were introduced,
// a 100x75 frame at 5 mm and half band 8 took 33.3 us with half as many slots and
// 26.9 us with these (two threads a point).
template <int TPP>
using TileTables = TileShared<TPP == 1 ? 1024 : 512>;

constexpr unsigned kNoTag = 0xFFFFFFFFu;       // (no tag has all fields full)
constexpr unsigned kSlotNone = 0x1FFFFFu;      // block outside the directory
constexpr int kGroup = 3;                      // samples whose depth gathers are in flight together

// floor(x) by one addition rounded down: 1.5 * 2^23 + floor(x), exact for
// |x| <= 2^22, whose low mantissa bits are the integer. It replaces a floor,
// a conversion to integer and one back, all on the quarter-rate pipe.
constexpr float kFloorMagic = 12582912.0f;     // 1.5 * 2^23
constexpr int kMagicBits = 0x4B400000;         // its bits

__device__ __forceinline__ float floor_magic(float x) { return __fadd_rd(x, kFloorMagic); }

// Biased block coordinate (pack_key's field) of a voxel coordinate in
// floor_magic bits.
__device__ __forceinline__ unsigned magic_block(int bits) {
  return static_cast<unsigned>(bits - (kMagicBits - 8 * kKeyBias)) >> 3;
}

// The three voxel coordinates of a sample in one word, modulo 2^32: minus the
// point's packed base they are 10-bit offsets (512 at the base), since a band
// stays within kPackedReach voxels of its point (packed_walk_limit). Two
// samples of a point have the same voxel exactly when their words are equal.
__device__ __forceinline__ unsigned pack_magic(float tx, float ty, float tz) {
  return __float_as_uint(tx) + (__float_as_uint(ty) << 10) + (__float_as_uint(tz) << 20);
}

// Block fields of a packed voxel (after >> 3; never all zero).
constexpr unsigned kPackBlockBits = 0x07F1FC7Fu;

// The packed base of a point whose block-aligned voxel is (ox, oy, oz)
// in floor_magic bits.
__device__ __forceinline__ unsigned packed_base(int ox, int oy, int oz) {
  return static_cast<unsigned>(ox - 512) + (static_cast<unsigned>(oy - 512) << 10) +
         (static_cast<unsigned>(oz - 512) << 20);
}

// Whether every sample of a point's band lies in floor_magic's range and fits
// a packed word, and the block-aligned voxel of the point. (walk_limit is
// negative where the pose stretches the band beyond kPackedReach.)
__device__ __forceinline__ bool band_in_range(const FrameArgs& f, const Ray& r, int& ox, int& oy,
                                              int& oz) {
  const float ax = __fmul_rn(r.px, f.inv_v);
  const float ay = __fmul_rn(r.py, f.inv_v);
  const float az = __fmul_rn(r.pz, f.inv_v);
  ox = __float_as_int(floor_magic(ax)) & ~7;
  oy = __float_as_int(floor_magic(ay)) & ~7;
  oz = __float_as_int(floor_magic(az)) & ~7;
  return fabsf(ax) < f.walk_limit && fabsf(ay) < f.walk_limit && fabsf(az) < f.walk_limit;
}

// Local index of a packed voxel: its three 3-bit fields at bits 0, 10 and 20
// brought together at bit 14 by one multiplication (no two terms overlap).
__device__ __forceinline__ unsigned pack_local(unsigned p) {
  return ((p & 0x00701C07u) * ((1u << 14) + (1u << 7) + 1u) >> 14) & 511u;
}

// Key of a tag: block offsets biased by 512, 512 and 2048 from the base block.
__device__ __forceinline__ unsigned long long tag_key(unsigned long long base, unsigned tag) {
  return base + (static_cast<unsigned long long>(static_cast<long long>(tag & 1023u) - 512) << 42) +
         (static_cast<unsigned long long>(static_cast<long long>((tag >> 10) & 1023u) - 512) << 21) +
         static_cast<unsigned long long>(static_cast<long long>(tag >> 20) - 2048);
}

// voxel_project for a voxel in floor_magic form: the centre's camera depth zc
// and the row-major index of its nearest pixel, -1 when it is not `wanted`,
// behind the camera or outside the image. The pixel's floor takes the same
// form; read as an unsigned number it is beyond any image size for every
// input outside [0, 2^22), infinities and NaN among them.
__device__ __forceinline__ int project_magic(const FrameArgs& f, float tx, float ty, float tz,
                                             bool wanted, float& zc) {
  const float gx = __fsub_rn(tx, kFloorMagic), gy = __fsub_rn(ty, kFloorMagic),
              gz = __fsub_rn(tz, kFloorMagic);
  const float cz = __fmaf_rn(f.A[8], gz, __fmaf_rn(f.A[7], gy, __fmaf_rn(f.A[6], gx, f.b[2])));
  const float cx = __fmaf_rn(f.A[2], gz, __fmaf_rn(f.A[1], gy, __fmaf_rn(f.A[0], gx, f.b[0])));
  const float cy = __fmaf_rn(f.A[5], gz, __fmaf_rn(f.A[4], gy, __fmaf_rn(f.A[3], gx, f.b[1])));
  zc = cz;
  const float iz = __frcp_rn(cz);
  const int iu = __float_as_int(floor_magic(
                     __fadd_rn(__fmaf_rn(f.fx, __fmul_rn(cx, iz), f.cx), 0.5f))) - kMagicBits;
  const int iv = __float_as_int(floor_magic(
                     __fadd_rn(__fmaf_rn(f.fy, __fmul_rn(cy, iz), f.cy), 0.5f))) - kMagicBits;
  const bool ok = wanted && cz > 0.0f && static_cast<unsigned>(iu) < static_cast<unsigned>(f.W) &&
                  static_cast<unsigned>(iv) < static_cast<unsigned>(f.H);
  return ok ? iv * f.W + iu : -1;
}

// Directory slots of the tags of the lanes that `want` one, added if absent;
// kSlotNone when the directory is full. Every lane of the warp calls it. The
// first probe, which nearly always finds the block, has no branch; the loop
// is kept converged, since a diverged warp repeats what follows it.
template <class Tables>
__device__ __forceinline__ void dir_find(Tables& S, unsigned tag, bool want, unsigned& slot) {
  constexpr int D = Tables::kSlots;
  unsigned s = (tag * 0x9E3779B1u) >> (32 - __builtin_ctz(D));
  bool pend = want && *reinterpret_cast<volatile unsigned*>(&S.dir[s]) != tag;
  slot = want ? s : slot;
  int left = D;
  while (__any_sync(0xffffffffu, pend)) {
    if (pend) {
      unsigned k = *reinterpret_cast<volatile unsigned*>(&S.dir[s]);
      if (k == kNoTag) {
        k = atomicCAS(&S.dir[s], kNoTag, tag);
        if (k == kNoTag) {
          S.list[atomicAdd(&S.n, 1)] = static_cast<unsigned short>(s);
          k = tag;
        }
      }
      if (k == tag) {
        slot = s;
        pend = false;
      } else if (--left == 0) {
        slot = kSlotNone;
        pend = false;
      }
      s = (s + 1) & (D - 1);
    }
  }
}

// The outcome of a key that has been probed for: its pool index (>= 0), one of
// these with the table slot it was settled at, or another negative value when
// it has none (stage B: absent; else the table is full).
constexpr int kPending = -4;  // present, its winner has not published the index yet
constexpr int kWon = -5;      // claimed here, its index not taken yet

// Probes for up to four keys a warp, eight lanes each (every lane of a group
// holds the group's key; `has` is the same in all eight). A probe reads eight
// consecutive slots, and the group takes the first that holds the key or is
// empty: the slot a sequential probe (Listing 1, Section 2.3) would stop at,
// since an occupied slot never changes. A slot read as EMPTY is settled by the
// compare-exchange; when that is lost to another key the group goes on to its
// next candidate. Op: kOpFused and kOpAllocate insert, kOpIntegrate looks up.
// The lane that settles a key returns the outcome, every other lane -1 or
// kAbsent.
//
// What bounds it is round trips to the table, not lanes: a tile has 10-50
// blocks, and the CTA waits for the slowest. One round trip settles a chain of
// up to eight slots; spread over all warps of the CTA, four keys each. A chain
// that goes on is scanned by the whole warp, 128 slots a step (four loads in
// flight a lane): a 640x480 frame at load 0.88 took 118 us with eight slots a
// step throughout, 55 with these.
template <int Op, int P>
__device__ __forceinline__ int group_resolve(const VolumeArgs& vol, unsigned long long key, bool has,
                                            unsigned& at) {
  const unsigned lane = threadIdx.x & 31u, gl = lane & 7u, shift = lane & 24u;
  int bx, by, bz;
  unpack_key(key, bx, by, bz);
  unsigned s0 = hash_block(bx, by, bz) & vol.mask;
  unsigned probe = 0;
  bool todo = has;
  int result = Op == kOpIntegrate ? kAbsent : -1;
  while (__any_sync(0xffffffffu, todo)) {
    const unsigned left = vol.probe_limit - probe;
    const bool reads = todo && gl < left;
    const unsigned s = (s0 + gl) & vol.mask;
    Entry* e = vol.table + s;
    unsigned long long k = 0;
    int idx = -1;
    if (reads && slot_ok(vol, s)) load_entry<P>(e, k, idx);
    unsigned m = (__ballot_sync(0xffffffffu, reads && (k == key || k == kEmptyKey)) >> shift) & 255u;
    bool won = false;
    // the candidates in order, until one settles it
    while (__any_sync(0xffffffffu, todo && m)) {
      const unsigned c = m ? static_cast<unsigned>(__ffs(m) - 1) : 0u;
      int out = 0;   // 0: another key came first, 1: settled
      if (todo && m && gl == c) {
        if (k == kEmptyKey) {
          if (Op == kOpIntegrate) {
            out = 1;
          } else {
            const unsigned long long prev = atomicCAS(&e->key, kEmptyKey, key);
            if (prev == kEmptyKey) {
              won = true;
              out = 1;
            } else {
              k = prev;
              idx = kUnpublished;
            }
          }
        }
        if (k == key) {
          out = 1;
          if (vol.slot_index)
            result = static_cast<int>(s);
          else if (Op == kOpFused && idx == kUnpublished)
            result = kPending;
          else
            result = idx;
        }
      }
      out = __shfl_sync(0xffffffffu, out, static_cast<int>(c), 8);
      if (todo && m) {
        m &= m - 1u;
        if (out) {
          todo = false;
          m = 0;
        }
      }
    }
    if (Op != kOpIntegrate && vol.slot_index) {
      // the slot is the index: the blocks only have to be counted
      const unsigned wins = __ballot_sync(0xffffffffu, won);
      if (wins && lane == static_cast<unsigned>(__ffs(wins) - 1))
        red_add_u32(&vol.hdr->count, __popc(wins));
      if (won) result = static_cast<int>(s);
    } else if (Op != kOpIntegrate && won) {
      result = kWon;
    }
    if (todo) {
      s0 = (s0 + 8) & vol.mask;
      probe += 8;
      if (probe >= vol.probe_limit) {
        if (Op != kOpIntegrate && gl == 0) probe_exhausted(vol);
        todo = false;
      }
    }
    // a chain that goes on past its first slots: the whole warp reads 128 of
    // them at a time, one group's chain after another's
    unsigned longs = __ballot_sync(0xffffffffu, todo && gl == 0);
    while (longs) {
      const int L = __ffs(longs) - 1;
      longs &= longs - 1;
      const unsigned long long lkey = __shfl_sync(0xffffffffu, key, L);
      unsigned ls = __shfl_sync(0xffffffffu, s0, L);
      unsigned lprobe = __shfl_sync(0xffffffffu, probe, L);
      bool found = false, stopped = false;
      for (unsigned step = 0; !found && lprobe < vol.probe_limit; ++step) {
        // a poisoned volume stops long scans early
        if ((step & 3u) == 3u && warp_overflowed(vol.hdr)) {
          stopped = true;
          break;
        }
        unsigned long long kk[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const unsigned off = lane + 32u * j;
          kk[j] = 0;
          if (off < vol.probe_limit - lprobe && slot_ok(vol, (ls + off) & vol.mask))
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];"
                         : "=l"(kk[j])
                         : "l"(&vol.table[(ls + off) & vol.mask].key)
                         : "memory");
        }
        unsigned off = 128;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          // (slots past the limit read as key 0, which no block of the walk's range has)
          const bool stop = lane + 32u * j < vol.probe_limit - lprobe &&
                            (kk[j] == kEmptyKey || kk[j] == lkey);
          const unsigned b = __ballot_sync(0xffffffffu, stop);
          if (off == 128 && b) off = 32u * j + static_cast<unsigned>(__ffs(b) - 1);
        }
        found = off < 128;
        ls = (ls + off) & vol.mask;
        lprobe += off;
      }
      if (static_cast<int>(lane & 24u) == L) {
        s0 = ls;
        probe = lprobe;
        if (!found) {
          if (!stopped && Op != kOpIntegrate && gl == 0) probe_exhausted(vol);
          todo = false;
        }
      }
    }
  }
  at = (s0 + gl) & vol.mask;  // (a settled key's slots stay)
  if (Op == kOpIntegrate) result = resolve_for_update(vol, result);
  return result;
}

// Keys a warp from which a tile looks at all home slots first, a key a lane.
// Where voxels are finer than pixels a tile has hundreds of blocks, and eight
// lanes a block take as many round trips as there are blocks for 32 threads,
// where one settles most keys of a sparse table; with few blocks it is a
// barrier and a round trip more. Frames into an empty volume, us without / from
// 4 / 8 / 16 keys a warp: 100x75 at 2 mm 18.4 / 14.3 / 14.3 / 18.4, 240x180 at
// 2 mm and half band 8 54 / 44 / 44 / 43, 640x480 at 2 mm 100 / 92 / 92 / 100;
// at table load 0.89, mapped, 320x240 at 2 mm 45 / 39 / 39 / 39, but at 5 mm and
// load 0.88 36.9 / 39.5 / 37.0. 640x480 at 5 mm is the same with all. The fused and stage B kernels of several rounds with one
// thread a point are compiled without it: there it costs registers (1280x720 at
// half band 8 115.0 -> 119.4 us) and gives less (640x480 at 2 mm and half band 8
// 189 -> 179 us).
constexpr int kHomeFirst = 8;

// One probe of the home slot, one key a lane (every lane of the warp calls it).
// `open` stays set for a key that it does not settle.
template <int Op, int P>
__device__ __forceinline__ int home_settle(const VolumeArgs& vol, unsigned long long key, bool& open,
                                           unsigned& at) {
  const unsigned lane = threadIdx.x & 31u;
  int bx, by, bz, result = Op == kOpIntegrate ? kAbsent : -1;
  unpack_key(key, bx, by, bz);
  at = hash_block(bx, by, bz) & vol.mask;
  bool won = false;
  if (open && slot_ok(vol, at)) {
    Entry* e = vol.table + at;
    unsigned long long k;
    int idx;
    load_entry<P>(e, k, idx);
    if (k == kEmptyKey) {
      if (Op == kOpIntegrate) {
        open = false;
      } else {
        const unsigned long long prev = atomicCAS(&e->key, kEmptyKey, key);
        won = prev == kEmptyKey;
        if (won) {
          open = false;
          result = kWon;
        }
        k = prev;
        idx = kUnpublished;
      }
    }
    if (k == key) {
      open = false;
      result = Op == kOpFused && idx == kUnpublished ? kPending : idx;
    }
    if (!open && vol.slot_index && (won || k == key)) result = static_cast<int>(at);
  }
  if (Op != kOpIntegrate && vol.slot_index) {
    const unsigned wins = __ballot_sync(0xffffffffu, won);
    if (wins && lane == static_cast<unsigned>(__ffs(wins) - 1))
      red_add_u32(&vol.hdr->count, __popc(wins));
  }
  if (Op == kOpIntegrate) result = resolve_for_update(vol, result);
  return result;
}

// Keeps the outcome of directory slot s's key.
template <int Op, int D>
__device__ __forceinline__ void note_settled(TileShared<D>& S, int s, int res, unsigned at) {
  if (Op != kOpAllocate && res >= 0) S.idx[s] = res;
  if (Op != kOpIntegrate && (res == kWon || (Op == kOpFused && res == kPending))) {
    // (claims are listed from the front, waits from the back)
    S.todo[res == kWon ? atomicAdd(&S.won, 1) : D - 1 - atomicAdd(&S.pending, 1)] =
        static_cast<unsigned short>(s);
    S.idx[s] = static_cast<int>(at);
  }
}

// Samples k0 .. k1-1 of a point on their own: each tested, resolved and added
// by its thread. For the rare points that the packed walk or the directory
// cannot hold; out of line, with one call site, to keep the registers of the
// hot code (a call in the unrolled walk costs 14 spilled registers).
template <int Op, int P>
__device__ __noinline__ void point_alone(const FrameArgs& f, const VolumeArgs& vol, float depth,
                                         int u, int v, int k0, int k1) {
  Ray r;
  if (!make_ray(f, u, v, depth, r)) return;
  float cr = 0.0f, cg = 0.0f, cb = 0.0f;
  const bool colour = Op != kOpAllocate && f.rgb != nullptr;
  if (colour) load_colour(f, u, v, cr, cg, cb);
  BlockCacheT bc;
  WalkDedupe walk;
  for (int k = k0 > 0 ? k0 - 1 : 0; k < k1; ++k) {
    int gx, gy, gz;
    float zc;
    if (!sample_voxel(f, r, k, gx, gy, gz) || walk.seen_then_push(gx, gy, gz) || k < k0 ||
        !voxel_test(f, gx, gy, gz, zc))
      continue;
    const unsigned long long key = block_key_of(gx, gy, gz);
    if (key != bc.key) {
      bc.key = key;
      bc.idx = resolve_single<Op, P>(vol, key);
    }
    if (Op != kOpAllocate && bc.idx >= 0)
      add_contribution(vol, static_cast<size_t>(bc.idx) * kBlockVoxels + local_index(gx, gy, gz),
                       tsdf_value(f, r.d, zc), colour, cr, cg, cb);
  }
}

// What a tile has claimed and what it waits for, by all threads of the CTA once
// every key of the round is settled: the indices of its claims by one addition
// to the block counter, published, and then the indices that other tiles have
// claimed and not published yet. Out of line: a tile of a mapped place never
// comes here, and its code between steps 2 and 3 costs small frames 1 %.
//
// The block counter is one word for the whole volume. With an addition for
// every four keys of a warp, made as they were settled, first frames queued for
// it: four 640x480 frames of 9,000 to 22,000 new blocks took 62 us on average,
// 45 like this, and 61 with one for every sixteen keys; a batch of 24 first
// frames 1,400 and 921 us.
template <int Op, int D, int NT>
__device__ __noinline__ void publish_and_wait(TileShared<D>& S, const VolumeArgs& vol) {
  const int won = S.won, pending = Op == kOpFused ? S.pending : 0;
  if (won) {
    if (threadIdx.x == 0) S.first = atomicAdd(&vol.hdr->count, static_cast<unsigned>(won));
    __syncthreads();
    for (int j = threadIdx.x; j < won; j += NT) {
      const int s = S.todo[j];
      const unsigned i = S.first + static_cast<unsigned>(j);
      int* out = &vol.table[static_cast<unsigned>(S.idx[s])].idx;
      if (i >= vol.pool) {
        atomicOr(&vol.hdr->err, TSDF_ERRBIT_POOL_FULL);
        atomicExch(out, kFailedIdx);
        S.idx[s] = -1;
      } else {
        int bx, by, bz;
        unpack_key(tag_key(S.base, S.dir[s]), bx, by, bz);
        store_coords(vol, i, bx, by, bz);
        *reinterpret_cast<volatile int*>(out) = static_cast<int>(i);
        S.idx[s] = static_cast<int>(i);
      }
    }
  }
  for (int j = threadIdx.x; j < pending; j += NT) {
    const int s = S.todo[D - 1 - j];
    S.idx[s] = wait_published(vol, vol.table + static_cast<unsigned>(S.idx[s]));
  }
  __syncthreads();
  if (threadIdx.x == 0) S.won = S.pending = 0;  // (the next round lists after its barrier)
}

// One tile of 16 pixels x tile_rows, TPP consecutive threads a point, each
// with a contiguous span of the point's 2M+1 band samples, C at a time (MULTI:
// as many rounds as the span needs; otherwise the span fits one). A round:
//   1. every thread walks its samples once and keeps each accepted one as a
//      packed word and its tsdf value; the tile's distinct blocks are
//      collected in the directory;
//   2. the directory's new blocks are inserted (stage B: looked up), eight
//      lanes each; the CTA takes the pool indices of all that it claimed with
//      one addition, publishes them, and then waits for those that others
//      claimed and have not published; the indices stay in shared memory;
//   3. every accepted voxel's five sums are added with two fire-and-forget
//      reductions (a 16-byte vector and a scalar).
// No grid barrier is needed: a point only touches blocks whose indices it has
// resolved, and a CTA never waits before it has published what it claimed (so
// points on their own come last: they may wait). Per voxel the
// arithmetic is the paper's in every form, and so is the result.
//
// The walk is bound by instructions (89 a sample and warp, 158 with floors and
// conversions on the quarter-rate pipe, a range check a sample and two
// dedupe windows), step 2 by round trips to the table and step 3 by the
// reductions' work in L2. The half band is a run-time number: the samples held
// between the steps, not the band, set the registers, so every truncation
// takes this path. What it takes now stands with the rules of the dispatch
// (auto_threads_per_point); the kernel before it, its walk unrolled for half
// bands 2, 4 and 8 and run twice for the others, took in the same runs
//   640x480, 5 mm, half band 4             51.6 us mapped (now 41), 53.9 empty (44)
//   1280x720, 5 mm, half band 8            260 (183), 269 (195)
//   320x240, 2 mm, table at load 0.89      94 (39), 188 (117)
// Summing a tile's contributions in shared memory first (integers, one entry
// a voxel, 40 % fewer reduction requests) measured 48 us at 640x480 but 161 us
// at 1280x720 (120 without): its atomics and two more barriers cost more than
// L2 saves.
template <int Op, int P, int C, int TPP, bool MULTI>
__device__ __forceinline__ void tile_body(TileTables<TPP>& S, const FrameArgs& f,
                                          const VolumeArgs& vol, int tile_x, int tile_y) {
  constexpr int NT = tile_threads<TPP>();
  constexpr int D = TileTables<TPP>::kSlots;
  int u, v;
  if constexpr (TPP == 1)
    tile_pixel_at(tile_x, tile_y, u, v);
  else
    tile_pixel_shared<TPP>(tile_x, tile_y, u, v);
  const bool inside = u < f.W && v < f.H;
  const bool colour = Op != kOpAllocate && f.rgb != nullptr;
  float d = 0.0f;
  if (inside) d = load_depth(f, static_cast<long long>(v) * f.W + u);
  // (the poisoned flag is looked at before the first write, not here: its
  // round trip overlaps the walk)
  if (threadIdx.x == 0) {
    S.err = load_err_volatile(vol.hdr);
    S.n = S.n_open = S.won = S.pending = 0;
  }
  const int4 none4 = make_int4(-1, -1, -1, -1);
  for (int i = threadIdx.x; i < D / 4; i += NT) reinterpret_cast<int4*>(S.dir)[i] = none4;
  const unsigned lane = threadIdx.x & 31u;
  Ray r;
  const bool valid = inside && make_ray(f, u, v, d, r);
  bool alone = false;             // the point goes to point_alone
  int ox = 0, oy = 0, oz = 0;     // block-aligned base of the packed voxels (floor_magic bits)
  if (valid) alone = !band_in_range(f, r, ox, oy, oz);
  // the tile's base block: any of its points'
  const unsigned who = __ballot_sync(0xffffffffu, valid && !alone);
  if (who && lane == static_cast<unsigned>(__ffs(who) - 1))
    S.base = (static_cast<unsigned long long>(magic_block(ox)) << 42) |
             (static_cast<unsigned long long>(magic_block(oy)) << 21) |
             static_cast<unsigned long long>(magic_block(oz));
  // this thread's samples: lo .. hi-1
  const int K = 2 * f.M + 1;
  int lo = 0, hi = K;
  if constexpr (TPP > 1) {
    const int j = static_cast<int>(threadIdx.x) % TPP;
    lo = j * K / TPP;
    hi = (j + 1) * K / TPP;
  }
  if (!valid) hi = lo;
  __syncthreads();
  unsigned base = 0, delta = 0;
  if (valid && !alone) {
    const unsigned long long tbase = S.base;
    const unsigned long long m = (1ull << 21) - 1;
    const int ddx = static_cast<int>(magic_block(ox)) - static_cast<int>((tbase >> 42) & m);
    const int ddy = static_cast<int>(magic_block(oy)) - static_cast<int>((tbase >> 21) & m);
    const int ddz = static_cast<int>(magic_block(oz)) - static_cast<int>(tbase & m);
    // a tag's fields hold +-512 blocks; the band reaches 7 blocks from its base
    alone = abs(ddx) > 500 || abs(ddy) > 500 || abs(ddz) > 500;
    base = packed_base(ox, oy, oz);
    // a packed voxel's block fields are biased by 64, a tag's by 512, 512, 2048
    delta = static_cast<unsigned>(ddx + 512 - 64) + (static_cast<unsigned>(ddy + 512 - 64) << 10) +
            (static_cast<unsigned>(ddz + 2048 - 64) << 20);
  }
  const int walked = alone ? lo : hi;  // the samples walked here end before this one
  unsigned last = 0;  // the previous sample's packed voxel (0: none)
  if (TPP > 1 && lo > 0) {
    const float tk = __fmul_rn(static_cast<float>(lo - 1 - f.M), f.v);
    last = pack_magic(floor_magic(__fmul_rn(__fmaf_rn(tk, r.dx, r.px), f.inv_v)),
                      floor_magic(__fmul_rn(__fmaf_rn(tk, r.dy, r.py), f.inv_v)),
                      floor_magic(__fmul_rn(__fmaf_rn(tk, r.dz, r.pz), f.inv_v))) -
           base;
  }
  const int span = (K + TPP - 1) / TPP;
  unsigned cur = 0;           // packed block of the directory slot held (0: none)
  unsigned slot = kSlotNone;
  int listed = 0;             // blocks resolved in earlier rounds
  for (int at = 0; at < (MULTI ? span : 1); at += C) {
    // 1. the walk: each accepted sample as one word and its tsdf value, its
    // block in the directory
    unsigned smp[C];          // accepted flag (bit 31), slot << 9, local index
    float tv[C];
    bool homeless = false;    // a block found no room in the directory
#pragma unroll
    for (int g = 0; g < C; g += kGroup) {
      // (the same in the whole warp: past its span, or no point of it to walk,
      // as where a frame has no depth: 640x480 without any 18.4 -> 8.2 us)
      if ((MULTI && at + g >= span) || !who) {
#pragma unroll
        for (int i = g; i < g + kGroup && i < C; ++i) smp[i] = 0u;
        continue;
      }
      unsigned p[kGroup];
      float zc[kGroup];
      int q[kGroup];
      const float fk = static_cast<float>(lo + at + g - f.M);
#pragma unroll
      for (int i = 0; i < kGroup; ++i) {
        if (g + i >= C) break;
        const float tk = __fmul_rn(fk + static_cast<float>(i), f.v);
        const float tx = floor_magic(__fmul_rn(__fmaf_rn(tk, r.dx, r.px), f.inv_v));
        const float ty = floor_magic(__fmul_rn(__fmaf_rn(tk, r.dy, r.py), f.inv_v));
        const float tz = floor_magic(__fmul_rn(__fmaf_rn(tk, r.dz, r.pz), f.inv_v));
        p[i] = pack_magic(tx, ty, tz) - base;
        const bool fresh = lo + at + g + i < walked && p[i] != last;
        last = p[i];
        q[i] = project_magic(f, tx, ty, tz, fresh, zc[i]);
      }
      float d2[kGroup];
#pragma unroll
      for (int i = 0; i < kGroup; ++i) {
        if (g + i >= C) break;
        d2[i] = q[i] >= 0 ? load_depth(f, q[i]) : 0.0f;
      }
#pragma unroll
      for (int i = 0; i < kGroup; ++i) {
        if (g + i >= C) break;
        const bool a = voxel_accept(f, d2[i], zc[i]);
        const unsigned b = (p[i] >> 3) & kPackBlockBits;
        const bool changed = a && b != cur;
        if (__any_sync(0xffffffffu, changed)) {
          cur = changed ? b : cur;
          dir_find(S, b + delta, changed, slot);
        }
        homeless = homeless || (a && slot == kSlotNone);
        if (Op == kOpAllocate) continue;
        tv[g + i] = tsdf_value(f, d, zc[i]);
        smp[g + i] = a ? (kSampleValid | (slot << 9) | pack_local(p[i])) : 0u;
      }
    }
    float cr = 0.0f, cg = 0.0f, cb = 0.0f;
    if (colour && valid) load_colour(f, u, v, cr, cg, cb);
    __syncthreads();
    if (S.err) return;  // poisoned volume: do nothing (uniform across the CTA)
    const bool solo = homeless || (valid && alone);
    if (solo) {
#pragma unroll
      for (int i = 0; i < C; ++i) smp[i] = 0u;
    }
    // 2. the directory's new blocks, eight lanes each, four a warp; many: what
    // their home slots do not settle
    constexpr bool kHome = TPP > 1 || !MULTI || Op == kOpAllocate;
    const int n = S.n;
    int k1 = n;
    if (kHome && n - listed > kHomeFirst * (NT / 32)) {
      for (int c0 = listed; c0 < n; c0 += NT) {
        const int i = c0 + static_cast<int>(threadIdx.x);
        const bool has = i < n;
        const int s = has ? S.list[i] : 0;
        if (Op != kOpAllocate && has) S.idx[s] = -1;
        bool open = has;
        unsigned at_slot = 0;
        const int res =
            home_settle<Op, P>(vol, has ? tag_key(S.base, S.dir[s]) : kEmptyKey, open, at_slot);
        if (has && !open) note_settled<Op, D>(S, s, res, at_slot);
        // (the open ones come to the front of the list, over what has been read)
        __syncthreads();
        if (open) S.list[listed + atomicAdd(&S.n_open, 1)] = static_cast<unsigned short>(s);
      }
      __syncthreads();
      k1 = listed + S.n_open;
    }
    for (int b0 = listed + (static_cast<int>(threadIdx.x) >> 5) * 4; b0 < k1; b0 += NT / 8) {
      const int i = b0 + static_cast<int>(lane >> 3);
      const bool has = i < k1;
      const int s = S.list[has ? i : 0];  // (no branch: 56 registers instead of 60)
      if (Op != kOpAllocate && has && (lane & 7u) == 0) S.idx[s] = -1;
      __syncwarp();
      unsigned at_slot = 0;
      const int res =
          group_resolve<Op, P>(vol, has ? tag_key(S.base, S.dir[s]) : kEmptyKey, has, at_slot);
      if (has) note_settled<Op, D>(S, s, res, at_slot);
    }
    listed = n;
    __syncthreads();
    if (threadIdx.x == 0) S.n_open = 0;  // (the next round lists after its barrier)
    if (Op != kOpIntegrate && (S.won | S.pending)) publish_and_wait<Op, D, NT>(S, vol);
    // 3. the sums, each block's index from the directory
#pragma unroll
    for (int i = 0; i < (Op == kOpAllocate ? 0 : C); ++i) {
      if (!(smp[i] & kSampleValid)) continue;
      const int o = S.idx[(smp[i] & ~kSampleValid) >> 9];
      if (o >= 0)
        add_contribution(vol, static_cast<size_t>(o) * kBlockVoxels + (smp[i] & 511u), tv[i], colour,
                         cr, cg, cb);
    }
    // (last: a thread here may wait for another tile, whose blocks and this
    // one's must have their indices by then)
    if (solo) point_alone<Op, P>(f, vol, d, u, v, lo + at, lo + at + C < hi ? lo + at + C : hi);
  }
}

// At most 64 registers a thread (four 256-thread CTAs per SM).
template <int Op, int P, int C, int TPP, bool MULTI>
__global__ void __launch_bounds__(tile_threads<TPP>(), 4 * kThreads / tile_threads<TPP>())
    tile_kernel(const __grid_constant__ FrameArgs f, const __grid_constant__ VolumeArgs vol) {
  __shared__ TileTables<TPP> S;
  tile_body<Op, P, C, TPP, MULTI>(S, f, vol, blockIdx.x, blockIdx.y);
}

inline int tiles_of(int n) { return (n + kTile - 1) / kTile; }

// Launch with C samples a round: the whole span when it fits, else rounds.
template <int Op, int P, int C, int TPP, bool MULTI = false>
cudaError_t launch_tile_c(const FrameArgs& f, const VolumeArgs& vol, cudaStream_t s) {
  constexpr int rows = tile_rows<TPP>();
  const dim3 grid(static_cast<unsigned>(tiles_of(f.W)), static_cast<unsigned>((f.H + rows - 1) / rows));
  tile_kernel<Op, P, C, TPP, MULTI><<<grid, tile_threads<TPP>(), 0, s>>>(f, vol);
  return cudaGetLastError();
}

// Nine samples a round at most: more are not held in 64 registers without
// spills that cost more than a second round. A round longer than the span walks
// masked samples: stage A of 640x480 at half band 2 takes 16.4 us with five and
// 20.5 with nine, 1280x720 33 and 43 us.
template <int Op, int P, int TPP>
cudaError_t launch_tile(const FrameArgs& f, const VolumeArgs& vol, cudaStream_t s) {
  constexpr int kMaxSpan = (2 * kMaxHalfBand + TPP) / TPP;
  const int span = (2 * f.M + TPP) / TPP;
  if constexpr (Op == kOpAllocate || P != kLoadCached) {  // (the rarer forms: three of them)
    if (span <= 5) return launch_tile_c<Op, P, 5, TPP>(f, vol, s);
    if (span <= 9) return launch_tile_c<Op, P, 9, TPP>(f, vol, s);
    return launch_tile_c<Op, P, 9, TPP, true>(f, vol, s);
  } else {
    if (span <= 3) return launch_tile_c<Op, P, 3, TPP>(f, vol, s);
    if (kMaxSpan <= 5 || span <= 5) return launch_tile_c<Op, P, 5, TPP>(f, vol, s);
    if constexpr (kMaxSpan > 5) {
      if (span <= 7) return launch_tile_c<Op, P, 7, TPP>(f, vol, s);
      if (kMaxSpan <= 9 || span <= 9) return launch_tile_c<Op, P, 9, TPP>(f, vol, s);
    }
    if constexpr (kMaxSpan > 9) return launch_tile_c<Op, P, 9, TPP, true>(f, vol, s);
    return cudaErrorInvalidValue;  // not reached: the half band is at most 16
  }
}

}  // namespace tsdf
