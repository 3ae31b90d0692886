"""One tile of the tile kernel on the host (CPU): 256 or 128 threads that meet in
every warp operation and barrier (emulated_warp.h), against a plain walk of
the same points.
  * the tile's blocks, their coordinates and every voxel's weight are those of
    the walk; pool indices are given out without a gap;
  * the volume's block counter, one word for the whole volume, is added to once
    a round of the walk, however many blocks the tile claims: each addition
    waits for those of all other tiles;
  * a tile of many blocks reads little more than one table entry a block where
    the table is sparse (a block at a time is looked at by eight lanes, and a
    round trip later the next);
  * blocks that another tile has claimed but not published are waited for."""
import subprocess

import pytest

from test_warp_uniform import device_header, on_host, program, source  # noqa: F401

TILE = r"""
#include <cstdio>
#include <cstdlib>
#include <set>
#include <tuple>
using namespace tsdf;
constexpr unsigned kSlots = 1 << 14;
static Entry table[kSlots];
static Header hdr;
static int32_t coords[3 * kSlots];
static float4* sums;
static float* blues;
static float depth[256];
static uint8_t rgb[768];

template <int TPP, bool MULTI>
static void run(const FrameArgs& f, const VolumeArgs& v) {
  static TileTables<TPP> S;
  const bool ok = emu::run_cta(tile_threads<TPP>(), [&](unsigned) {
    tile_body<kOpFused, kLoadCached, 9, TPP, MULTI>(S, f, v, 0, 0);
  });
  if (!ok) std::printf("lanes apart ");
}

int main(int, char** argv) {
  const int tpp = std::atoi(argv[1]), band = std::atoi(argv[2]);
  const double voxel = std::atof(argv[3]);
  const bool contested = argv[4][0] == 'c';
  for (auto& e : table) e = {kEmptyKey, kUnpublished, 0};
  const float spread = static_cast<float>(std::atof(argv[5]));  // of the depths, metres
  for (int i = 0; i < 256; ++i) depth[i] = 1.0f + spread * static_cast<float>((i * 37) % 256) / 256;
  for (int i = 0; i < 16 * std::atoi(argv[8]); ++i) depth[i] = 0.0f;  // rows without depth
  FrameArgs f{};
  f.depth = depth;
  f.rgb = rgb;
  f.W = 16;
  f.H = tpp == 1 ? 16 : tile_rows<2>();
  f.cx = f.cy = static_cast<float>(std::atof(argv[6]));
  f.fx = f.fy = static_cast<float>(std::atof(argv[7]));
  f.v = static_cast<float>(voxel);
  f.inv_v = 1.0f / f.v;
  f.M = band;
  f.tau = f.v * static_cast<float>(band);
  f.neg_tau = -f.tau;
  f.inv_tau = 1.0f / f.tau;
  for (int i = 0; i < 3; ++i) {
    f.R[4 * i] = 1.0f;
    f.A[4 * i] = f.v;
    f.b[i] = 0.5f * f.v;
  }
  f.walk_limit = packed_walk_limit(f.R, f.M);
  VolumeArgs v{};
  v.table = table;
  v.mask = kSlots - 1;
  v.slots = v.probe_limit = v.pool = kSlots;
  v.coords = coords;
  v.hdr = &hdr;
  v.timeout_ns = 1000000000ull;
  sums = static_cast<float4*>(std::calloc(static_cast<size_t>(kSlots) * kBlockVoxels, sizeof(float4)));
  blues = static_cast<float*>(std::calloc(static_cast<size_t>(kSlots) * kBlockVoxels, sizeof(float)));
  v.twrg = sums;
  v.blue = blues;

  // the plain walk: the weight of every voxel
  std::map<std::tuple<int, int, int>, int> want;
  std::set<std::tuple<int, int, int>> blocks;
  for (int p = 0; p < f.W * f.H; ++p) {
    Ray r;
    if (!make_ray(f, p % 16, p / 16, depth[p], r)) continue;
    WalkDedupe walk;
    for (int k = 0; k <= 2 * f.M; ++k) {
      int x, y, z;
      float zc;
      if (!sample_voxel(f, r, k, x, y, z) || walk.seen_then_push(x, y, z) || !voxel_test(f, x, y, z, zc))
        continue;
      ++want[{x, y, z}];
      blocks.insert({x >> 3, y >> 3, z >> 3});
    }
  }
  // contested: every third block has been claimed elsewhere, and is published
  // while the tile waits
  std::vector<unsigned> late;
  if (contested) {
    int n = 0;
    for (const auto& b : blocks) {
      if (n++ % 3) continue;
      int x, y, z;
      std::tie(x, y, z) = b;
      unsigned s = hash_block(x, y, z) & v.mask;
      while (table[s].key != kEmptyKey) s = (s + 1) & v.mask;
      table[s].key = pack_key(x, y, z);
      late.push_back(s);
    }
  }
  g_watched = &hdr.count;
  g_reciprocals = 0;
  std::thread other([&] {
    std::this_thread::sleep_for(std::chrono::milliseconds(30));
    for (unsigned s : late) {
      const unsigned i = __atomic_fetch_add(&hdr.count, 1u, __ATOMIC_SEQ_CST);
      unpack_key(table[s].key, coords[3 * i], coords[3 * i + 1], coords[3 * i + 2]);
      __atomic_store_n(&table[s].idx, static_cast<int>(i), __ATOMIC_SEQ_CST);
    }
  });
  if (tpp == 1 && band <= 4)
    run<1, false>(f, v);
  else if (tpp == 1)
    run<1, true>(f, v);
  else if (band <= 8)
    run<2, false>(f, v);
  else
    run<2, true>(f, v);
  other.join();

  long wrong = hdr.err != 0 || hdr.count != blocks.size(), weight = 0, total = 0;
  for (const auto& e : want) total += e.second;
  std::set<int> used;
  for (const auto& e : table) {
    if (e.key == kEmptyKey) continue;
    int x, y, z;
    unpack_key(e.key, x, y, z);
    if (!blocks.count({x, y, z}) || e.idx < 0 || e.idx >= static_cast<int>(hdr.count) ||
        !used.insert(e.idx).second || coords[3 * e.idx] != x || coords[3 * e.idx + 1] != y ||
        coords[3 * e.idx + 2] != z) {
      ++wrong;
      continue;
    }
    for (int l = 0; l < kBlockVoxels; ++l) {
      const float w = sums[static_cast<size_t>(e.idx) * kBlockVoxels + l].y;
      const auto it = want.find({8 * x + (l & 7), 8 * y + (l >> 3 & 7), 8 * z + (l >> 6)});
      wrong += w != static_cast<float>(it == want.end() ? 0 : it->second);
      weight += static_cast<long>(w);
    }
  }
  wrong += weight != total;
  std::printf("%ld %zu %u %u %u\n", wrong, blocks.size(), g_watched_adds, emu::g_entry_loads,
              g_reciprocals);
}
"""


def tile_program(program):  # noqa: F811
    tile = source("tsdf_tile.cuh").replace("#pragma once", "").replace('#include "tsdf_device.cuh"', "")
    tile = tile[:tile.index("// At most 64 registers a thread (four")] + "}\n"
    return program("tile", "#include <chrono>\n#include <math.h>\n" + device_header() + on_host(tile) + TILE)


def run_tile(program, *args, empty=0):  # noqa: F811
    """(wrong voxels, blocks, additions to the block counter, table entries read, projections)
    of one tile whose first `empty` rows have no depth."""
    r = subprocess.run([tile_program(program), *(str(a) for a in (*args, empty))],
                       capture_output=True, text=True, timeout=100)
    return (int(x) for x in r.stdout.split())


@pytest.mark.parametrize("others", ["alone", "contested"])
@pytest.mark.parametrize("tpp,band,voxel,least,rounds",
                         [(1, 2, 0.08, 8, 1), (1, 4, 0.01, 100, 1), (1, 4, 0.004, 400, 1), (1, 8, 0.004, 600, 2),
                          (1, 16, 0.01, 200, 4), (2, 4, 0.01, 40, 1), (2, 16, 0.004, 200, 2)])
def test_one_addition_a_round(program, tpp, band, voxel, least, rounds, others):  # noqa: F811
    wrong, blocks, additions, *_ = run_tile(program, tpp, band, voxel, others, 0.25, 8, 40)
    assert wrong == 0 and blocks >= least
    assert additions <= rounds


@pytest.mark.parametrize("tpp,band,voxel", [(1, 4, 0.004), (2, 16, 0.004)])
def test_many_blocks_in_a_sparse_table(program, tpp, band, voxel):  # noqa: F811
    wrong, blocks, _, loads, _ = run_tile(program, tpp, band, voxel, "alone", 0.25, 8, 40)
    assert wrong == 0 and blocks >= 200
    assert loads <= 2 * blocks


@pytest.mark.parametrize("empty,projected", [(0, 256 * 9), (3, 256 * 9), (8, 128 * 9), (16, 0)])
def test_nothing_is_walked_without_depth(program, empty, projected):  # noqa: F811
    """A warp (eight by four pixels) whose points have no depth projects no sample."""
    wrong, *_, projections = run_tile(program, 1, 4, 0.01, "alone", 0.25, 8, 40, empty=empty)
    assert wrong == 0 and projections == projected


@pytest.mark.parametrize("others", ["alone", "contested"])
@pytest.mark.parametrize("band", [9, 16])
def test_more_blocks_than_the_directory(program, band, others):  # noqa: F811
    """The points whose blocks find no room, beside blocks that found some, in later
    rounds of the walk (rays along a diagonal, which cross most blocks). With two
    threads or more a point a tile has 64 points at most, of 8 blocks: none overflows."""
    wrong, blocks, *_ = run_tile(program, 1, band, 0.004, others, 2.0, -16, 20)
    assert wrong == 0 and blocks > 1024
