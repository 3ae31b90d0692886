"""Warp-wide operations of the table probes under a poisoned flag that changes
while the warp reads it (CPU): the device functions are compiled for the host
and run by 32 threads that meet in every `_sync` operation
(emulated_warp.h). Half of the lanes see a volume that has just been poisoned
by another CTA, the others one that has not: every lane must still take part
in every operation of the scan, and the scan must end."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_08287_gb300", "csrc")


def closing(text, i):
    """Index just past the bracket that closes the one at i (strings skipped)."""
    depth, j = 0, i
    while True:
        if text[j] == '"':
            j = text.index('"', j + 1)
        elif text[j] in "([{":
            depth += 1
        elif text[j] in ")]}":
            depth -= 1
            if depth == 0:
                return j + 1
        j += 1


def on_host(text):
    """PTX statements as calls of the functions of the same name in emulated_warp.h."""
    out, at = [], 0
    while True:
        i = text.find("asm volatile(", at)
        if i < 0:
            return "".join(out) + text[at:]
        j = closing(text, i + len("asm volatile"))
        body = text[i + len("asm volatile("):j - 1]
        name = re.match(r'"([a-z0-9_.]+)', body).group(1).replace(".", "_")
        args, k = [], body.index('"', 1) + 1
        while True:
            m = re.compile(r'"=?[lrf]"\s*\(').search(body, k)
            if not m:
                break
            k = closing(body, m.end() - 1)
            args.append(body[m.end():k - 1])
        out.append(text[at:i] + f"emu::{name}({', '.join(args)})")
        at = j


def source(name):
    return open(os.path.join(CSRC, name)).read()


def function(text, head):
    """The function definition that starts with `head`, with its template line."""
    i = text.index(head)
    start = text.rindex("template <", 0, i)
    return text[start:closing(text, text.index("{", i))]


SCAN = r"""
#include <cstdio>
using namespace tsdf;
alignas(16) static Entry table[1 << 12];
static Header headers[32];
static unsigned poisoned_lanes;

static VolumeArgs volume(unsigned lane) {
  VolumeArgs v{};
  v.table = table;
  v.mask = (1 << 12) - 1;
  v.slots = v.probe_limit = 1 << 12;
  v.pool = 1 << 12;
  v.hdr = &headers[lane];
  v.slot_index = 1;
  headers[lane].err = (poisoned_lanes >> lane & 1u) ? TSDF_ERRBIT_POOL_FULL : 0u;
  return v;
}

int main(int argc, char** argv) {
  const unsigned long long key = pack_key(5, 6, 7);
  const unsigned home = hash_block(5, 6, 7) & 4095u, at = 3000;
  for (unsigned i = 0; i < 4096; ++i) table[i] = {pack_key(900 + static_cast<int>(i), 0, 0), 0, 0};
  table[(home + at) & 4095u].key = key;
  const bool group = argv[1][0] == 'g';
  poisoned_lanes = argv[2][0] == 'n' ? 0u : argv[2][0] == 'a' ? 0xffffffffu : 0xffff0000u;
  int found = -1;
  const bool ok = emu::run_warp([&](unsigned lane) {
    const VolumeArgs vol = volume(lane);
    if (group) {
      unsigned at = 0;
      const int r = group_resolve<kOpFused, kLoadCached>(vol, key, lane < 8, at);
      if (r >= 0) found = r;
    } else {
      bool todo = lane == 3;
      unsigned s = (home + 4) & 4095u, probe = 4;
      warp_skip_long_chains(vol, key, todo, s, probe);
      if (lane == 3 && todo) found = static_cast<int>(s);
    }
    __syncwarp();  // (the callers go on together)
  });
  if (!ok) {
    std::printf("lanes apart\n");
    return 0;
  }
  std::printf("%s\n", found < 0 ? "stopped" : found == static_cast<int>((home + at) & 4095u) ? "found" : "wrong");
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    made = {}

    def build(name, text):
        if name not in made:
            d = tmp_path_factory.mktemp(name)
            (d / "cuda_runtime.h").write_text('#pragma once\n#include "emulated_warp.h"\n')
            (d / "main.cpp").write_text(text)
            cmd = [gxx, "-std=c++17", "-O1", "-w", "-pthread", "-ffp-contract=off", "-I", str(d),
                   "-I", os.path.join(ROOT, "tests"), "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                   str(d / "main.cpp"), "-o", str(d / "run")]
            r = subprocess.run(cmd, capture_output=True, text=True)
            assert r.returncode == 0, r.stderr[-3000:]
            made[name] = str(d / "run")
        return made[name]

    return build


def device_header():
    return on_host(source("tsdf_device.cuh")).replace("#pragma once", "")


@pytest.mark.parametrize("which", ["group", "chain"])
@pytest.mark.parametrize("poisoned,want", [("none", "found"), ("all", "stopped"), ("half", "stopped")])
def test_long_scan_ends_together(program, which, poisoned, want):
    tile = source("tsdf_tile.cuh")
    text = (device_header() +
            "namespace tsdf { enum TileOp { kOpAllocate = 0, kOpIntegrate = 1, kOpFused = 2 };\n"
            "constexpr int kPending = -4, kWon = -5;\n" +
            on_host(function(tile, "__device__ __forceinline__ int group_resolve")) + "}\n" + SCAN)
    r = subprocess.run([program("scan", text), which, poisoned], capture_output=True, text=True,
                       timeout=60)
    assert r.stdout.strip() == want, r.stdout + r.stderr


FRAME = r"""
#include <cstdio>
using namespace tsdf;
static Entry table[1 << 8];
static Header headers[32];
static float4 sums[(1 << 8) * kBlockVoxels];
static float blues[(1 << 8) * kBlockVoxels], depth[32];
static uint8_t rgb[96];

int main(int, char** argv) {
  for (auto& e : table) e = {kEmptyKey, kUnpublished, 0};
  for (int i = 0; i < 32; ++i) depth[i] = 1.0f + 0.02f * static_cast<float>(i);
  const unsigned poisoned = argv[1][0] == 'n' ? 0u : argv[1][0] == 'a' ? 0xffffffffu : 0x0f0f00ffu;
  FrameArgs f{};
  f.depth = depth;
  f.rgb = rgb;
  f.W = 8;
  f.H = 4;
  f.fx = f.fy = 20.0f;
  f.cx = 4.0f;
  f.cy = 2.0f;
  f.v = 0.02f;
  f.inv_v = 50.0f;
  f.tau = 0.08f;
  f.neg_tau = -0.08f;
  f.inv_tau = 12.5f;
  f.M = 4;
  for (int i = 0; i < 3; ++i) {
    f.R[4 * i] = 1.0f;
    f.A[4 * i] = f.v;
    f.b[i] = 0.5f * f.v;
  }
  const bool ok = emu::run_warp([&](unsigned lane) {
    VolumeArgs v{};
    v.table = table;
    v.mask = 255;
    v.slots = v.probe_limit = v.pool = 256;
    v.twrg = sums;
    v.blue = blues;
    v.hdr = &headers[lane];
    v.slot_index = 1;
    headers[lane].err = (poisoned >> lane & 1u) ? TSDF_ERRBIT_TABLE_FULL : 0u;
    warp_body<kOpFused, kLoadCached, 4>(f, v, 0, 1);
  });
  double weight = 0;
  for (const auto& s : sums) weight += s.y;
  std::printf("%s\n", !ok ? "lanes apart" : weight > 100 ? "fused" : weight > 0 ? "in part" : "nothing");
}
"""


@pytest.mark.parametrize("poisoned,want", [("none", "fused"), ("all", "nothing"), ("half", "nothing")])
def test_warp_kernel_leaves_together(program, poisoned, want):
    tile, kernels = source("tsdf_tile.cuh"), source("tsdf_kernels.cu")

    def between(text, a, b):
        return on_host(text[text.index(a):text.index(b)])

    text = (device_header() + "namespace tsdf {" +
            between(tile, "constexpr int kThreads", "// Insert into the CTA's") +
            between(tile, "// Walk state of one point", "// -----------------------------------"
                    "-----------------------------------------\n// stage A, the paper's") +
            between(tile, "// One-entry cache", "// Pixel of this thread when TPP") +
            between(kernels, "template <int Op, int P>\n__device__ __forceinline__ int warp_resolve",
                    "// MinBlocks:") + "}\n" + FRAME)
    r = subprocess.run([program("frame", text), poisoned], capture_output=True, text=True, timeout=60)
    assert r.stdout.strip() == want, r.stdout + r.stderr
