"""The packed walk against the plain one over poses that are not rigid (CPU): a
pose is any twelve finite numbers, and a rotation part that stretches the ray
takes the band's samples further from their point than a packed word holds.
Every point that the kernels would walk packed must give, sample by sample, the
voxel and block of sample_voxel; the device functions are compiled for the
host (emulated_warp.h). The GPU results of such poses are compared with the
oracle in test_gpu_edges.py."""
import subprocess

import pytest

from test_warp_uniform import device_header, on_host, program, source  # noqa: F401

POSES = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
using namespace tsdf;

int main(int, char** argv) {
  const double scale = std::atof(argv[1]);
  std::mt19937 rng(7);
  std::uniform_real_distribution<double> u(-1, 1);
  long packed = 0, wrong = 0;
  for (int band = 1; band <= kMaxHalfBand; ++band) {
    for (int n = 0; n < 200; ++n) {
      FrameArgs f{};
      f.W = f.H = 64;
      f.fx = f.fy = 50.0f;
      f.cx = f.cy = 32.0f;
      f.v = 0.01f;
      f.inv_v = 1.0f / f.v;
      f.M = band;
      // a rotation about a random axis (Rodrigues), stretched
      double a[3] = {u(rng), u(rng), u(rng)}, th = 3.1 * u(rng);
      const double l = std::sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
      for (double& x : a) x /= l;
      const double c = std::cos(th), s = std::sin(th);
      const double K[3][3] = {{0, -a[2], a[1]}, {a[2], 0, -a[0]}, {-a[1], a[0], 0}};
      for (int i = 0; i < 3; ++i) {
        for (int j = 0; j < 3; ++j)
          f.R[3 * i + j] = static_cast<float>(
              scale * ((i == j ? c : 0.0) + s * K[i][j] + (1 - c) * a[i] * a[j]));
        f.t[i] = static_cast<float>(30 * u(rng));
      }
      f.walk_limit = packed_walk_limit(f.R, f.M);
      Ray r;
      int ox, oy, oz;
      if (!make_ray(f, n % 64, n / 4, static_cast<float>(2.1 + u(rng)), r) ||
          !band_in_range(f, r, ox, oy, oz))
        continue;
      ++packed;
      const unsigned base = packed_base(ox, oy, oz);
      const unsigned long long key0 = (static_cast<unsigned long long>(magic_block(ox) - 64u) << 42) |
                                      (static_cast<unsigned long long>(magic_block(oy) - 64u) << 21) |
                                      static_cast<unsigned long long>(magic_block(oz) - 64u);
      for (int k = 0; k <= 2 * band; ++k) {
        int gx, gy, gz;
        const bool in = sample_voxel(f, r, k, gx, gy, gz);
        const float tk = __fmul_rn(static_cast<float>(k - f.M), f.v);
        const unsigned p = pack_magic(floor_magic(__fmul_rn(__fmaf_rn(tk, r.dx, r.px), f.inv_v)),
                                      floor_magic(__fmul_rn(__fmaf_rn(tk, r.dy, r.py), f.inv_v)),
                                      floor_magic(__fmul_rn(__fmaf_rn(tk, r.dz, r.pz), f.inv_v))) -
                           base;
        const unsigned b = (p >> 3) & kPackBlockBits;
        const unsigned long long key = key0 + (static_cast<unsigned long long>(b & 127u) << 42) +
                                       (static_cast<unsigned long long>((b >> 10) & 127u) << 21) +
                                       (b >> 20);
        // a tag adds up to 500 blocks to each field, which must stay within its bits
        const unsigned fx = b & 127u, fy = (b >> 10) & 127u, fz = b >> 20;
        const bool near = fx - 53u <= 22u && fy - 53u <= 22u && fz - 53u <= 22u;
        wrong += !in || !near || key != pack_key(gx >> 3, gy >> 3, gz >> 3) ||
                 pack_local(p) != static_cast<unsigned>(local_index(gx, gy, gz));
      }
    }
  }
  std::printf("%ld %ld\n", packed, wrong);
}
"""


@pytest.mark.parametrize("scale", [0.01, 1.0, 1.001, 2.9, 3.1, 20.0, 200.0, 5000.0])
def test_packed_walk_is_the_walk(program, scale):  # noqa: F811
    tile = source("tsdf_tile.cuh")
    walk = tile[tile.index("// floor(x) by one addition"):tile.index("// Key of a tag")]
    text = device_header() + "namespace tsdf {" + on_host(walk) + "}\n" + POSES
    r = subprocess.run([program("poses", text), str(scale)], capture_output=True, text=True, timeout=60)
    packed, wrong = (int(x) for x in r.stdout.split())
    assert wrong == 0
    if scale <= 2.9:
        assert packed == 16 * 200     # every band of a pose that is rigid, or nearly, is packed
