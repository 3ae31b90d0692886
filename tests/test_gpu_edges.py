"""Forms of a call that the other GPU tests do not reach, against the CPU oracle
(blocks and weights exact, means within the tolerance of test_gpu_parity.py,
which is derived there)."""
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import test_gpu_tile
from paper_2608_08287_gb300 import synth, tsdf
from test_gpu_parity import (_built, assert_same_volume, gpu_volume, oracle_volume,  # noqa: F401
                             to_dev)
from test_gpu_tile import check

pytestmark = pytest.mark.gpu


STRETCHED = synth.VolumeSpec(0.05, 0.8, 1 << 14, 1 << 13)     # half band 16


def stretched_frame(scale, seed=11, width=24, height=16):
    """A pose whose rotation part is `scale` times a rotation. The centre map takes its
    transpose for its inverse, so a voxel's depth is scale^2 times the sample's, and what is
    accepted is where the band comes back to the camera: depths of a whole number of steps
    and a little more, and a camera just behind the centre of a voxel."""
    rs = np.random.RandomState(seed)
    intr = np.array([20, 20, 11.5, 7.5], np.float32)
    u, v = np.meshgrid((np.arange(width) - intr[2]) / intr[0], (np.arange(height) - intr[3]) / intr[1])
    steps = rs.randint(2, 16, (height, width))
    depth = steps * STRETCHED.voxel_size / np.sqrt(u * u + v * v + 1) + 0.2 / scale ** 2
    rgb = rs.randint(0, 256, (height, width, 3)).astype(np.uint8)
    turn = synth.rotation(0.4, -0.3, 0.2)
    at = np.array([0.325, 0.125, -0.175]) - turn[:, 2] * 0.4 / scale
    pose = synth.make_pose(turn * scale, at).astype(np.float32)
    return synth.Frame(depth=depth.astype(np.float32), rgb=rgb, intr=intr, pose=pose)


@pytest.mark.parametrize("opts", [dict(), dict(threads_per_point=1),
                                  dict(fuse_mode=0, allocate_mode=1),
                                  dict(fuse_mode=0, allocate_mode=0, integrate_mode=0)],
                         ids=["auto", "one", "staged", "paper"])
@pytest.mark.parametrize("scale", [1.0, 2.9, 20.0, 40.0, 90.0])
def test_stretched_pose(scale, opts):
    """A band that reaches further from its point than the packed walk holds."""
    frame = stretched_frame(scale)
    ov = oracle_volume(STRETCHED)
    assert ov.fuse_frame(frame) == "OK" and ov.last_stats["contributions"] > 100
    check([frame], STRETCHED, **opts)


@pytest.mark.parametrize("opts", [dict(batch_streams=0), dict(batch_streams=0, use_graph=1, ctas_per_sm=1),
                                  dict(batch_streams=3)], ids=["persistent", "graph", "streams"])
@pytest.mark.parametrize("band", [1, 4, 9])
def test_batch_with_the_papers_update(band, opts):
    """Stage B mode 0 set for a batch: per-thread lookups in both of its forms."""
    spec = synth.VolumeSpec(0.02, 0.02 * band, 1 << 14, 1 << 13)
    frames = [synth.room_frame(9 * i, width=w, height=h) for i, (w, h) in
              enumerate([(160, 120), (97, 61), (320, 240), (33, 50)])]
    vols = [gpu_volume(spec) for _ in frames]
    batch = tsdf.Batch(4, fuse_mode=0, integrate_mode=0, **opts)
    items = [(v, *to_dev(f), f.intr, f.pose) for v, f in zip(vols, frames)]
    for _ in range(2):
        assert batch.fuse_async(items) == "OK" and batch.status(4)[0] == "OK"
    for v, f in zip(vols, frames):
        ov = oracle_volume(spec)
        assert ov.fuse_frame(f) == ov.fuse_frame(f) == "OK"
        assert assert_same_volume(v, ov) > 50
        v.close()
    batch.close()


# (stage A with a tile's directory, stage B with the paper's per-thread lookups)
PAPER = dict(fuse_mode=0, allocate_mode=1, integrate_mode=0)


@pytest.mark.parametrize("opts", [dict(), dict(fuse_mode=0), PAPER], ids=["fused", "staged", "paper"])
@pytest.mark.parametrize("band", [1, 3, 5, 6, 7, 9, 12, 16])
def test_bands_at_two_threads_a_point(band, opts):
    """300 tiles: two threads a point, rounds of every length and bands of two rounds."""
    spec = synth.VolumeSpec(0.02, 0.02 * band, 1 << 14, 1 << 13)
    check([synth.room_frame(3 * band, width=320, height=240)], spec, **opts)


@pytest.mark.parametrize("opts", [dict(), dict(fuse_mode=0), PAPER], ids=["fused", "staged", "paper"])
@pytest.mark.parametrize("band", [2, 7, 16])
def test_bands_at_one_thread_a_point(band, opts):
    """1,230 tiles, a mapped second frame beside the first."""
    spec = synth.VolumeSpec(0.04, 0.04 * band, 1 << 13, 1 << 12)
    check([synth.room_frame(k, width=656, height=480) for k in (0, 3)], spec, **opts)


@pytest.mark.parametrize("shift", [41943.04, -41943.04, 60000.0, 83886.0])
def test_far_with_the_papers_update(shift):
    test_gpu_tile.test_far(shift, PAPER)


@pytest.mark.parametrize("deepest", [3.0, 60.0])
def test_scattered_with_the_papers_update(deepest):
    test_gpu_tile.test_scattered(deepest, PAPER)


def test_long_chains_with_the_papers_update():
    test_gpu_tile.test_long_chains(PAPER)


@pytest.mark.parametrize("opts", [dict(), dict(threads_per_point=1), dict(fuse_mode=0), dict(slot_index=1),
                                  dict(probe_load=2)],
                         ids=["auto", "one", "staged", "slot", "relaxed"])
@pytest.mark.parametrize("band", [9, 16])
def test_more_blocks_than_the_directory(band, opts):
    """Tiles of 256 points with more blocks than the 1,024 slots of their directory, in later
    rounds of the walk: rays along a diagonal, which cross most blocks. (With two threads or
    more a point a tile has 64 points at most, of 8 blocks each.) The frame has 1,230 tiles,
    so that every form takes one thread a point, and depths in a few of them."""
    rs = np.random.RandomState(band)
    depth = np.zeros((480, 656), np.float32)
    full = [(0, 0), (2, 3), (29, 40), (17, 8)]          # tiles (row, column)
    for r, c in full:
        depth[16 * r:16 * r + 16, 16 * c:16 * c + 16] = 1 + 2 * rs.permutation(256).reshape(16, 16) / 256
    rgb = rs.randint(0, 256, (480, 656, 3)).astype(np.uint8)
    pose = np.eye(4, dtype=np.float32)
    fr = synth.Frame(depth=depth, rgb=rgb, intr=np.array([20, 20, -16, -16], np.float32), pose=pose)
    spec = synth.VolumeSpec(0.004, 0.004 * band, 1 << 14, 1 << 14)
    one = np.zeros_like(depth)
    one[:16, :16] = depth[:16, :16]
    ov = oracle_volume(spec)
    assert ov.fuse_frame(synth.Frame(depth=one, rgb=rgb, intr=fr.intr, pose=pose)) == "OK"
    assert ov.block_count() > 1024
    check([fr, fr], spec, **opts)


def test_tile_kernel_under_range_checks():
    """The tile kernel's edges against the checked library (as test_gpu_checked.py does for the
    parity tests): an index out of range would be reported as BOUNDS."""
    from paper_2608_08287_gb300.build import build_library
    build_library(checked=True)
    env = dict(os.environ, TSDF_CHECKED="1")
    r = subprocess.run([sys.executable, "-m", "pytest", "-x", "-q", "-p", "no:cacheprovider",
                        os.path.join("tests", "test_gpu_tile.py"), os.path.join("tests", "test_gpu_edges.py"),
                        "-m", "gpu", "-k", "not under_range_checks"],
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))), env=env,
                       capture_output=True, text=True, timeout=1800)
    assert r.returncode == 0 and " passed" in r.stdout, (r.stdout + r.stderr)[-3000:]
