"""The tile kernel where its packed walk, block directory and table probe have
edges, against the CPU oracle (blocks and weights exact, means within the
tolerance of test_gpu_parity.py, which is derived there):
  * every count of samples a round can hold, and bands of several rounds;
  * images smaller than a tile and with ragged tiles;
  * voxel coordinates at and beyond the packed walk's range (2^22 voxels);
  * tiles whose points lie further apart than a directory tag reaches, and
    tiles with more blocks than the directory holds;
  * probe chains longer than a group's window and than a scan step, wrapping
    around the end of the table.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2608_08287_gb300 import synth
from test_gpu_parity import (_built, assert_same_volume, gpu_volume, oracle_volume,  # noqa: F401
                             to_dev)

pytestmark = pytest.mark.gpu

STAGED = dict(fuse_mode=0, allocate_mode=1, integrate_mode=2)


def check(frames, spec, rgb=True, **opts):
    gv, ov = gpu_volume(spec, **opts), oracle_volume(spec)
    for fr in frames:
        d, c = to_dev(fr, rgb)
        assert gv.fuse(d, fr.intr, fr.pose, c) == "OK"
        if not rgb:
            fr = synth.Frame(depth=fr.depth, rgb=None, intr=fr.intr, pose=fr.pose)
        assert ov.fuse_frame(fr) == "OK"
    assert_same_volume(gv, ov, rgb)
    gv.close()


@pytest.mark.parametrize("opts", [dict(threads_per_point=0), dict(threads_per_point=1), STAGED],
                         ids=["auto", "one", "staged"])
@pytest.mark.parametrize("band", [1, 2, 3, 4, 5, 6, 8, 9, 13, 14, 16])
def test_bands(band, opts):
    spec = synth.VolumeSpec(0.02, 0.02 * band, 1 << 14, 1 << 13)
    check([synth.plane_sphere_frame(seed=band, width=90, height=61, intr=(80.0, 80.0, 45.0, 30.0))],
          spec, **opts)


@pytest.mark.parametrize("size", [(1, 1), (17, 3), (15, 33), (129, 2)])
@pytest.mark.parametrize("rgb", [True, False])
def test_ragged(size, rgb):
    w, h = size
    fr = synth.plane_sphere_frame(seed=w, width=w, height=h, dropout=0.0,
                                  intr=(60.0, 60.0, w / 2.0, h / 2.0))
    check([fr], synth.VolumeSpec(0.01, 0.04, 1 << 13, 1 << 12), rgb)


@pytest.mark.parametrize("opts", [dict(), STAGED], ids=["fused", "staged"])
@pytest.mark.parametrize("shift", [41943.04, -41943.04, 41941.5, 60000.0, 83886.0])
def test_far(shift, opts):
    """The camera beside 2^22 voxels, beyond it, and at the last blocks (2^23 voxels)."""
    fr = synth.plane_sphere_frame(seed=5, width=48, height=40, intr=(40.0, 40.0, 24.0, 20.0))
    for axis in (0, 2):
        pose = fr.pose.copy()
        pose[axis, 3] += np.float32(shift)
        moved = synth.Frame(depth=fr.depth, rgb=fr.rgb, intr=fr.intr, pose=pose)
        check([moved], synth.VolumeSpec(0.01, 0.04, 1 << 14, 1 << 13), **opts)


@pytest.mark.parametrize("opts", [dict(threads_per_point=1), dict(threads_per_point=2), STAGED],
                         ids=["one", "two", "staged"])
@pytest.mark.parametrize("deepest", [3.0, 60.0])
def test_scattered(deepest, opts):
    """Unrelated depths: at 2 mm, more blocks a tile than the directory has slots; up to 60 m,
    further apart than a tag reaches."""
    rs = np.random.RandomState(3)
    depth = rs.uniform(0.3, deepest, (64, 64)).astype(np.float32)
    rgb = rs.randint(0, 256, (64, 64, 3)).astype(np.uint8)
    pose = synth.make_pose(synth.rotation(0.7, 0.3, 0.1), (0.2, -0.1, 0.4)).astype(np.float32)
    fr = synth.Frame(depth=depth, rgb=rgb, intr=np.array([50, 50, 32, 32], np.float32), pose=pose)
    check([fr], synth.VolumeSpec(0.002, 0.008, 1 << 16, 1 << 16), **opts)


@pytest.mark.parametrize("opts", [dict(), STAGED, dict(slot_index=1)], ids=["fused", "staged", "slot"])
def test_long_chains(opts):
    """A table filled to 0.97: chains of hundreds of slots, over its end."""
    spec = synth.VolumeSpec(0.01, 0.04, 1 << 12, 1 << 12)
    frames, n = [], 0
    ov = oracle_volume(spec)
    for i in range(200):
        fr = synth.random_frame(seed=100 + i, width=24, height=16)
        probe = oracle_volume(synth.VolumeSpec(0.01, 0.04, 1 << 14, 1 << 14))
        for g in frames + [fr]:
            assert probe.fuse_frame(g) == "OK"
        n = len(probe.export()[0])
        if n > 4000:
            continue
        frames.append(fr)
        if n > 3900:
            break
    assert n > 3900
    check(frames, spec, **opts)
    del ov
