"""Forms of a call that the other GPU tests do not reach, against the CPU oracle
(blocks and weights exact, means within the tolerance of test_gpu_parity.py,
which is derived there)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

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
