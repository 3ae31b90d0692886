"""Which kernels a call launches (CPU): the public calls against a CUDA runtime that
records launches (fake_cudart.cpp). A stage B strategy that a program has set is the one
that runs, beside every strategy of stage A, for volumes and both forms of a batch; where
none has been set it goes with stage A's."""
import ctypes

import numpy as np
import pytest

import fake_library
from paper_2608_08287_gb300 import tsdf


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    """The Python binding, on the library with the recording runtime."""
    path = fake_library.build(tmp_path_factory.mktemp("fake"))
    real, tsdf._lib = tsdf._lib, None
    load, ctypes.CDLL = ctypes.CDLL, lambda *a, **k: load(path)
    try:
        lib = tsdf.lib()
    finally:
        ctypes.CDLL = load
    lib.fake_launched.restype = ctypes.c_char_p
    yield lib
    tsdf._lib = real


def kernels(lib):
    """Short names of the kernels launched since the last look."""
    out = []
    for name in lib.fake_launched().decode().split():
        for k in ("integrate_scatter_kernel", "batch_scatter_kernel", "batch_tile_kernel",
                  "batch_point_kernel", "allocate_kernel", "warp_kernel", "tile_kernel"):
            if k in name:
                out.append(k)
                break
        else:
            out.append(name)
    return out


INTR, POSE = (60.0, 60.0, 32.0, 24.0), np.eye(4, dtype=np.float32)
STAGE_A = {0: "allocate_kernel", 1: "tile_kernel", 2: "warp_kernel"}
STAGE_B = {0: "integrate_scatter_kernel", 1: "warp_kernel", 2: "tile_kernel"}


@pytest.mark.parametrize("a", [0, 1, 2])
@pytest.mark.parametrize("b", [None, 0, 1, 2])
def test_stages_of_a_volume(L, a, b):
    v = tsdf.Volume(0.005, 0.02, 1 << 8, 1 << 7)
    assert v.set_option("fuse_mode", 0) == "OK" and v.set_option("allocate_mode", a) == "OK"
    if b is not None:
        assert v.set_option("integrate_mode", b) == "OK"
    kernels(L)
    assert tsdf.tsdf_fuse_frame_async(v.handle, 4096, 64, 48, INTR, POSE) == "OK"
    unset = STAGE_B[0 if a == 0 else 2]
    assert kernels(L) == [STAGE_A[a], unset if b is None else STAGE_B[b]]
    v.close()


@pytest.mark.parametrize("streams", [0, 2])
@pytest.mark.parametrize("b", [None, 0, 1])
def test_stages_of_a_batch(L, streams, b):
    vols = [tsdf.Volume(0.005, 0.02, 1 << 8, 1 << 7) for _ in range(3)]
    batch = tsdf.Batch(4, fuse_mode=0, batch_streams=streams)
    if b is not None:
        assert batch.set_option("integrate_mode", b) == "OK"
    frames = tsdf.make_frames([(v.handle, (4096, 64, 48), None, INTR, POSE) for v in vols])
    kernels(L)
    assert tsdf.tsdf_fuse_batch_async(batch.handle, frames) == "OK"
    if streams:
        want = ["tile_kernel", STAGE_B[2 if b is None else b]] * 3
    else:
        want = ["batch_tile_kernel", {None: "batch_tile_kernel", 0: "batch_scatter_kernel",
                                      1: "batch_point_kernel"}[b]]
    assert kernels(L) == want
    batch.close()
    for v in vols:
        v.close()


@pytest.mark.parametrize("load", [0, 1, 2])
@pytest.mark.parametrize("band,held", [(1, 5), (2, 5), (3, 9), (4, 9), (5, 9), (16, 9)])
def test_samples_held_by_stage_a(L, band, held, load):
    """Stage A walks its samples in rounds; a round is no longer than a narrow band needs."""
    v = tsdf.Volume(0.01, 0.01 * band, 1 << 8, 1 << 7)
    assert v.set_option("probe_load", load) == "OK"
    kernels(L)
    assert tsdf.tsdf_allocate_async(v.handle, 4096, 64, 48, INTR, POSE) == "OK"
    name = L.fake_launched().decode()
    assert f"tile_kernelILi0ELi{load}ELi{held}ELi1ELb{int(band > 4)}E" in name, name
    v.close()


@pytest.mark.parametrize("size,band,threads", [((640, 480), 1, 1), ((640, 480), 2, 1), ((640, 480), 3, 2),
                                               ((320, 240), 2, 2), ((480, 320), 2, 2), ((480, 336), 2, 1),
                                               ((1280, 720), 8, 1)])
def test_threads_of_stage_b(L, size, band, threads):
    """One thread a point above four 16x16 tiles an SM (of 152) at half bands 1 and 2."""
    v = tsdf.Volume(0.01, 0.01 * band, 1 << 8, 1 << 7)
    kernels(L)
    assert tsdf.tsdf_integrate_async(v.handle, 4096, *size, INTR, POSE) == "OK"
    name = L.fake_launched().decode()
    assert "tile_kernelILi1ELi0E" in name and f"ELi{threads}ELb" in name, name
    v.close()
