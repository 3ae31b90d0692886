"""The waiting read of a volume's status on the host side (CPU): the library's own
objects linked with a runtime that only counts (fake_cudart.cpp). The status word
is read by a launch where the volume's device is current; with another device
current a launch would read one GPU's memory from another's, and a stream of
another device takes no launch, so the words are copied, which works from any. An error that an earlier call of the program left
behind is neither returned nor cleared."""
import ctypes

import pytest

import fake_library


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    lib = ctypes.CDLL(fake_library.build(tmp_path_factory.mktemp("fake")))
    lib.tsdf_volume_create.argtypes = [ctypes.c_float, ctypes.c_float, ctypes.c_uint32,
                                       ctypes.c_uint32, ctypes.c_void_p]
    lib.tsdf_volume_status.argtypes = [ctypes.c_void_p] * 2
    lib.tsdf_volume_destroy.argtypes = [ctypes.c_void_p]
    lib.tsdf_volume_block_count.argtypes = [ctypes.c_void_p] * 3
    return lib


class Counts:
    def __init__(self, lib):
        self.lib = lib

    def __getattr__(self, name):
        return ctypes.c_int.in_dll(self.lib, "fake_" + name)


@pytest.fixture
def volume(L):
    c = Counts(L)
    c.device.value = 2
    v = ctypes.c_void_p()
    assert L.tsdf_volume_create(0.01, 0.04, 64, 32, ctypes.byref(v)) == 0
    for n in ("launches", "copies", "waits", "last_error", "launch_error"):
        getattr(c, n).value = 0
    yield v, c
    L.tsdf_volume_destroy(v)


def test_volume_device_current(L, volume):
    v, c = volume
    assert L.tsdf_volume_status(v, None) == 0
    assert (c.launches.value, c.copies.value, c.waits.value) == (1, 0, 1)


def test_other_device_current(L, volume):
    v, c = volume
    c.device.value = 0
    n = ctypes.c_uint32(7)
    assert L.tsdf_volume_status(v, None) == 0
    assert L.tsdf_volume_block_count(v, None, ctypes.byref(n)) == 0 and n.value == 0
    assert (c.launches.value, c.copies.value, c.waits.value) == (0, 2, 2)


def test_error_of_an_earlier_call(L, volume):
    v, c = volume
    c.last_error.value = 2          # an allocation of the program that failed
    assert L.tsdf_volume_status(v, None) == 0
    assert c.waits.value == 1 and c.last_error.value == 2


def test_stream_of_another_device(L, volume):
    v, c = volume
    c.launch_error.value = 400      # an invalid resource handle: not a stream of this device
    assert L.tsdf_volume_status(v, None) == 0
    assert (c.copies.value, c.waits.value, c.last_error.value) == (1, 1, 0)


def test_launch_that_fails(L, volume):
    v, c = volume
    c.launch_error.value = 98
    assert L.tsdf_volume_status(v, None) == 8      # TSDF_ERR_CUDA
