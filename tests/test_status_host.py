"""The waiting read of a volume's status on the host side (CPU): the library's own
objects linked with a runtime that only counts (fake_cudart.cpp). The status word
is read by a launch where the volume's device is current; with another device
current a launch would read one GPU's memory from another's, so the words are
copied, which works from any. An error that an earlier call of the program left
behind is neither returned nor cleared."""
import ctypes
import os
import re
import shutil
import subprocess

import pytest

from paper_2608_08287_gb300 import build as tb

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE = os.path.join(ROOT, "tests", "fake_cudart.cpp")


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    if shutil.which("g++") is None or shutil.which("nm") is None:
        pytest.skip("g++ or nm not found")
    tb.build_library()
    objs = [os.path.join(tb.BUILD, s.replace(".cu", ".o")) for s in tb.SOURCES]
    names = set(re.findall(r"U (_*cuda\w+)", subprocess.run(["nm", "-u", *objs], check=True,
                                                            capture_output=True, text=True).stdout))
    given = set(re.findall(r"\b(_*cuda\w+)\(", open(FAKE).read()))
    d = tmp_path_factory.mktemp("fake")
    rest = d / "rest.cpp"
    rest.write_text("".join(f'extern "C" int {n}() {{ return 0; }}\n' for n in sorted(names - given)))
    out = str(d / "libtsdf_fake.so")
    r = subprocess.run(["g++", "-shared", "-fPIC", "-w", "-Wl,-Bsymbolic", FAKE, str(rest), *objs,
                        "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    lib = ctypes.CDLL(out)
    lib.tsdf_volume_create.argtypes = [ctypes.c_float, ctypes.c_float, ctypes.c_uint32,
                                       ctypes.c_uint32, ctypes.c_void_p]
    for f in (lib.tsdf_volume_status, lib.tsdf_volume_destroy):
        f.argtypes = [ctypes.c_void_p, ctypes.c_void_p][:2 if f is lib.tsdf_volume_status else 1]
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


def test_launch_that_fails(L, volume):
    v, c = volume
    c.launch_error.value = 98
    assert L.tsdf_volume_status(v, None) == 8      # TSDF_ERR_CUDA
