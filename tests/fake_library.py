"""The library's own objects linked with a CUDA runtime that only counts
(fake_cudart.cpp), for host-side tests without a GPU."""
import ctypes
import os
import re
import shutil
import subprocess

import pytest

from paper_2608_08287_gb300 import build as tb

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE = os.path.join(ROOT, "tests", "fake_cudart.cpp")


def build(directory):
    """Path of the library, built in `directory` (a pathlib path)."""
    if shutil.which("g++") is None or shutil.which("nm") is None:
        pytest.skip("g++ or nm not found")
    tb.build_library()
    objs = [os.path.join(tb.BUILD, s.replace(".cu", ".o")) for s in tb.SOURCES]
    names = set(re.findall(r"U (_*cuda\w+)", subprocess.run(["nm", "-u", *objs], check=True,
                                                            capture_output=True, text=True).stdout))
    given = set(re.findall(r"\b(_*cuda\w+)\(", open(FAKE).read()))
    rest = directory / "rest.cpp"
    rest.write_text("".join(f'extern "C" int {n}() {{ return 0; }}\n' for n in sorted(names - given)))
    out = str(directory / "libtsdf_fake.so")
    r = subprocess.run(["g++", "-shared", "-fPIC", "-w", "-Wl,-Bsymbolic", FAKE, str(rest), *objs,
                        "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return out
