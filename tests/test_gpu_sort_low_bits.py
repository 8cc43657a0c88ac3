"""The radix sort by the low bits of keys that carry something above them, as
the accepted matches do (the distance in the top six bits of a pair key of up
to 58): bits above the sorted ones must not order anything."""
import os
import shutil
import subprocess

import pytest

from paper_1111_7171_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    lib = build.build()
    exe = str(tmp_path_factory.mktemp("low_bits") / "low_bits_check")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-I", build.INCLUDE, "-I", build.CSRC,
                    os.path.join(HERE, "gpu_logic", "low_bits_check.cu"), "-o", exe, lib,
                    "-Xlinker", "-rpath", "-Xlinker", build.LIB_DIR], check=True, capture_output=True)
    return exe


# the one-block sort, its last size, the first of the tiled sort, many tiles
@pytest.mark.parametrize("n", [2, 1000, 8192, 8193, 70_001])
def test_bits_above_do_not_order(program, n):
    r = subprocess.run([program, str(n), str(n + 3)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
