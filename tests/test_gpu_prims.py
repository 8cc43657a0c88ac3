"""The device primitives (exclusive sum, stable radix sort) at the edges of
their tiles, against the host's standard library."""
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
    exe = str(tmp_path_factory.mktemp("prims") / "prims_check")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-I", build.INCLUDE, "-I", build.CSRC,
                    os.path.join(HERE, "gpu_logic", "prims_check.cu"), "-o", exe, lib,
                    "-Xlinker", "-rpath", "-Xlinker", build.LIB_DIR], check=True, capture_output=True)
    return exe


# one item; a warp's edge; the radix tile (4096), the one-block sort (8192)
# and scan (16384) with one less, one more; many tiles with a remainder
@pytest.mark.parametrize("n", [1, 31, 33, 4095, 4096, 4097, 8191, 8192, 8193, 16383, 16384, 16385, 70_001, 1_200_003])
def test_primitives_match_the_host(program, n):
    r = subprocess.run([program, str(n), str(n + 7)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
