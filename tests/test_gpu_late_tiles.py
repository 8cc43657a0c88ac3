"""Scans and sorts whose look-back never waits: every tile before a tile that
has not published its sum yet is summed again from the input, as a launch does
whose blocks do not run at the same time."""
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
    exe = str(tmp_path_factory.mktemp("late") / "prims_check")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-DPJ_LB_POLLS=0", "-I", build.INCLUDE, "-I", build.CSRC,
                    os.path.join(HERE, "gpu_logic", "prims_check.cu"), os.path.join(build.CSRC, "pj_prims.cu"),
                    "-o", exe, lib, "-Xlinker", "-rpath", "-Xlinker", build.LIB_DIR], check=True, capture_output=True)
    return exe


# two tiles, a few, more than a warp looks at in one step
@pytest.mark.parametrize("n", [4097, 70_001, 200_003])
def test_late_tiles_are_counted_again(program, n):
    r = subprocess.run([program, str(n), str(n + 7)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
