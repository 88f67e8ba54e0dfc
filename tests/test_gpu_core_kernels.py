"""The recompression cores on their own (tests/host/core_check.cu, linked against the
library): rank decisions of the basis kernel at singular values 1e-3 apart around
its threshold, orthogonality and range, for sketches in and beyond shared memory and
near both ends of the float range; the core kernel's ranks, orthogonality and
reconstruction in both storage forms, for cores of 1 to 56 columns."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_core_kernels(tmp_path):
    from paper_1712_08872_gb300 import _build
    lib = _build.build()
    exe = str(tmp_path / "core_check")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc] + _build.ARCH + ["-O2", "-std=c++17", "-I" + _build.INCLUDE,
                    "-I" + _build.CSRC, os.path.join(ROOT, "tests", "host", "core_check.cu"), lib,
                    "-Xlinker", "-rpath=" + os.path.dirname(lib), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
