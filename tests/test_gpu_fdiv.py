"""GPU: the branch-free quotients of the series functions (csrc/fdiv.cuh) equal
the IEEE division for every argument of their ranges."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_argument(tmp_path):
    exe = str(tmp_path / "fdiv")
    from paper_2208_05795_gb300 import build
    subprocess.run([build.nvcc()] + build.ARCH + ["-std=c++17", "-O3", "-I", build.CSRC, "-I",
                    os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "fdiv_ref.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True, timeout=120).stdout
    rows = [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    assert [r[0] for r in rows] == [0, 0, 1, 2]
    assert all(n > 0 and bad == 0 for _, n, bad in rows), rows
