"""The partition pass's bit-plane arithmetic (planes of elements of 1, 2 and 4
bytes, key counts, stable splits) on the host, against its definition element
by element: every number of bits, of levels and of elements."""
import os
import subprocess

from paper_1610_03524_gb300 import build as cuda_build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_planes_counts_and_splits(tmp_path):
    exe = str(tmp_path / "bitplane_check")
    r = subprocess.run([cuda_build.nvcc(), *cuda_build.ARCH, "-std=c++17", "-O1", "-I",
                        cuda_build.CSRC, os.path.join(HERE, "bitplane_check.cu"), "-o", exe],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
