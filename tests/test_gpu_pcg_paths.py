"""The grid PCG with a block's share in and out of shared memory (tests/csrc/pcg_paths_check.cu, which checks
itself; linked with the library for what newton.cu calls)."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
PKG = os.path.join(os.path.dirname(HERE), "paper_2206_11009_gb300")


def test_shares_in_and_out_of_shared_memory(tmp_path):
    import __graft_entry__
    __graft_entry__.build()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "pcg_paths_check")
    lib = os.path.join(PKG, "_build")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I" + os.path.join(os.path.dirname(HERE), "include"), "-I" + os.path.join(PKG, "csrc"), "-o", exe,
                    os.path.join(HERE, "csrc", "pcg_paths_check.cu"), "-L" + lib, "-lotipm", "-Xlinker", "-rpath=" + lib],
                   check=True, capture_output=True, timeout=600)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    print(out.stdout)
    assert out.returncode == 0 and out.stdout.strip().endswith("OK"), out.stdout + out.stderr
