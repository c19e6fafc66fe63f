"""Index arithmetic of the Poisson solve's column-marching kernels, on the CPU,
compiled from the library's own headers into a host program (no GPU call):
every node in exactly one chunk, every coarse node written once from all its
children, neighbour offsets as the general neighbour function gives them."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_march_and_restriction_maps(tmp_path):
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = cand if os.path.exists(cand) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "march_check")
    src = os.path.join(HERE, "host", "march_check.cu")
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-w", "-o", exe, src], check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    got = re.findall(r"(\S+) ok=(\d)", out)
    assert len(got) == 17, out
    assert all(ok == "1" for _, ok in got), out
