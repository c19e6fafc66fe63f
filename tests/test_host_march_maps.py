"""The index functions of the column-marching kernels, on the CPU: the very
functions that the kernels call, compiled into a host program (no GPU call), with
the single lattice's planes per thread and with a batch's."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_kernels_index_functions(tmp_path):
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = cand if os.path.exists(cand) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "march_maps_check")
    src = os.path.join(HERE, "host", "march_maps_check.cu")
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-w", "-o", exe, src], check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    got = re.findall(r"(\S+) ok=(\d)", out)
    assert len(got) == 16, out
    assert all(ok == "1" for _, ok in got), out
