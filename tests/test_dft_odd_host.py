"""The odd-frequency DFTs of the fused y/z pass and the DFTs with coprime factors (csrc/dft.cuh), compiled as host code,
against direct sums."""
import os
import shutil
import subprocess

import pytest


def test_odd_frequency_dfts_match_direct_sums(tmp_path, repo_root):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "check"
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", os.path.join(repo_root, "include"), "-I",
                        os.path.join(repo_root, "paper_1910_13844_gb300", "csrc"), "-x", "cu",
                        os.path.join(repo_root, "tests", "dft_odd_host_check.cu"), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    assert out.stdout.count("bound") == 22
