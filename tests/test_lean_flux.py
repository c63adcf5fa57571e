"""The Riemann solvers of the FP64 kernels, which reach the same
fluxes with fewer operations, against the plain ones (tests/cuda/flux_check.cu,
built here with nvcc) on random faces: large and small jumps, supersonic
faces, vanishing fields, equal states and degenerate star states.  The
difference stays within 64 roundings times the conditioning of the star
states.  The reciprocals, roots and characteristic slopes of the same kernels
likewise."""
import json
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.mark.parametrize("where", ["host", pytest.param("device", marks=pytest.mark.gpu)])
def test_lean_solvers_match_the_plain_ones(tmp_path, where):
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc is not on the path")
    exe = str(tmp_path / "flux_check")
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                           "-I", os.path.join(ROOT, "paper_2606_12753_gb300", "csrc"),
                           "-o", exe, os.path.join(HERE, "cuda", "flux_check.cu")])
    out = subprocess.run([exe, where], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    for name, excess in json.loads(out.stdout.strip().splitlines()[-1]).items():
        assert excess <= 1.0, (name, excess)
