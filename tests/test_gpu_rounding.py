"""Rounding of the FP64 reciprocal, reciprocal root and root of the FP64
kernels (tests/cuda/rounding_check.cu, built here with nvcc), which take two
or three operations of the FP64 pipe, against exact residuals and against the
plain ones, which take more.

Bounds on the largest error, in ulps: the last operation rounds by 1/2; the
reciprocal adds nothing else but the cube of its seed's error (below 0.02);
the reciprocal root forms x y, whose rounding moves it by up to 1/2 (0.25
m_y / m_x, m the mantissas of y and x y); the root's product moves it by up to
1/4 and its second-order term, in whole ulps, by up to 1/2, where the plain
form rounds its reciprocal root by 1 and the product by 1/2.  Neither the largest nor the mean error is above the plain
form's (sampling: one in a hundred, one in a thousand)."""
import json
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_short_forms_round_no_worse_than_the_plain_ones(tmp_path):
    exe = str(tmp_path / "rounding_check")
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                           "-I", os.path.join(ROOT, "paper_2606_12753_gb300", "csrc"), "-o", exe,
                           os.path.join(HERE, "cuda", "rounding_check.cu")])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    r = json.loads(out.stdout.strip().splitlines()[-1])
    print(r)
    for name, bound in (("rcp", 0.52), ("rsqrt", 1.02), ("root", 1.27)):
        assert r[name][0] <= bound, (name, r)
        assert r[name][0] <= r["plain_" + name][0] * 1.01, (name, r)
        assert r[name][1] <= r["plain_" + name][1] * 1.001, (name, r)
