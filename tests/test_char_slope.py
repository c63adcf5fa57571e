"""The FP64 characteristic half slope with a small transverse field, where
the plain form's own roots cancel, against long double roots that do not
(tests/cuda/slope_check.cu, built here with nvcc).  A slope that is not a
number fails, and so does one whose smaller wave strength is lost: planted on
the host, both must."""
import json
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2606_12753_gb300", "csrc")


def _check(tmp_path, where, include=CSRC):
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc is not on the path")
    exe = str(tmp_path / "slope_check")
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", include,
                           "-o", exe, os.path.join(HERE, "cuda", "slope_check.cu")])
    out = subprocess.run([exe, where], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    return json.loads(out.stdout.strip().splitlines()[-1])


@pytest.mark.parametrize("where", ["host", pytest.param("device", marks=pytest.mark.gpu)])
def test_small_transverse_fields(tmp_path, where):
    r = _check(tmp_path, where)
    print(r)
    assert len(r) == 12 and max(r.values()) <= 1.0, r


@pytest.mark.parametrize("mistake", [("small = quarter_(q) * qrcp_(big)", "small = 0.0 * big"),
                                     ("slope[0] = rho * w + dc[3];", "slope[0] = (rho * w + dc[3]) * (0.0 / 0.0);")])
def test_planted_mistakes_are_seen(tmp_path, mistake):
    text = open(os.path.join(CSRC, "physics.cuh")).read()
    assert text.count(mistake[0]) == 1
    (tmp_path / "physics.cuh").write_text(text.replace(*mistake))
    r = _check(tmp_path, "host", str(tmp_path))
    assert min(r.values()) > 1.0, r
