"""The stopping decision of the iterative refinement on synthetic residual
histories: several contraction rates, one slow column among fast ones, and
histories that reach the level of FP32 rounding.  A host program, no GPU."""
import os
import subprocess

import pytest

from test_host_helpers import CSRC, ROOT, _nvcc


def test_refinement_stops_at_its_floor_only(tmp_path):
    nvcc = _nvcc()
    if not nvcc:
        pytest.skip("needs nvcc")
    exe = tmp_path / "refine_check"
    src = os.path.join(ROOT, "tests", "host", "refine_check.cpp")
    subprocess.run([nvcc, "-x", "cu", "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, src, "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    assert r.stdout.strip() == "ok"
