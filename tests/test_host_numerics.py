"""Host programs on numerical helpers of the CUDA engine, no GPU.

refine_check: the refinement's stopping decision on synthetic residual
histories: several contraction rates, one slow column among fast ones, and
histories that reach the level of FP32 rounding.  carry_check: the solution
update's additions with neighbours of equal and of very different magnitudes.
residual_check: the items and slots of the residual, with the usual memory and
with less.  sum_check: the Build epilogue's sums against FP64 ones.  alloc_check:
a buffer's capacity after a failed allocation."""
import os
import subprocess

import pytest

from test_host_helpers import CSRC, ROOT, _nvcc


@pytest.mark.parametrize("name", ["refine_check", "carry_check", "residual_check", "sum_check", "alloc_check"])
def test_on_the_host(tmp_path, name):
    nvcc = _nvcc()
    if not nvcc:
        pytest.skip("needs nvcc")
    exe = tmp_path / name
    src = os.path.join(ROOT, "tests", "host", name + ".cpp")
    subprocess.run([nvcc, "-x", "cu", "-std=c++17", "-O1", "-Xcompiler", "-ffp-contract=off", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I", CSRC, src, "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    assert r.stdout.strip().splitlines()[-1] == "ok"
