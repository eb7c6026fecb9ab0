"""The cost estimate of the batch's lane assignment against measured solves
(host code, compiled with nvcc; no GPU needed)."""
import os
import subprocess

import pytest

from test_native_helpers import HERE, nvcc


def test_estimates_follow_the_measured_solves(tmp_path):
    exe = nvcc()
    if exe is None:
        pytest.skip("nvcc not found")
    out = str(tmp_path / "solve_cost")
    res = subprocess.run([exe, "-std=c++17", "-O2", "-o", out, os.path.join(HERE, "native", "solve_cost.cu")],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    run = subprocess.run([out], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0, run.stdout + run.stderr
