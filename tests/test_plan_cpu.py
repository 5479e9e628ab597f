"""How a lattice's steps are split into launches (plan.h), compiled for the
host and checked over sizes and storage types: strips and tiles cover the
lattice once and fit the kernels' limits, and the launches of n steps add up
to n (tests/native/plan_check.cu)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_plan_host_check(tmp_path):
    nvcc = shutil.which("nvcc")
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "plan_check")
    src = os.path.join(HERE, "native", "plan_check.cu")
    subprocess.run([nvcc, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-x", "cu", src, "-o",
                    exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout[-2000:]
