"""The packed double-FP32 functions of csrc/df2.cuh on the host (no GPU): both
halves of every result equal those of the scalar functions of csrc/df.cuh,
whose error bounds tests/test_df_host.py proves, bit for bit; df_from gives the value of the
float conversions it replaces over its whole range."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_packed_functions_equal_the_scalar_ones(tmp_path):
    nvcc = next((c for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc"))
                 if c and os.path.exists(c)), None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = tmp_path / "df2_host_check"
    subprocess.check_call([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off",
                           "-I", os.path.join(ROOT, "paper_2306_15511_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "df2_host_check.cu"), "-o", str(exe)])
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["from", "0", "add", "0", "sub", "0", "mul", "0", "fma", "0"]
