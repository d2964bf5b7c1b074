"""The run-time planner of the prime-radix FFT and the kernel's index
arithmetic for every length it serves, checked on the host without a GPU
(tests/native/prime_plan_check.cu)."""
import pathlib
import shutil
import subprocess

import pytest

ROOT = pathlib.Path(__file__).resolve().parent.parent


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="needs nvcc")
def test_prime_radix_plans(tmp_path):
    exe = tmp_path / "prime_plan_check"
    subprocess.run(["nvcc", "-std=c++17", "-O2", "-I", str(ROOT / "paper_2310_16214_gb300" / "csrc"),
                    str(ROOT / "tests" / "native" / "prime_plan_check.cu"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout
    assert out.stdout.strip() == "OK 1813", out.stdout
