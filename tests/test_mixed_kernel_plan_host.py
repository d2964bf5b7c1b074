"""The plans the mixed-radix FFT kernels are compiled with (kernel_plan of
fft_mixed.cuh: radices up to 25), checked on the host without a GPU:
tests/native/mixed_kernel_plan_check.cu runs, for all 172 lengths, the index
arithmetic of every exchange (distinct places, every read finds its entry) and
checks the block's limits and the twiddle blocks."""
import pathlib
import shutil
import subprocess

import pytest

ROOT = pathlib.Path(__file__).resolve().parent.parent


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="needs nvcc")
def test_mixed_kernel_plans(tmp_path):
    exe = tmp_path / "mixed_kernel_plan_check"
    subprocess.run(["nvcc", "-std=c++17", "--expt-relaxed-constexpr", "-I",
                    str(ROOT / "paper_2310_16214_gb300" / "csrc"),
                    str(ROOT / "tests" / "native" / "mixed_kernel_plan_check.cu"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout
    assert out.stdout.startswith("OK 172 "), out.stdout
