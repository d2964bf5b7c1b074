"""Tables copied to the device are on it when the copying call returns
(tests/native/upload_check.cpp against a stand-in for the CUDA runtime), and
every table goes through that call."""
import os
import pathlib
import re
import shutil
import subprocess

import pytest

ROOT = pathlib.Path(__file__).resolve().parent.parent
CSRC = ROOT / "paper_2310_16214_gb300" / "csrc"


def test_no_unwaited_upload():
    for p in sorted(CSRC.glob("*.cu")):
        assert not re.search(r"\bcudaMemcpy\s*\(", p.read_text()), p.name


@pytest.mark.skipif(shutil.which("nvcc") is None or shutil.which("g++") is None, reason="needs g++ and CUDA's headers")
def test_upload_waits(tmp_path):
    cuda = pathlib.Path(os.path.realpath(shutil.which("nvcc"))).parent.parent / "include"
    exe = tmp_path / "upload_check"
    subprocess.run(["g++", "-std=c++17", "-x", "c++", "-I", str(cuda), "-I", str(CSRC), "-I", str(ROOT / "include"),
                    str(CSRC / "upload.cu"), str(ROOT / "tests" / "native" / "upload_check.cpp"), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.strip() == "OK", out.stdout
