"""The integer form of the FP64 to float-float split gives the bits of the FP64 form (host build of the
same inline function): exponents over the whole range, ties, carries, zeros and special values."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_integer_split_matches_fp64_split(tmp_path):
    cc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "ff_from_double_check")
    subprocess.run([cc, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1611_05677_gb300", "csrc"), "-I",
                    os.path.join(ROOT, "include"), "-o", exe, os.path.join(ROOT, "tests", "ff_from_double_check.cu")],
                   check=True, capture_output=True, timeout=600)
    out = subprocess.run([exe, "400000"], capture_output=True, text=True, timeout=300)
    checked, bad = (int(v) for v in out.stdout.split())
    assert checked >= 2_000_000
    assert bad == 0 and out.returncode == 0, out.stdout
