"""A failure of the exact-slice product inside the MP2 step is a status, and the
call gives back what it allocated (tests/c/mp2_failure.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_a_failed_product_leaks_nothing(tmp_path):
    from paper_2412_18553_gb300 import build as B
    B.build()
    obj = os.path.join(B.BUILD, "mp2.cu.o")
    if not os.path.exists(obj):
        B.build(force=True)
    exe = str(tmp_path / "mp2_failure")
    r = subprocess.run(["g++", "-std=c++17", "-I", B.CSRC, "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(CUDA, "include"), os.path.join(ROOT, "tests", "c", "mp2_failure.cpp"), obj,
                        "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.stdout.split() == ["5", "0"], out.stdout + out.stderr
