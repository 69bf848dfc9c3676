"""The sweep's products on the integer units (csrc/ase_df_imul.cuh), compiled for the host against
the host's FP64 product: the same bits, ties and zeros included, over the ranges they are stated for."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2410_05489_gb300", "csrc")


def test_products_equal_the_fp64_unit(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    (tmp_path / "cuda_runtime.h").write_text("")  # the check defines the few intrinsics itself
    exe = str(tmp_path / "imul_check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", str(tmp_path), "-I", CSRC,
                    os.path.join(HERE, "imul_check.cpp"), "-o", exe], check=True, capture_output=True, text=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0, res.stdout + res.stderr
    assert res.stdout.startswith("ok 4002000 "), res.stdout
