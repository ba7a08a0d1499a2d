"""CPU: the far form in FP32 words, one multipole order at a time (a product of an
s and a p function on one centre has no monopole): in the root mean square its
error is no larger than that of the FP64 code it stands for, and every order
keeps FP64's accuracy.  Bound 2.5e-16 of the sum of absolute terms: the
conversion of the sum adds 3 roundings of 2^-54 and the coefficients come from at
most 6 such operations, 3 x 5.6e-17 in the root mean square.  (48 bits would show
as 1e-15.)"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.mark.parametrize("seed", [1, 2])
def test_every_order_at_fp64_accuracy(seed, tmp_path):
    cxx = os.environ.get("CXX", "g++")
    if not shutil.which(cxx) or not os.path.exists(os.path.join(CUDA, "include", "vector_types.h")):
        pytest.skip("needs a C++ compiler and the CUDA headers")
    exe = str(tmp_path / "words_orders_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(CUDA, "include"), "-I",
                    os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1011_4687_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "words_orders_check.cpp")], check=True)
    out = subprocess.run([exe, str(seed)], check=True, capture_output=True, text=True).stdout
    rows = [line.split() for line in out.splitlines()]
    assert len(rows) == 15
    for L, order, words, f64 in rows:
        assert float(words) <= float(f64) and float(words) <= 2.5e-16, (L, order, words, f64)
