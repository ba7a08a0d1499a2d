"""CPU: the FP32-word form of far entries and point charges (three-word sums)
against the FP64 code that they stand for and an extended-precision sum, for
every class, odd and even record counts, coordinates on and off the grid.  Bound
of the words: the final FP64 conversion adds five numbers (4 x 2^-53 of the
result) and orders N >= 1 keep 48 bits, about 20 roundings of 2^-48 each of a
part that is at most the sum of absolute terms: 8e-14; for charges and L = 0
there is no such part, 5e-16."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.mark.parametrize("seed", [1, 2])
def test_words_against_extended_precision(seed, tmp_path):
    cxx = os.environ.get("CXX", "g++")
    if not shutil.which(cxx) or not os.path.exists(os.path.join(CUDA, "include", "vector_types.h")):
        pytest.skip("needs a C++ compiler and the CUDA headers")
    exe = str(tmp_path / "words_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(CUDA, "include"), "-I",
                    os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1011_4687_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "words_check.cpp")], check=True)
    out = subprocess.run([exe, str(seed)], check=True, capture_output=True, text=True).stdout
    rows = [line.split() for line in out.splitlines()]
    assert len(rows) == 30
    for cls, n, words, f64 in rows:
        exact = int(cls) in (0, 5)
        assert float(words) <= (5e-16 if exact else 8e-14), (cls, n, words, f64)
