"""The float-pair steps that must leave out no rounding (fft_engine.cuh), on the
CPU: the radix-3 butterfly bitwise against its definition in normalised
float-pair arithmetic, and the product with the spectrum, whose results must be
normalised pairs.  No GPU: nvcc compiles host code only here."""
import os
import subprocess

import pytest

from test_engine_host import BUILD, CSRC, HERE, _nvcc


@pytest.fixture(scope="module")
def counts():
    os.makedirs(BUILD, exist_ok=True)
    exe = os.path.join(BUILD, "df64_rounding_check")
    src = os.path.join(HERE, "df64_rounding_check.cu")
    subprocess.run([_nvcc(), "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I", CSRC, "-o", exe, src], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return {line.split()[0]: tuple(int(v) for v in line.split()[1:]) for line in out.strip().splitlines()}


def test_radix3_leaves_out_no_rounding(counts):
    assert counts["radix3"] == (6000000, 0)


def test_spectrum_product_is_normalised(counts):
    assert counts["product"] == (2000000, 0)
