"""The integer conversion of doubles to float pairs (df64.cuh), on the CPU,
against the FP64 arithmetic it stands in for: bitwise, special values and
range edges included.  No GPU: nvcc compiles host code only here."""
import os
import subprocess

from test_engine_host import BUILD, CSRC, HERE, _nvcc


def test_integer_conversion_matches_fp64_arithmetic():
    os.makedirs(BUILD, exist_ok=True)
    exe = os.path.join(BUILD, "df64_convert_check")
    src = os.path.join(HERE, "df64_convert_check.cu")
    subprocess.run([_nvcc(), "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I", CSRC, "-o", exe, src], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert int(out[0]) > 8000000 and int(out[1]) == 0, out
