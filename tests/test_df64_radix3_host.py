"""The float-pair radix-3 butterfly (fft_engine.cuh), on the CPU, bitwise against
its definition in normalised float-pair arithmetic: no rounding is left out.
No GPU: nvcc compiles host code only here."""
import os
import subprocess

from test_engine_host import BUILD, CSRC, HERE, _nvcc


def test_radix3_leaves_out_no_rounding():
    os.makedirs(BUILD, exist_ok=True)
    exe = os.path.join(BUILD, "df64_radix3_check")
    src = os.path.join(HERE, "df64_radix3_check.cu")
    subprocess.run([_nvcc(), "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I", CSRC, "-o", exe, src], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert int(out[0]) == 6000000 and int(out[1]) == 0, out
