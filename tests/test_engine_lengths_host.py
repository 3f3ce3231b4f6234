"""The line shapes of the lengths between powers of two and 3/2 of them, on the
CPU: engine_lengths_check.cu drives them through the exact stage code of
fft_engine.cuh against a long-double DFT, as test_engine_host.py does for the
others and with its bounds.  No GPU: nvcc compiles host code only here."""
import os
import subprocess

import pytest

from test_engine_host import BUILD, CSRC, HERE, TOL, _nvcc


@pytest.fixture(scope="module")
def errors():
    os.makedirs(BUILD, exist_ok=True)
    exe = os.path.join(BUILD, "engine_lengths_check")
    src = os.path.join(HERE, "engine_lengths_check.cu")
    deps = [src, os.path.join(HERE, "engine_host_check.cu")]
    deps += [os.path.join(CSRC, f) for f in ("fft_engine.cuh", "df64.cuh")]
    if not os.path.exists(exe) or os.path.getmtime(exe) < max(os.path.getmtime(d) for d in deps):
        subprocess.run([_nvcc(), "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I", CSRC, "-I", HERE, "-o", exe,
                        src], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return {name: float(val) for name, val in (line.split() for line in out.strip().splitlines())}


@pytest.mark.parametrize("tag,count", [("f32", 54), ("f64", 48), ("df64", 40)])
def test_new_lengths_match_direct_dft(errors, tag, count):
    mine = {n: e for n, e in errors.items() if "_%s_" % tag in n}
    assert len(mine) >= count, len(mine)
    assert not {n: e for n, e in mine.items() if not e <= TOL[tag]}
