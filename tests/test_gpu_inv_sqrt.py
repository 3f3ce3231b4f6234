"""The estimated inverse square root of the FP32 spectra's build (inv_sqrt.cuh), on
the device, against long double over the whole float range, past it and at its
ends."""
import os
import subprocess

import pytest

from test_engine_host import BUILD, CSRC, HERE, _nvcc

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_inv_sqrt_is_within_an_ulp_and_a_little():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    os.makedirs(BUILD, exist_ok=True)
    exe = os.path.join(BUILD, "inv_sqrt_check")
    subprocess.run([_nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O3", "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "inv_sqrt_check.cu")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.split()
    assert int(out[0]) > 1800000
    # half an ulp from the rounding of x w, half from the last sum, and the third-order term
    assert float(out[1]) <= 1.05, out
    # the library's rsqrt: one ulp
    assert float(out[2]) <= 1.05, out
