"""A launch that the runtime refuses is reported by the call and by nothing else:
the error does not stay behind for the caller's next check of its own (torch
makes one after every kernel).  No GPU: a stand-in refuses the launch."""
import os
import subprocess

from test_engine_host import BUILD, CSRC, HERE, _nvcc


def test_refused_launch_leaves_no_error_behind():
    os.makedirs(BUILD, exist_ok=True)
    exe = os.path.join(BUILD, "launch_error_check")
    src = os.path.join(HERE, "launch_error_check.cu")
    subprocess.run([_nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1",
                    "--expt-relaxed-constexpr", "-I", CSRC, "-o", exe, src], check=True)
    returned, left = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert int(returned) == 9  # cudaErrorInvalidConfiguration
    assert int(left) == 0, left
