"""The FP64 reciprocal and square root of two FP64 operations each
(csrc/fp64.cuh), compiled for the host: within half a unit of the result (and
2^-20 of one) over the exponent range, around powers of two and with the
hardware approximations off by up to two units; special values as documented."""
import os
import shutil
import subprocess

import pytest

from c_harness import ROOT


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    gxx = shutil.which("g++")
    cuda_inc = "/usr/local/cuda/include"
    if gxx is None or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("no g++ or CUDA headers")
    out = str(tmp_path_factory.mktemp("fp64") / "fp64_host")
    subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", cuda_inc,
                    "-I", os.path.join(ROOT, "paper_2608_21150_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "c", "fp64_host.cpp"), "-o", out], check=True)
    return out


@pytest.mark.parametrize("off", [-2, -1, 0, 1, 2])
def test_reciprocal_and_square_root(exe, off):
    out = subprocess.run([exe, str(off)], check=True, capture_output=True, text=True).stdout
    assert out.split() == ["0", "0"], out
