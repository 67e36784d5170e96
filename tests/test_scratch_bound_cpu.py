"""The allocation-free column solve's static scratch holds what every accepted
size addresses, by the rule of forms that the library's own sources give."""
import os
import shutil
import subprocess

import pytest

from c_harness import ROOT


def test_every_accepted_size_fits(tmp_path):
    gxx = shutil.which("g++")
    cuda_inc = "/usr/local/cuda/include"
    if gxx is None or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("no g++ or CUDA headers")
    exe = str(tmp_path / "scratch_bound_check")
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", cuda_inc,
                    "-I", os.path.join(ROOT, "paper_2608_21150_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "c", "scratch_bound_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out[0] == "ok" and int(out[1]) > 4_000_000, out
