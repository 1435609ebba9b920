"""GPU: the sweeps' reciprocal without a slow path (rcp_rn) is the correctly rounded 1 / g.

The loops that use it and those that divide leave the same spectra, so it has to be the division's value
at every significand and sign and every exponent whose reciprocal is in FP32's normal range.
"""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reciprocal_equals_the_division(tmp_path):
    import torch
    so = str(tmp_path / "rcp.so")
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                           "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_1609_07936_gb300", "csrc"), "-o", so,
                           os.path.join(ROOT, "tests", "cuda", "rcp_rn_all.cu")])
    wrong = torch.zeros(1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert ctypes.CDLL(so).rcp_rn_all(-125, 125, ctypes.c_void_p(wrong.data_ptr())) == 0
    assert wrong.item() == 0
