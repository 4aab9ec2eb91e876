"""Conversions between FP64 and float-float (`ff_check.cu`): 47 bits over the FP32 range, and numbers
that are not finite, or too large for FP32, never become finite ones."""
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_conversions(tmp_path):
    from paper_2407_06409_gb300 import build
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    exe = tmp_path / "ff_check"
    r = subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", "-o", str(exe),
                        os.path.join(HERE, "ff_check.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
