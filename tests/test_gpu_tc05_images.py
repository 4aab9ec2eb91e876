"""The tcgen05 products in the shapes, layouts and loops that the library runs (`tc_images_check.cu`), bit for
bit: the pair product's main loop (two slots, 256 tensor-memory columns, image copies, partial tiles, K
not a multiple of 32) and the persistent chain kernel itself, several tiles per block."""
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_products_on_tile_images_are_exact(tmp_path):
    from paper_2407_06409_gb300 import build
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    exe = tmp_path / "tc_images_check"
    r = subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-o", str(exe),
                        os.path.join(HERE, "tc_images_check.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    lines = r.stdout.splitlines()
    assert len(lines) == 6 + 6 + 21 + 15 + 1 and lines[-1] == "all exact", r.stdout
