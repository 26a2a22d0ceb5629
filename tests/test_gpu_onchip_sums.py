"""The sums over a particle's cells in the on-chip mixed-precision solver (tests/onchip_sums.cu): no error beyond that of
FP32 sums over 256 cells.  The bound there, 2^-36 of the largest such sum, is that of up to 128 fixed-point terms that keep 44 bits."""
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_sums(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_16028_gb300 import build
    lib = os.path.dirname(build.build())
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "onchip_sums")
    b = subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe,
                        os.path.join(HERE, "onchip_sums.cu"), "-L" + lib, "-lsmcgm", "-Xlinker", "-rpath=" + lib], capture_output=True, text=True)
    assert b.returncode == 0, b.stderr[-3000:]
    run = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0 and "on-chip sums ok" in run.stdout, run.stdout + run.stderr
