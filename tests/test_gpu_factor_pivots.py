"""The Cholesky factor of the mixture covariances at the ends of FP64's range (tests/factor_pivots.cu)."""
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_pivots_over_the_range(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_16028_gb300 import build
    lib = os.path.dirname(build.build())
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "factor_pivots")
    b = subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe,
                        os.path.join(HERE, "factor_pivots.cu"), "-L" + lib, "-lsmcgm", "-Xlinker", "-rpath=" + lib], capture_output=True, text=True)
    assert b.returncode == 0, b.stderr[-3000:]
    run = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0 and "factor pivots ok" in run.stdout, run.stdout + run.stderr
