"""smc_init with a prior whose fields leave the mixed solver's range |u| < 64: an error, not an abort (in a process of its
own)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import sys
sys.path.insert(0, %r)
from paper_2503_16028_gb300 import inputs, smcgm
smcgm.load_library()
for n, tk in ((64, 0), (64, 2), (512, 0)):
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n, alpha=1e-9)       # 1024 modes of unit variance: u ~ N(0, 32^2)
    try:
        smcgm.Sampler(smcgm.make_config(wl, n_particles=4, n_components=1, tile_kernel=tk))
        raise SystemExit("accepted")
    except smcgm.SMCError as e:
        assert e.status == smcgm.SMC_EINVAL and "64" in str(e), e
    s = smcgm.Sampler(smcgm.make_config(dict(wl, alpha=0.02), n_particles=4, n_components=1, tile_kernel=tk))   # and the GPU goes on
    s.close()
print("refused")
"""


def test_a_prior_outside_the_range_is_refused():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_16028_gb300 import build
    build.build()
    run = subprocess.run([sys.executable, "-c", PROGRAM % ROOT], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0 and "refused" in run.stdout, run.stdout + run.stderr
