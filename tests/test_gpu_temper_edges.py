"""The effective sample size that a tempering step reports when no step is possible: potentials that are not finite."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402


@pytest.mark.parametrize("N", [2, 257, 2500])
@pytest.mark.parametrize("bad", ["nan", "all_nan", "degenerate"])
def test_ess_without_a_step(N, bad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = inputs.load_workload("darcy64_bimodal")
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=N, n_components=1, gm_rank=4, kl_modes=4, ess_frac=1.0))
    X, Phi = s.particles()
    Phi = np.abs(np.random.default_rng(0).standard_normal(N))
    if bad == "nan":
        Phi[N // 2] = np.nan
    elif bad == "all_nan":
        Phi[:] = np.nan
    else:                       # no h above 0 keeps a target of N
        Phi[0] = 1e300
    s.smc_set_particles(X, Phi)
    h, ess, lz, done = ctypes.c_double(-1), ctypes.c_double(-1), ctypes.c_double(), ctypes.c_int()
    rc = s.lib.smc_temper_step(s.ctx, ctypes.byref(h), ctypes.byref(ess), ctypes.byref(lz), ctypes.byref(done))
    assert rc == smcgm.SMC_EDEGENERATE and h.value == 0.0
    assert ess.value == N if bad == "degenerate" else np.isnan(ess.value) and np.isnan(lz.value)
    s.close()
