"""The variances of a fit in an iteration in which a mean jumps: one component, whose first mean is a particle far from
all others, so that the new mean lies sqrt(N) standard deviations from the old one (the largest jump that the E-step
allows).  One iteration; the reference is the two-pass variance in extended precision.

Tolerance 2e-13: a sum of N squares about the mean has a rounding error of a few 1e-16 here (trees of partial sums); about the
old mean N times as much, 4e-12 at N = 32768, is cancelled away."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402
from oracle import gm, prior  # noqa: E402


@pytest.mark.parametrize("full", [0, 1])
@pytest.mark.parametrize("N,r", [(32768, 16), (32767, 5), (4099, 64)])
def test_variances_after_a_jump(full, N, r):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = inputs.load_workload("darcy64_bimodal")
    floor_frac = 1e-9
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=N, n_components=1, gm_rank=r, kl_modes=8, em_iters=1, full_cov=full, var_floor=floor_frac))
    modes = s.smc_get_mixture()[3]
    rng = np.random.default_rng(7)
    X = 1e-9 * rng.standard_normal((N, s.d))
    X[gm.init_indices(wl["seed"], 0, N, 1)[0]] = 30.0 + rng.standard_normal(s.d)
    s.smc_set_particles(X, np.zeros(N))
    s.smc_set_schedule(0.0, 0.2, 0, 0)
    s.gm_fit()
    _, m, lam, _ = s.smc_get_mixture()
    x = X[:, modes].astype(np.longdouble)
    mean = x.mean(0)
    var = ((x - mean) ** 2).mean(0)
    floor = floor_frac * prior.eigenvalues(2, 8, wl["alpha"])[modes]
    ref = var + floor if full else np.maximum(var, floor)
    assert np.max(np.abs(m[0] - mean) / np.abs(mean)) <= 1e-13
    assert np.max(np.abs(lam[0] - ref) / ref) <= 2e-13
    s.close()

