"""The mixture fit at the edges of its kernels against the oracle's EM: populations below, at and just
past a block's share, ranks that are not a multiple of four or of the padding, one component and
the most, and the sizes at which shared memory no longer holds the particles or the factor.

Tolerance 1e-7 as in the other EM parity tests: both sides sum in FP64, and EM amplifies 1e-16
differences in the sums by some orders over its iterations."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402
from oracle import problem as oproblem, gm as ogm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_16028_gb300 import build
    build.build()
    smcgm.load_library()


def _clusters(N, K, lam, seed):
    rng = np.random.default_rng(seed)
    c = rng.standard_normal((K, lam.size)) * np.sqrt(lam)
    return c[rng.integers(0, K, N)] + 0.6 * rng.standard_normal((N, lam.size)) * np.sqrt(lam)


@pytest.mark.parametrize("N,K,r,full", [(2, 1, 1, 0), (9, 2, 5, 0), (153, 3, 12, 0), (1217, 16, 33, 0), (5000, 2, 256, 0),
                                        (64, 1, 1, 1), (70, 2, 6, 1), (1300, 3, 33, 1), (900, 2, 160, 1), (900, 1, 164, 1)])
def test_fit_matches_oracle_em(N, K, r, full):
    wl = inputs.load_workload("darcy64_bimodal")
    iters = 6
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=N, n_components=K, gm_rank=r, em_iters=iters, full_cov=full))
    prob = oproblem.from_workload(wl)
    X = _clusters(N, K, prob.lam, 11 + N)
    s.smc_set_particles(X, np.zeros(N))
    ll = s.gm_fit()
    fit = ogm.fit_full if full else ogm.fit
    mix, hist = fit(X, prob.gm_modes(r), prob.lam, K, iters, wl["seed"], 0, var_floor=s.cfg.var_floor)
    w, m, lam, modes = s.smc_get_mixture()
    assert np.array_equal(modes, mix.S)
    assert np.allclose(w, mix.w, rtol=1e-7, atol=1e-12)
    assert np.linalg.norm(m - mix.m) <= 1e-7 * np.linalg.norm(mix.m)
    assert np.linalg.norm(lam - mix.lam) <= 1e-7 * np.linalg.norm(mix.lam)
    if full:
        assert np.linalg.norm(s.smc_get_mixture_cov() - mix.cov) <= 1e-7 * np.linalg.norm(mix.cov)
    assert abs(ll - hist[-1]) <= 1e-8 * abs(hist[-1])
    s.close()
