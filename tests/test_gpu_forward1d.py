"""The 1D forward map at grid sizes around a block's 128 threads, odd ones, and the size from which its
arrays leave shared memory, against the oracle's banded solve; and the moments for odd grids.

Tolerance 1e-11: sums of n terms in FP64 on both sides, amplified by the misfit's cancellation in Phi."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import smcgm  # noqa: E402
from oracle import problem as oproblem, prior  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_16028_gb300 import build
    build.build()
    smcgm.load_library()


@pytest.mark.parametrize("n,km", [(4, 2), (5, 2), (127, 30), (128, 64), (129, 64), (257, 64), (8192, 32), (8193, 32)])
def test_forward1d_and_moments(n, km):
    obs = np.array([0.0101, 0.25, 0.5, 0.77, 0.993])
    p = dict(dim=1, n=n, kl_modes=km, alpha=0.01, sigma=0.05, source_kind=1, src_amp=3.0, src_width=4.0, n_particles=3,
             n_components=1, gm_rank=1, beta0=0.2, ess_frac=0.5, seed=5, obs=obs, data=np.full(5, 0.1))
    s = smcgm.Sampler(smcgm.make_config(p))
    prob = oproblem.Problem(**{k: p[k] for k in ("dim", "n", "kl_modes", "alpha", "sigma", "source_kind", "src_amp", "src_width", "obs", "data")})
    X, Phi = s.particles()
    W = torch.empty(3, n - 1, dtype=torch.float64, device="cuda")
    P = torch.empty(3, dtype=torch.float64, device="cuda")
    s.smc_forward(torch.tensor(X, device="cuda"), P, W)
    for i in range(3):
        w = prob.solve(X[i])
        assert np.linalg.norm(W[i].cpu().numpy() - w) <= 1e-11 * np.linalg.norm(w)
        assert abs(Phi[i] - prob.potential(X[i])) <= 1e-11 * max(1.0, abs(Phi[i]))
        assert P[i].item() == Phi[i]
    mean, var, mg, vg = s.smc_posterior_moments(grid=True)
    U = prior.synthesize_1d(X, n, km)
    assert np.allclose(mean, X.mean(0), rtol=0, atol=1e-13) and np.allclose(var, X.var(0), rtol=1e-12, atol=1e-14)
    assert np.allclose(mg, U.mean(0), rtol=0, atol=1e-12) and np.allclose(vg, U.var(0), rtol=1e-11, atol=1e-12)
    s.close()
