"""The 1D forward map at grid sizes around a block's 128 threads, odd ones, and the size from which its
arrays leave shared memory; and the moments for odd grids.

The reference is the oracle's system eliminated in extended precision: in FP64 the elimination itself
is off by the system's condition (~n^2) times 1e-16, 1e-10 at n = 8192, while the kernel's sums are
off by ~1e-15.  Tolerance 1e-11: the sums, amplified by the misfit's cancellation in Phi."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import smcgm  # noqa: E402
from oracle import observe, problem as oproblem, prior  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_16028_gb300 import build
    build.build()
    smcgm.load_library()


def _solve_extended(prob, x):
    L = np.longdouble
    n, K = prob.n, np.exp(prob.field(x)).astype(L)
    b = prob.f.astype(L) / (L(n) * L(n))
    c, y = [L(0)], [L(0)]
    for i in range(n - 1):
        den = K[i] + K[i + 1] - K[i] * c[-1]
        c.append(K[i + 1] / den)
        y.append((b[i] + K[i] * y[-1]) / den)
    w = [y[-1]]
    for i in range(n - 2, 0, -1):
        w.append(y[i] + c[i] * w[-1])
    return np.array(w[::-1]).astype(np.float64)


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
        w = _solve_extended(prob, X[i])
        assert np.linalg.norm(W[i].cpu().numpy() - w) <= 1e-11 * np.linalg.norm(w)
        phi = float(observe.potential(prob.observe(w), prob.data, prob.sigma))
        assert abs(Phi[i] - phi) <= 1e-11 * max(1.0, abs(Phi[i]))
        assert P[i].item() == Phi[i]
    mean, var, mg, vg = s.smc_posterior_moments(grid=True)
    U = prior.synthesize_1d(X, n, km)
    assert np.allclose(mean, X.mean(0), rtol=0, atol=1e-13) and np.allclose(var, X.var(0), rtol=1e-12, atol=1e-14)
    assert np.allclose(mg, U.mean(0), rtol=0, atol=1e-12) and np.allclose(vg, U.var(0), rtol=1e-11, atol=1e-12)
    s.close()
