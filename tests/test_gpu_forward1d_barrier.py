"""The 1D forward map behind barriers of very low permeability, where the flux through the barrier is small and its
resistance huge: one cell, neighbours, two apart, at the walls and the middle, for sources of either sign and one that
fades towards the walls.  Reference: the system's solution in 50 decimal digits and more for the same field.

Tolerance 2e-12 relative to the largest value: the field (64 or 128 products of order 5) is rounded by ~4e-14, which
e^u passes on to w in full; the sums themselves add ~1e-15."""
from decimal import Decimal, getcontext

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import smcgm  # noqa: E402
from oracle import problem as oproblem  # noqa: E402


def _exact(u, f):
    getcontext().prec = 50 + int(-0.5 * min(u))           # beyond the digits that the largest resistance takes
    n = len(u)
    R = [(-Decimal(float(x))).exp() for x in u]
    B = [Decimal(0)]
    for x in f:
        B.append(B[-1] + Decimal(float(x)) / (n * n))
    g = sum(b * r for b, r in zip(B, R)) / sum(R)
    w = [Decimal(0)]
    for b, r in zip(B, R):
        w.append(w[-1] + (g - b) * r)
    return np.array([float(x) for x in w[1:n]])


CELLS = {"first": [0], "second": [1], "below_middle": [-2], "middle": [-1], "last": [-3], "pair": [20, 21], "apart": [11, 40], "walls": [0, -3]}


@pytest.mark.parametrize("n", [64, 128])
@pytest.mark.parametrize("amp,kind,width", [(10.0, 0, 0.0), (-3.0, 1, 4.0), (10.0, 1, 200.0)])
def test_barriers(n, amp, kind, width):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    obs = np.array([0.02, 0.26, 0.5, 0.77, 0.993])
    p = dict(dim=1, n=n, kl_modes=n, alpha=0.01, sigma=0.05, source_kind=kind, src_amp=amp, src_width=width, n_particles=2,
             n_components=1, gm_rank=1, beta0=0.2, ess_frac=0.5, seed=5, obs=obs, data=np.zeros(5))
    prob = oproblem.Problem(**{k: p[k] for k in ("dim", "n", "kl_modes", "alpha", "sigma", "source_kind", "src_amp", "src_width", "obs", "data")})
    basis = prob.field(np.eye(n))                              # rows: the fields of the unit vectors
    rng = np.random.default_rng(3)
    X = []
    for name, cells in CELLS.items():
        for depth in (20.0, 30.0):
            u = 0.5 * rng.standard_normal(n)
            for c in cells:
                u[{-1: n // 2, -2: n // 2 - 1, -3: n - 1}.get(c, c)] = -depth
            X.append(np.linalg.solve(basis.T, u))
    X = np.array(X)
    s = smcgm.Sampler(smcgm.make_config(p))
    W = torch.empty(len(X), n - 1, dtype=torch.float64, device="cuda")
    P = torch.empty(len(X), dtype=torch.float64, device="cuda")
    s.smc_forward(torch.tensor(X, device="cuda"), P, W)
    for i in range(len(X)):
        w = _exact(prob.field(X[i]), prob.f)
        assert np.max(np.abs(W[i].cpu().numpy() - w)) <= 2e-12 * np.max(np.abs(w)), (i, list(CELLS)[i // 2])
        y = prob.observe(w)
        phi = float(y @ y) / (2 * p["sigma"] ** 2)
        assert abs(P[i].item() - phi) <= 1e-11 * phi, (i, list(CELLS)[i // 2])
    s.close()


@pytest.mark.parametrize("low", [590.0, 610.0, 705.0, 720.0])
def test_fields_below_the_range_of_the_exponential(low):
    """e^{-u} beyond 1.8e308 in one cell, and in all of them with a source small enough for w to fit.  Tolerance 5e-11: the
    field's rounding, 64 products of up to 700, is ~5e-12 in the worst case."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 64
    p = dict(dim=1, n=n, kl_modes=n, alpha=0.01, sigma=0.05, source_kind=0, src_amp=1e-12, src_width=0.0, n_particles=2,
             n_components=1, gm_rank=1, beta0=0.2, ess_frac=0.5, seed=5, obs=np.array([0.5]), data=np.zeros(1))
    prob = oproblem.Problem(**{k: p[k] for k in ("dim", "n", "kl_modes", "alpha", "sigma", "source_kind", "src_amp", "src_width", "obs", "data")})
    basis = prob.field(np.eye(n))
    one = np.zeros(n)
    one[20] = -low
    X = np.array([np.linalg.solve(basis.T, u) for u in (one, np.full(n, -low))])
    s = smcgm.Sampler(smcgm.make_config(p))
    W = torch.empty(2, n - 1, dtype=torch.float64, device="cuda")
    P = torch.empty(2, dtype=torch.float64, device="cuda")
    s.smc_forward(torch.tensor(X, device="cuda"), P, W)
    for i in range(2):
        w = _exact(prob.field(X[i]), prob.f)
        assert np.max(np.abs(W[i].cpu().numpy() - w)) <= 5e-11 * np.max(np.abs(w)), i
    s.close()
