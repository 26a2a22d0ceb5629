"""The sums over a particle's cells in the on-chip mixed-precision solve, seen through its last decision: whether |b - A w|
has reached tol_outer |b|.  One refinement phase, whose result does not depend on tol_outer, is measured in extended
precision; the solve has to call itself converged with a tolerance 3e-8 above that residual and not with one 3e-8 below.

3e-8: the squares are added in FP32 within 256 cells only, with a relative error of ~1e-7 per partial sum at random, so
~1e-8 for the total of the 16 partial sums of a 64^2 grid, half of that for its root, and less for larger grids.
Sums or thresholds in FP32 throughout are off by up to 1e-7."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402
from oracle import problem as oproblem  # noqa: E402


def _relative_residual(prob, x, w):
    """|b - A w| / |b| by face fluxes."""
    L = np.longdouble
    n = prob.n
    k, w, b = np.exp(prob.field(x).astype(L)), w.reshape(n, n).astype(L), prob.f.astype(L) / (n * n)
    q = np.zeros_like(w)
    fx = 2 * k[:, 1:] * k[:, :-1] / (k[:, 1:] + k[:, :-1]) * (w[:, 1:] - w[:, :-1])
    fy = 2 * k[1:] * k[:-1] / (k[1:] + k[:-1]) * (w[1:] - w[:-1])
    q[:, 1:] += fx; q[:, :-1] -= fx; q[1:] += fy; q[:-1] -= fy
    for side in (np.s_[:, 0], np.s_[:, -1], np.s_[0, :], np.s_[-1, :]):
        q[side] += 2 * k[side] * w[side]
    return float(np.sqrt(np.sum((b - q) ** 2) / np.sum(b ** 2)))


@pytest.mark.parametrize("n", [64, 128, 256])
def test_convergence_is_decided_by_the_residual(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n)
    prob = oproblem.from_workload(wl)
    X = np.random.default_rng(n).standard_normal((6, prob.lam.size)) * np.sqrt(prob.lam)
    W = torch.empty(1, n * n, dtype=torch.float64, device="cuda")
    P = torch.empty(1, dtype=torch.float64, device="cuda")

    def solve(x, tol):
        s = smcgm.Sampler(smcgm.make_config(wl, n_particles=2, n_components=1, gm_rank=4, max_refine=1, tol_outer=tol))
        try:
            s.smc_forward(torch.tensor(x[None], device="cuda"), P, W)
            return True
        except smcgm.SMCError as e:
            assert e.status == smcgm.SMC_ENOCONV
            return False
        finally:
            s.close()

    for x in X:
        assert not solve(x, 1e-10)
        r = _relative_residual(prob, x, W[0].cpu().numpy())
        assert 1e-5 < r < 6e-4                            # one phase's reduction
        assert solve(x, r * (1 + 3e-8)) and not solve(x, r * (1 - 3e-8)), r
