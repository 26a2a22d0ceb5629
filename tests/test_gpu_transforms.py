"""The cosine transforms where the input (synthesis) or the used output (analysis) ends early: two modes,
odd halves of them, and n/2 at every transform length.

Synthesis against the dense cosine sums: the network's secants, up to n / pi, multiply the rounding errors of its log2 n
levels, so n log2 n 2^-53 of the field's largest value per axis, with a margin of two.  Analysis through the gradient of
the potential against the oracle's adjoint: both solve to a relative residual of 1e-10, so 1e-9."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402
from oracle import adjoint as oadjoint, problem as oproblem  # noqa: E402

SIZES = [(64, 2), (64, 6), (64, 30), (64, 32), (128, 2), (128, 64), (256, 34), (256, 128), (512, 10), (512, 256)]


def _sampler(n, km, precision, **kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n, kl_modes=km)
    return smcgm.Sampler(smcgm.make_config(wl, n_particles=3, n_components=1, gm_rank=4, precision=precision, **kw))


@pytest.mark.parametrize("n,km", SIZES)
def test_synthesis_of_early_ending_input(n, km):
    s = _sampler(n, km, smcgm.SMC_P_FP64)
    X, _ = s.particles()
    _, _, mg, vg = s.smc_posterior_moments(grid=True)
    k, x = np.arange(km), (np.arange(n) + 0.5) / n
    C = np.cos(np.pi * k[:, None] * x[None, :]) * np.where(k == 0, 1.0, np.sqrt(2.0))[:, None]
    U = np.einsum("pkl,ki,lj->pji", X.reshape(3, km, km), C, C, optimize=True)
    tol = 4 * n * np.log2(n) * 2.0 ** -53 * np.abs(U).max()
    assert np.abs(mg.reshape(n, n) - U.mean(0)).max() <= tol
    assert np.abs(vg.reshape(n, n) - U.var(0)).max() <= 4 * tol * np.abs(U).max()
    s.close()


@pytest.mark.parametrize("n,km", SIZES)
def test_analysis_of_early_ending_output(n, km):
    s = _sampler(n, km, smcgm.SMC_P_FP32_REFINE, gradient=1)
    X, _ = s.particles()
    Phi = torch.empty(3, dtype=torch.float64, device="cuda")
    G = torch.empty(X.shape, dtype=torch.float64, device="cuda")
    s.smc_gradient(torch.tensor(X, device="cuda"), Phi, G)
    prob = oproblem.from_workload(dict(inputs.load_workload("darcy64_bimodal"), n=n, kl_modes=km))
    _, grad, _, _ = oadjoint.potential_and_gradient_2d(prob, X[2])
    assert np.linalg.norm(G[2].cpu().numpy() - grad) <= 1e-9 * np.linalg.norm(grad)
    s.close()
