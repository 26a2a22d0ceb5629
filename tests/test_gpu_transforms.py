"""The cosine synthesis where the input ends early: two modes,
odd halves of them, and n/2 at every transform length.

Synthesis against the dense cosine sums: the network's secants, up to n / pi, multiply the rounding errors of its log2 n
levels, so n log2 n 2^-53 of the field's largest value per axis, with a margin of two."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402

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
