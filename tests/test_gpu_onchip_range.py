"""Fields shifted as a whole towards the ends of the mixed solver's range: the solution scales by e^-u0, while r.z and p.Ap of
the on-chip solve scale by e^-u0 too and reach FP32's subnormal numbers.  Tolerance 1e-10, that of the other forward tests: both
solutions meet the same residual."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402


@pytest.mark.parametrize("n,shifts", [(64, (-50.0, -30.0, 30.0, 40.0, 50.0)), (128, (-50.0, 40.0, 50.0)), (256, (-50.0, 30.0, 40.0, 45.0))])
def test_shifted_fields(n, shifts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n)
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=2, n_components=1, gm_rank=4))
    x0 = s.particles()[0][0]
    X = np.array([x0 + np.eye(1, x0.size)[0] * u0 for u0 in (0.0,) + shifts])      # mode 0 is the constant one
    W = torch.empty(len(X), n * n, dtype=torch.float64, device="cuda")
    P = torch.empty(len(X), dtype=torch.float64, device="cuda")
    s.smc_forward(torch.tensor(X, device="cuda"), P, W)
    W = W.cpu().numpy()
    for w, u0 in zip(W[1:], shifts):
        assert np.linalg.norm(w * np.exp(u0) - W[0]) <= 1e-10 * np.linalg.norm(W[0]), u0
    s.close()
