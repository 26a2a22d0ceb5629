"""The on-chip mixed-precision solve (default tile kernels) against the oracle's sparse LU: every block
grid (one block, 2 x 2, 4 x 4 blocks per particle), one and two sweeps, sources scaled to the ends of
the FP32 range, a zero source, and populations that leave the last wave nearly empty.

Tolerance 1e-10 relative for w and Phi: the solver stops at a relative residual of 1e-10, which these
operators turn into an error of ~1e-13 (the bound of the other forward parity tests)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402
from oracle import problem as oproblem  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_16028_gb300 import build
    build.build()
    smcgm.load_library()


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n,fine,coarse,amp,precision", [(64, 1, 2, 10.0, 1), (64, 2, 1, 10.0, 1), (64, 1, 2, 1e-30, 1), (64, 1, 2, 1e25, 1),
                                                         (128, 1, 2, 10.0, 2), (128, 2, 2, 10.0, 1), (128, 1, 1, 1e-20, 1),
                                                         (256, 1, 2, 10.0, 1), (256, 2, 1, 10.0, 2)])
def test_solve_matches_oracle(n, fine, coarse, amp, precision):
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n, src_amp=amp)
    wl["data"] = wl["data"] * (amp / 10.0)
    wl["sigma"] = wl["sigma"] * (amp / 10.0)
    N = 3
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=N, n_components=1, gm_rank=4, fine_sweeps=fine, smooth_sweeps=coarse,
                                        precision=precision, solve_batch=2))
    prob = oproblem.from_workload(wl)
    X, Phi = s.particles()
    W = torch.empty(N, n * n, dtype=torch.float64, device="cuda")
    P = torch.empty(N, dtype=torch.float64, device="cuda")
    s.smc_forward(torch.tensor(X, device="cuda"), P, W)
    for i in range(N if n < 256 else 1):
        w = prob.solve(X[i])
        assert _rel(W[i].cpu().numpy(), w.reshape(-1)) < 1e-10
        phi = prob.potential(X[i])
        assert abs(Phi[i] - phi) <= 1e-10 * phi and P[i].item() == Phi[i]
    s.close()


@pytest.mark.parametrize("n", [64, 128, 256])
def test_zero_source_gives_zero(n):
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n, src_amp=0.0)
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=2, n_components=1, gm_rank=4))
    X, Phi = s.particles()
    W = torch.full((2, n * n), 7.0, dtype=torch.float64, device="cuda")
    P = torch.empty(2, dtype=torch.float64, device="cuda")
    s.smc_forward(torch.tensor(X, device="cuda"), P, W)
    assert torch.count_nonzero(W).item() == 0
    assert abs(Phi[0] - np.sum(wl["data"] ** 2) / (2 * wl["sigma"] ** 2)) <= 1e-12 * Phi[0]
    s.close()


def test_particles_do_not_depend_on_their_batch():
    """307 particles (one more than the blocks resident at a time is a part wave) against the same ones in
    batches of 5: bit-identical."""
    wl = inputs.load_workload("darcy64_bimodal")
    out = []
    for b in (0, 5):
        s = smcgm.Sampler(smcgm.make_config(wl, n_particles=307, n_components=1, gm_rank=4, solve_batch=b))
        out.append(s.particles())
        s.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("fine,coarse", [(1, 2), (2, 1)])
def test_vcycle_below_the_passes(fine, coarse):
    """512^2 runs its levels from 128^2 down on chip (populations in ragged solve batches)."""
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=512)
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=7, n_components=1, gm_rank=4, solve_batch=3, fine_sweeps=fine, smooth_sweeps=coarse))
    X, _ = s.particles()
    W = torch.empty(7, 512 * 512, dtype=torch.float64, device="cuda")
    P = torch.empty(7, dtype=torch.float64, device="cuda")
    s.smc_forward(torch.tensor(X, device="cuda"), P, W)
    w = oproblem.from_workload(wl).solve(X[5]).reshape(-1)
    assert _rel(W[5].cpu().numpy(), w) < 1e-10
    s.close()
