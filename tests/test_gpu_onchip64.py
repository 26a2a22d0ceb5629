"""The on-chip FP64 solve (a block of 64^2, a cluster of 4 blocks of 128^2) against the oracle's sparse LU and,
bit for bit, against itself in other batches.

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


@pytest.mark.parametrize("n,fine,coarse,amp", [(64, 1, 2, 10.0), (64, 2, 1, 10.0), (64, 2, 2, 1e-30), (128, 1, 2, 10.0), (128, 2, 2, 1e25),
                                               (128, 1, 1, 10.0), (128, 2, 1, 10.0)])
def test_solve_matches_oracle(n, fine, coarse, amp):
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n, src_amp=amp)
    wl["data"] = wl["data"] * (amp / 10.0)
    wl["sigma"] = wl["sigma"] * (amp / 10.0)
    N = 3
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=N, n_components=1, gm_rank=4, fine_sweeps=fine, smooth_sweeps=coarse, precision=0,
                                        solve_batch=2))
    prob = oproblem.from_workload(wl)
    X, Phi = s.particles()
    W = torch.empty(N, n * n, dtype=torch.float64, device="cuda")
    P = torch.empty(N, dtype=torch.float64, device="cuda")
    s.smc_forward(torch.tensor(X, device="cuda"), P, W)
    for i in range(N):
        w = prob.solve(X[i])
        assert _rel(W[i].cpu().numpy(), w.reshape(-1)) < 1e-10
        phi = prob.potential(X[i])
        assert abs(Phi[i] - phi) <= 1e-10 * phi and P[i].item() == Phi[i]
    s.close()


@pytest.mark.parametrize("n", [64, 128])
def test_zero_source_gives_zero(n):
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n, src_amp=0.0)
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=2, n_components=1, gm_rank=4, precision=0))
    X, Phi = s.particles()
    W = torch.full((2, n * n), 7.0, dtype=torch.float64, device="cuda")
    P = torch.empty(2, dtype=torch.float64, device="cuda")
    s.smc_forward(torch.tensor(X, device="cuda"), P, W)
    assert torch.count_nonzero(W).item() == 0
    assert abs(Phi[0] - np.sum(wl["data"] ** 2) / (2 * wl["sigma"] ** 2)) <= 1e-12 * Phi[0]
    s.close()


@pytest.mark.parametrize("n,N", [(64, 155), (128, 41)])
def test_particles_do_not_depend_on_their_batch(n, N):
    """More particles than are resident at a time (152 blocks; 36 clusters) against the same ones in batches of 5."""
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n)
    out = []
    for b in (0, 5):
        s = smcgm.Sampler(smcgm.make_config(wl, n_particles=N, n_components=1, gm_rank=4, solve_batch=b, precision=0))
        out.append(s.particles())
        s.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("n,fine,coarse", [(256, 1, 2), (256, 2, 1)])
def test_vcycle_below_the_passes(n, fine, coarse):
    """Larger grids run their levels from 128^2 down on chip: the solution against the oracle, and a captured move
    (ragged solve batches of 3) bit for bit against the host loop's."""
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n)
    pair = [smcgm.Sampler(smcgm.make_config(wl, n_particles=7, n_components=1, gm_rank=4, precision=0, solve_batch=3, fine_sweeps=fine,
                                            smooth_sweeps=coarse)) for _ in range(2)]
    for s in pair:
        s.smc_temper_step()
        s.smc_resample()
        s.gm_fit()
    X, _ = pair[0].particles()
    W = torch.empty(7, n * n, dtype=torch.float64, device="cuda")
    P = torch.empty(7, dtype=torch.float64, device="cuda")
    pair[0].smc_forward(torch.tensor(X, device="cuda"), P, W)
    w = oproblem.from_workload(wl).solve(X[5]).reshape(-1)
    assert _rel(W[5].cpu().numpy(), w) < 1e-10
    b = smcgm.Batch([pair[1]], steps=1)
    acc, _ = pair[0].smc_move(1)
    assert b.move()[0] == acc
    for u, v in zip(pair[0].particles(), pair[1].particles()):
        assert np.array_equal(u, v)
    b.close()
    for s in pair:
        s.close()
