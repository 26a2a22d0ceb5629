"""The multi-pass solvers' CG application (tiles of 32 x 8 cells per warp) and FP64-accurate residual against the
oracle's sparse LU: grids of one and several tiles per row and of every wall position, FP64 and mixed precision.

Tolerance 1e-10 relative for w: the solver stops at a relative residual of 1e-10, which these operators turn
into an error of ~1e-13 (the bound of the other forward parity tests)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402
from oracle import problem as oproblem  # noqa: E402


@pytest.mark.parametrize("n,precision,tile_kernel", [(64, 0, 3), (64, 1, 3), (64, 1, 4), (128, 0, 3), (128, 1, 4), (256, 0, 0), (256, 1, 4), (512, 1, 0)])
def test_solve_matches_oracle(n, precision, tile_kernel):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n)
    N = 3
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=N, n_components=1, gm_rank=4, precision=precision, tile_kernel=tile_kernel))
    prob = oproblem.from_workload(wl)
    X, _ = s.particles()
    W = torch.empty(N, n * n, dtype=torch.float64, device="cuda")
    P = torch.empty(N, dtype=torch.float64, device="cuda")
    s.smc_forward(torch.tensor(X, device="cuda"), P, W)
    for i in range(N if n < 256 else 1):
        w = prob.solve(X[i]).reshape(-1)
        assert np.linalg.norm(W[i].cpu().numpy() - w) < 1e-10 * np.linalg.norm(w)
    s.close()
