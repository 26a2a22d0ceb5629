"""The multi-pass solvers by name (tile_kernel 2 and 3), which the default no longer runs on grids that are solved on chip:
in CUDA graphs against the host-driven loop (bit-identical, as tests/test_gpu_graph.py derives), and their
solutions and moves against the oracle.

Tolerance against the oracle 1e-9 relative, as in the other forward parity tests: the solvers stop at a relative residual
of 1e-10."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402
from oracle import problem as oproblem, smc as osmc, pcngm as opcngm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_16028_gb300 import build
    build.build()
    smcgm.load_library()


def _twins(name, **over):
    wl = inputs.load_workload(name)
    out = []
    for _ in range(2):
        s = smcgm.Sampler(smcgm.make_config(wl, **over))
        s.smc_temper_step()
        s.smc_resample()
        s.gm_fit()
        out.append(s)
    return out


@pytest.mark.parametrize("cases", [
    # 256^2: the TMA-staged finest level and three tiled levels, 7 launch-size buckets per stage
    [("darcy256_precision", dict(n_particles=64, tile_kernel=2))],
    # uneven branches with conditional nodes each: BF16 faces, FP64, warp tiles from global memory, beside an on-chip one
    [("darcy256_precision", dict(n=128, kl_modes=64, n_particles=40, tile_kernel=2, precision=smcgm.SMC_P_BF16SMOOTH_REFINE)),
     ("darcy64_bimodal", dict(n_particles=40, tile_kernel=2, precision=smcgm.SMC_P_FP64)),
     ("darcy64_bimodal", dict(n_particles=96, tile_kernel=3)),
     ("darcy64_bimodal", dict(n_particles=33))],
    # 512^2 by default: the V-cycle from 128^2 down on chip, which reads the active count on the device (4 buckets)
    [("darcy256_precision", dict(n=512, n_particles=13, solve_batch=12, precision=smcgm.SMC_P_BF16SMOOTH_REFINE))],
    [("darcy256_precision", dict(n=256, n_particles=12, precision=smcgm.SMC_P_FP64))],
], ids=["staged_256", "mixed_batch", "bf16_512", "fp64_256"])
def test_graph_equals_host_loop(cases):
    pairs = [_twins(name, n_components=2, **over) for name, over in cases]
    b = smcgm.Batch([g for _, g in pairs], steps=2)
    rates = b.move()
    for (h, g), r in zip(pairs, rates):
        acc, _ = h.smc_move(2)
        assert r == acc
        for x, y in zip(h.particles(), g.particles()):
            assert np.array_equal(x, y)
        assert h.smc_get_schedule() == g.smc_get_schedule()
    b.close()
    for h, g in pairs:
        h.close()
        g.close()


@pytest.mark.parametrize("n,precision,tile_kernel", [(64, 1, 2), (128, 1, 2), (128, 2, 2), (64, 0, 2), (256, 1, 2), (64, 1, 4)])
def test_solutions_and_a_move(n, precision, tile_kernel):
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n)
    prob = oproblem.from_workload(wl)
    N = 6
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=N, n_components=2, precision=precision, tile_kernel=tile_kernel))
    X, Phi = s.particles()
    W = torch.empty(N, n * n, dtype=torch.float64, device="cuda")
    P = torch.empty(N, dtype=torch.float64, device="cuda")
    s.smc_forward(torch.tensor(X, device="cuda"), P, W)
    for i in range(N if n < 256 else 1):
        w = prob.solve(X[i]).reshape(-1)
        assert np.linalg.norm(W[i].cpu().numpy() - w) <= 1e-9 * np.linalg.norm(w)
        phi = prob.potential(X[i])
        assert abs(P[i].item() - phi) <= 1e-9 * phi and P[i].item() == Phi[i]
    w, m, lam, modes = s.smc_get_mixture()
    m = np.random.default_rng(0).standard_normal(m.shape) * np.sqrt(lam)
    w = np.array([0.3, 0.7])
    s.smc_set_mixture(w, m, lam)
    s.smc_set_schedule(0.05, 0.3, 0, 0)
    s.smc_move(1)
    X2, _ = s.particles()
    diag = s.diagnostics()
    mix = opcngm.Mixture(modes, w, m, lam, prob.lam)
    for i in range(2 if n < 256 else 1):
        x, _, acc, la, _ = osmc.move_particle(X[i], Phi[i], mix, 0.3, 0.05, wl["seed"], i, 0, prob.potential)
        assert abs(la - diag["log_alpha"][i]) <= 1e-7 * max(1.0, abs(la)) and bool(acc) == bool(diag["accepted"][i])
        assert np.max(np.abs(X2[i] - x)) <= 1e-12 * np.max(np.abs(x))
    s.close()
