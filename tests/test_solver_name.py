"""smc_solver names the kernel that solves a context's problems, and bench.py takes its word for it."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402
from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402


def test_bench_goes_by_the_solvers_name():
    # an FP64 solve on chip moves 40 bytes per cell, and a pass may happen to move 24
    prof = dict(word_bytes=4, cells=65536, solves=100, cg_iterations=1471, inner_solves=315.5, residuals=315.5, dom_particles=100)
    for solver, per_cell in (("k_onchip<4>", 24.0), ("k_onchip64<2>", 40.0), ("passes", 24.0)):
        p = dict(prof, solver=solver, dom_bytes=per_cell * 100 * 65536)
        assert bench.on_chip(p) == solver.startswith("k_onchip")
        assert (bench.model_bytes_per_solve(p, 256, 16384) < 1e7) == bench.on_chip(p)


@pytest.mark.gpu
@pytest.mark.parametrize("over,name", [(dict(), "k_onchip<1>"), (dict(n=128), "k_onchip<2>"), (dict(n=256), "k_onchip<4>"), (dict(n=512), "passes"),
                                       (dict(precision=0), "k_onchip64<1>"), (dict(n=128, precision=0), "k_onchip64<2>"),
                                       (dict(n=256, precision=0), "passes"), (dict(tile_kernel=2), "passes")])
def test_names(over, name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = dict(inputs.load_workload("darcy64_bimodal"), **over)
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=2, n_components=1, gm_rank=4))
    assert s.smc_solver() == name
    s.smc_profile_query(enable=1, reset=True)
    s.smc_forward(*(torch.tensor(a, device="cuda") for a in s.particles()))
    launches = s.smc_profile_query(enable=0, reset=True)["dom_launches"]
    assert (launches == 1) == name.startswith("k_onchip")       # one launch for all phases and iterations
    s.close()
