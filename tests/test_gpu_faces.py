"""The mixed set-up's strips of rows: populations on both sides of the rule that picks their height (8 rows for a few
particles, 32 when those fill the SMs) give the same potentials bit for bit, at every grid's walls.

Each cell goes through the same operations whatever the strip, so the comparison is exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402


@pytest.mark.parametrize("n,N", [(64, 620), (128, 160), (512, 11)])
def test_strip_height_does_not_change_the_solution(n, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = dict(inputs.load_workload("darcy64_bimodal"), n=n)
    out = []
    for batch in (0, 3):
        s = smcgm.Sampler(smcgm.make_config(wl, n_particles=N, n_components=1, gm_rank=4, solve_batch=batch, tile_kernel=0))
        out.append(s.particles()[1])
        s.close()
    assert np.array_equal(out[0], out[1])
