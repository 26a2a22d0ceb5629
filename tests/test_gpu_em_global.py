"""The diagonal fit of populations whose modes do not fit shared memory (its particles are read from global memory):
at 256 modes from about 8700 particles with 16 components and 14200 with one.  Against the oracle's EM at its
tolerance in the other EM tests, 1e-7."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_16028_gb300 import inputs, smcgm  # noqa: E402
from oracle import problem as oproblem, gm as ogm  # noqa: E402


@pytest.mark.parametrize("N,K,r", [(9200, 16, 256), (15001, 1, 256), (32768, 3, 129)])
def test_fit_from_global_memory(N, K, r):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    # the fit's shared memory with the particles in it, 200 KB at most (em_smem in csrc/gm.cu)
    per, pad = -(-N // min(152, -(-N // 8))), (r + 11) // 16 * 16 + 4
    assert 8 * (2 * K * pad + 2 * K * per + 3 * K + 40 + 512 + per * pad) > 200 * 1024
    wl = inputs.load_workload("darcy64_bimodal")
    iters = 3
    s = smcgm.Sampler(smcgm.make_config(wl, n_particles=N, n_components=K, gm_rank=r, em_iters=iters))
    prob = oproblem.from_workload(wl)
    # unit noise around K centres two apart in as many modes, the first particles of the components at the centres:
    # soft responsibilities and no component that runs empty (whose re-seeding hangs on ties of rounding)
    rng = np.random.default_rng(N)
    modes = prob.gm_modes(r)
    centre = np.zeros((K, prob.lam.size))
    centre[np.arange(K), modes[:K]] = 2.0
    X = centre[rng.integers(0, K, N)] + rng.standard_normal((N, prob.lam.size))
    X[ogm.init_indices(wl["seed"], 0, N, K)] = centre
    X = X * np.sqrt(prob.lam)
    s.smc_set_particles(X, np.zeros(N))
    ll = s.gm_fit()
    mix, hist = ogm.fit(X, prob.gm_modes(r), prob.lam, K, iters, wl["seed"], 0, var_floor=s.cfg.var_floor)
    w, m, lam, _ = s.smc_get_mixture()
    assert np.allclose(w, mix.w, rtol=1e-7, atol=1e-12)
    assert np.linalg.norm(m - mix.m) <= 1e-7 * np.linalg.norm(mix.m)
    assert np.linalg.norm(lam - mix.lam) <= 1e-7 * np.linalg.norm(mix.lam)
    assert abs(ll - hist[-1]) <= 1e-8 * abs(hist[-1])
    s.close()
