"""The work this library is used for, as cases that can be timed: single moves and whole tempering
layers of SMC-pCN-GM, forward solves, adjoint gradients, the mixture fit, reweighting and
resampling, posterior moments, and a batch of uneven problems in one CUDA graph; from the 1D
problem and a handful of 64^2 solves up to the 256^2 problem with 4096 particles.

``prepare`` makes a problem (observations, data, particles, mixture) from a seed and sets up the
sampler; ``run`` puts the particles and the schedule back to that state and takes one pass through
the public calls; ``exact`` computes what ``run`` returns with plain numpy and torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_2503_16028_gb300 import smcgm

DEV = "cuda:0"
F64 = torch.float64
PRECISIONS = {"fp64": smcgm.SMC_P_FP64, "fp32": smcgm.SMC_P_FP32_REFINE, "bf16": smcgm.SMC_P_BF16SMOOTH_REFINE}
KERNELS = {"pcn": smcgm.SMC_K_PCN, "pcn_gm": smcgm.SMC_K_PCN_GM, "gm_indep": smcgm.SMC_K_GM_INDEP}
EM_ITERS, VAR_FLOOR, BETA, ESS = 50, 1e-3, 0.2, 0.5
# Floating-point operations per grid cell of one solve to 1e-10: about 14 multigrid-preconditioned CG
# iterations of some 100 operations (all levels), the synthesis and the refinement residuals.
SOLVE_FLOPS = 1500.0
# Grid problems of the batch cases: (grid, share of the case's particles).
BATCH_PARTS = ((64, 1.0), (128, 0.25), (256, 0.25), (512, 0.0625), (64, 0.3))


def listed():
    """The cases; the sizes are those of this repository's workloads unless said otherwise."""
    two_d = dict(dim=2, alpha=0.02, kernel="pcn_gm", rank=64)
    return [
        # A whole tempering layer of the 1D problem: the smallest inverse problem, all latency.
        dict(name="layer_1d", kind="layer", dim=1, n=128, km=64, alpha=0.01, particles=256, components=2, rank=64,
             obs=20, sigma=0.01, precision="fp64", kernel="pcn_gm", steps=5),
        # A few forward solves at 64^2 with their solutions: a MAP estimate's or a plot's call.
        dict(two_d, name="forward_64_few", kind="forward", n=64, km=32, particles=16, components=1, obs=16, sigma=0.005,
             precision="fp32"),
        # A whole tempering layer of the bimodal 64^2 problem: reweight, resample, fit, ten moves.
        dict(two_d, name="layer_64", kind="layer", n=64, km=32, particles=1024, components=4, obs=16, sigma=0.005,
             precision="fp32", steps=10),
        # The moves of such a layer in FP64, the arithmetic of a reference run.
        dict(two_d, name="move_64_fp64", kind="move", n=64, km=32, particles=1024, components=4, obs=16, sigma=0.005,
             precision="fp64", steps=10),
        # The potential and its gradient for a population: what each Langevin step or a MAP search asks for.
        dict(two_d, name="gradient_128", kind="gradient", n=128, km=64, particles=2048, components=1, obs=64, sigma=0.01,
             precision="fp32"),
        # One move of the 256^2 problem in mixed precision: the bulk of a production run.
        dict(two_d, name="move_256", kind="move", n=256, km=128, particles=4096, components=8, obs=64, sigma=0.01,
             precision="bf16", steps=1),
        # The same problem in FP64, on a smaller population: the check of a mixed-precision run.
        dict(two_d, name="move_256_fp64", kind="move", n=256, km=128, particles=256, components=8, obs=64, sigma=0.01,
             precision="fp64", steps=1),
        # The finest grid of a mesh-refinement study, with FP32 smoothing and a ragged population.
        dict(two_d, name="move_512", kind="move", n=512, km=64, particles=250, components=4, obs=128, sigma=0.01,
             precision="fp32", steps=1),
        # Independent problems of uneven grids moved by one graph launch.
        dict(two_d, name="batch_uneven", kind="batch", n=0, km=32, particles=1024, components=4, obs=48, sigma=0.01,
             precision="fp32", steps=2),
        # The mixture fit with full covariances on a large population.
        dict(two_d, name="fit_full", kind="fit", n=64, km=32, particles=4096, components=8, obs=16, sigma=0.005,
             precision="fp32", full_cov=True),
        # Reweighting and resampling of a large population.
        dict(two_d, name="reweight_8192", kind="reweight", n=64, km=32, particles=8192, components=1, obs=16, sigma=0.005,
             precision="fp32"),
        # The posterior summary at the end of a 256^2 run: KL moments and the pointwise mean and variance.
        dict(two_d, name="moments_256", kind="moments", n=256, km=128, particles=4096, components=1, obs=64, sigma=0.01,
             precision="fp32"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the same kinds: sizes over the logarithm of their range, odd ones among them."""
    kind = rng.choice(["move", "move", "move", "layer", "forward", "gradient", "fit", "reweight", "moments", "batch"])
    c = dict(kind=kind, dim=2, alpha=0.02, obs=_log_int(rng, 4, 256), sigma=round(rng.uniform(0.002, 0.02), 4),
             kernel="pcn_gm", components=rng.randint(1, 8), rank=rng.choice([8, 33, 40, 64]))
    if kind == "layer" and rng.random() < 0.4:        # the 1D problem
        c.update(dim=1, alpha=0.01, n=_log_int(rng, 48, 512), precision="fp64", particles=_log_int(rng, 64, 4096), steps=rng.randint(1, 5))
        c["km"] = min(64, c["n"] // 4 * 2)
        c["rank"] = min(c["rank"], c["km"])
        return c
    c["n"] = {"fit": 64, "reweight": 64, "batch": 0}.get(kind) if kind in ("fit", "reweight", "batch") else rng.choice(
        [64, 64, 128, 256] if kind != "move" else [64, 64, 128, 128, 256, 512])
    c["precision"] = rng.choice(["fp32", "fp32", "bf16", "fp64"]) if kind in ("move", "forward", "layer") else "fp32"
    side = c["n"] or 64
    c["km"] = 2 * _log_int(rng, 4, min(64, side // 2) // 2)
    c["rank"] = min(c["rank"], c["km"] ** 2)
    # solves of a pass: at most those of move_256 (2^28 cells), an eighth of that in FP64
    most = 2 ** 28 // (8 if c["precision"] == "fp64" else 2) // side ** 2
    if kind in ("move", "layer"):
        c["kernel"] = rng.choice(["pcn_gm", "pcn_gm", "pcn", "gm_indep"])
        c["steps"] = rng.randint(1, 4)
        c["particles"] = _log_int(rng, 8 if kind == "move" else 64, min(4096, most // c["steps"]))
    elif kind == "forward":
        c["particles"] = _log_int(rng, 2, min(2048, most // 4))
    elif kind == "gradient":
        c["particles"] = _log_int(rng, 2, min(2048, most // 4))
    elif kind == "batch":
        c.update(particles=_log_int(rng, 64, 1500), steps=rng.randint(1, 3), km=min(c["km"], 32))
        c["rank"] = min(c["rank"], c["km"] ** 2)
    else:
        c["particles"] = _log_int(rng, 300, {"fit": 6000, "reweight": 20000, "moments": min(8192, most // 2)}[kind])
        if kind == "fit":
            c["components"] = rng.randint(2, 8)
            c["full_cov"] = rng.random() < 0.5
    return c


# ---------------------------------------------------------------- inputs ----

def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)


def _eigenvalues(case):
    """Eigenvalues of the prior covariance in storage order, and the modes that carry the mixture."""
    Km, a = case["km"], case["alpha"]
    if case["dim"] == 1:
        k = np.arange(1, Km + 1, dtype=np.float64)
        return (1 + a * np.pi ** 2 * k ** 2) ** -2.0, np.arange(min(case["rank"], Km))
    k = np.arange(Km)
    q = (k[:, None] ** 2 + k[None, :] ** 2).reshape(-1)
    kk, ll = (v.reshape(-1) for v in np.meshgrid(k, k, indexing="ij"))
    return (1 + a * np.pi ** 2 * q) ** -2.0, np.sort(np.lexsort((ll, kk, q))[: case["rank"]])


def _problem(case, seed):
    """Observation points, data and particles. The data are a truth's (a prior draw on its own 64-cell
    grid, solved here in 64 bits) plus noise; the particles are draws of the prior, shifted towards
    one of a few centres where a mixture is fitted to them."""
    g = _gen(seed, 1)
    dim, N, m = case["dim"], case["particles"], case["obs"]
    lam, S = _eigenvalues(case)
    lam_t = torch.from_numpy(lam).to(DEV)
    truth = dict(case, n=64, km=min(case["km"], 32), rank=1)
    tl, _ = _eigenvalues(truth)
    x = torch.from_numpy(np.sqrt(tl)).to(DEV) * torch.randn(1, tl.size, dtype=F64, device=DEV, generator=g)
    if dim == 1:
        obs = (torch.arange(1, m + 1, dtype=F64, device=DEV) / (m + 1))
    else:
        obs = 0.05 + 0.9 * torch.rand(m, 2, dtype=F64, device=DEV, generator=g)
    y = _observe(truth, _solve(truth, x)[0], obs)[0]
    data = y + case["sigma"] * torch.randn(m, dtype=F64, device=DEV, generator=g)
    X = lam_t.sqrt() * torch.randn(N, lam.size, dtype=F64, device=DEV, generator=g)
    if case["kind"] == "fit":
        centres = lam_t.sqrt() * torch.randn(case["components"], lam.size, dtype=F64, device=DEV, generator=g)
        X = 0.6 * X + centres[torch.randint(case["components"], (N,), device=DEV, generator=g)]
    return obs, data, X, lam, S


def _mixture(case, seed, lam, S):
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 7])
    K, r = case["components"], len(S)
    w = rng.dirichlet(np.full(K, 3.0))
    m = 0.4 * rng.standard_normal((K, r)) * np.sqrt(lam[S])
    return w, m, lam[S] * rng.uniform(0.3, 1.2, size=(K, r))


def _seed64(seed):
    return 2503016028 + int(seed)


def _sampler(case, seed, obs, data):
    p = dict(dim=case["dim"], n=case["n"], kl_modes=case["km"], alpha=case["alpha"], sigma=case["sigma"],
             source_kind=1 if case["dim"] == 2 else 0, src_amp=10.0 if case["dim"] == 2 else 1.0,
             src_width=50.0 if case["dim"] == 2 else 0.0, n_particles=max(2, case["particles"]), n_components=case["components"],
             gm_rank=case["rank"], beta0=BETA, ess_frac=ESS, seed=_seed64(seed), em_iters=EM_ITERS, var_floor=VAR_FLOOR,
             obs=obs.cpu().numpy(), data=data.cpu().numpy(), precision=PRECISIONS[case["precision"]],
             kernel=KERNELS[case["kernel"]], gradient=int(case["kind"] == "gradient"), full_cov=int(case.get("full_cov", False)))
    return smcgm.Sampler(smcgm.make_config(p), device=DEV)


def _device_view(s, address, count, dtype):
    """The `count` values at a device address inside the sampler's workspace, as a tensor."""
    size = torch.empty(0, dtype=dtype).element_size()
    off = address - s.ws.data_ptr()
    return s.ws[off:off + count * size].view(dtype)


def _particles(s):
    x, p = smcgm.ctypes.c_void_p(), smcgm.ctypes.c_void_p()
    s._check(s.lib.smc_get_particles(s.ctx, smcgm.ctypes.byref(x), smcgm.ctypes.byref(p)), s.ctx)
    return {"X": _device_view(s, x.value, s.N * s.d, F64).view(s.N, s.d), "Phi": _device_view(s, p.value, s.N, F64)}


def _diagnostics(s):
    la, acc, pv, lw, idx = s.diagnostics_pointers()
    return {"log_alpha": _device_view(s, la, s.N, F64), "accepted": _device_view(s, acc, s.N, torch.uint8),
            "phi_proposed": _device_view(s, pv, s.N, F64), "logw": _device_view(s, lw, s.N, F64),
            "indices": _device_view(s, idx, s.N, torch.int32)}


def _put(s, X, Phi):
    """The particles (device tensors) into the sampler; Phi None: computed by the library."""
    s._check(s.lib.smc_set_particles(s.ctx, smcgm._ptr(X), smcgm._ptr(Phi), 1), s.ctx)


def _parts(case):
    """The problems of a batch case."""
    return [dict(case, n=n, particles=max(2, int(case["particles"] * share)), obs=case["obs"] + 3 * i, index=i)
            for i, (n, share) in enumerate(BATCH_PARTS)]


T0 = {"layer": 0.0, "reweight": 0.0}      # the temperature a pass starts from; a move's is 0.01


def prepare(case, seed):
    if case["kind"] == "batch":
        subs = [prepare(dict(p, kind="move"), seed + 7919 * (p["index"] + 1)) for p in _parts(case)]
        return {"case": case, "subs": subs, "batch": smcgm.Batch([u["s"] for u in subs], case["steps"])}
    obs, data, X, lam, S = _problem(case, seed)
    s = _sampler(case, seed, obs, data)
    st = {"case": case, "s": s, "X": X}
    kind = case["kind"]
    if kind in ("forward", "gradient"):
        N, n = case["particles"], case["n"]
        st["Phi"] = torch.empty(N, dtype=F64, device=DEV)
        st["out"] = torch.empty((N, n * n) if kind == "forward" else (N, s.d), dtype=F64, device=DEV)
        return st
    if kind == "reweight":                # potentials over a range of values, as after a few layers
        st["Phi"] = 400.0 * torch.rand(s.N, dtype=F64, device=DEV, generator=_gen(seed, 2)) ** 2
    elif kind in ("fit", "moments"):
        st["Phi"] = torch.zeros(s.N, dtype=F64, device=DEV)
    else:
        _put(s, X, None)
        st["Phi"] = _particles(s)["Phi"].clone()
    if kind == "move" and case["kernel"] != "pcn":
        s.smc_set_mixture(*_mixture(case, seed, lam, S))
    _put(s, X, st["Phi"])
    s.smc_set_schedule(T0.get(kind, 0.01), BETA if case["kernel"] != "gm_indep" else 1.0, 0, 0)
    return st


def _reset(st):
    _put(st["s"], st["X"], st["Phi"])
    st["s"].smc_set_schedule(T0.get(st["case"]["kind"], 0.01), BETA if st["case"]["kernel"] != "gm_indep" else 1.0, 0, 0)


def _moved(s, rate):
    d = _diagnostics(s)
    return dict(_particles(s), rate=float(rate), **{k: d[k] for k in ("log_alpha", "accepted", "phi_proposed")})


def _fitted(s, ll):
    w, m, lam, _ = s.smc_get_mixture()
    out = {"w": w, "m": m, "lam": lam, "loglik": float(ll)}
    if s.cfg.full_cov:
        out["cov"] = s.smc_get_mixture_cov()
    return out


def run(st):
    """One pass. A move in which over 1 % of the solves end above the tolerance (rough fields on the
    512^2 grid) still moves the particles, and a run goes on with them: allow_noconv."""
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        for u in st["subs"]:
            _reset(u)
        rates = st["batch"].move(allow_noconv=True)
        return [_moved(u["s"], r) for u, r in zip(st["subs"], rates)]
    s = st["s"]
    if kind == "forward":
        s.smc_forward(st["X"], st["Phi"], st["out"])
        return {"Phi": st["Phi"], "w": st["out"]}
    if kind == "gradient":
        s.smc_gradient(st["X"], st["Phi"], st["out"])
        return {"Phi": st["Phi"], "gradient": st["out"]}
    if kind == "fit":
        return _fitted(s, s.gm_fit())
    if kind == "moments":
        return dict(zip(("mean", "var", "mean_grid", "var_grid"), s.smc_posterior_moments(grid=True)))
    _reset(st)
    if kind == "move":
        return _moved(s, s.smc_move(case["steps"], allow_noconv=True)[0])
    h, ess, log_z, _ = s.smc_temper_step()
    s.smc_resample()
    out = {"h": h, "ess": ess, "log_z": log_z}
    if kind == "reweight":
        d = _diagnostics(s)
        return dict(out, logw=d["logw"], indices=d["indices"], **_particles(s))
    ll = s.gm_fit()
    if case["kernel"] != "pcn":
        out.update(_fitted(s, ll))
    return dict(out, **_moved(s, s.smc_move(case["steps"], allow_noconv=True)[0]))


def work(case):
    """Bytes: particles, potentials and results read and written once. Operations: the solves, the EM
    sums, the moments."""
    kind = case["kind"]
    if kind == "batch":
        ws = [work(dict(p, kind="move")) for p in _parts(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    N, K, r = case["particles"], case["components"], case["rank"]
    d = case["km"] ** 2 if case["dim"] == 2 else case["km"]
    cells = case["n"] ** case["dim"]
    state = 8.0 * N * (d + 1)
    solve = N * cells * (SOLVE_FLOPS if case["dim"] == 2 else 2.0 * case["km"] + 30)
    em = EM_ITERS * N * K * (2.0 * r * r if case.get("full_cov") else 10.0 * r)
    if kind == "forward":
        return {"bytes": state + 8.0 * N * cells, "flops": solve}
    if kind == "gradient":
        return {"bytes": 2 * state, "flops": 2 * solve}
    if kind == "fit":
        return {"bytes": 8.0 * N * r, "flops": em}
    if kind == "moments":
        return {"bytes": state + 16.0 * cells, "flops": N * (4.0 * d + cells * (3.0 + 10 * math.log2(case["n"])))}
    if kind == "reweight":
        return {"bytes": 2 * state + 12.0 * N, "flops": 100.0 * N}
    # each step of a move proposes from the particles and writes the accepted ones
    moves = {"bytes": 2 * state * case["steps"], "flops": case["steps"] * (solve + N * (8.0 * d + 20.0 * K * r))}
    if kind == "layer":
        moves["bytes"] += 2 * state
        moves["flops"] += em
    return moves


# ------------------------------------------- the same in 64 bits, plainly ----

def _basis(case):
    x = (torch.arange(case["n"], dtype=F64, device=DEV) + 0.5) / case["n"]
    if case["dim"] == 1:
        k = torch.arange(1, case["km"] + 1, dtype=F64, device=DEV)
        return math.sqrt(2.0) * torch.sin(math.pi * x[:, None] * k)
    k = torch.arange(case["km"], dtype=F64, device=DEV)
    return torch.cos(math.pi * x[:, None] * k) * torch.sqrt(2.0 - (k == 0).to(F64))


def _fields(case, X):
    B = _basis(case)
    if case["dim"] == 1:
        return X @ B.T
    return B @ X.view(-1, case["km"], case["km"]).transpose(-1, -2) @ B.T


def _inverse(A):
    """Inverses of symmetric positive definite matrices, by 2 x 2 blocks."""
    n = A.shape[-1]
    if n <= 16:
        return torch.linalg.inv(A)
    h = n // 2
    ai = _inverse(A[..., :h, :h])
    b = A[..., :h, h:]
    t = ai @ b
    si = _inverse(A[..., h:, h:] - b.transpose(-1, -2) @ t)
    ts = t @ si
    out = torch.empty_like(A)
    out[..., :h, :h] = ai + ts @ t.transpose(-1, -2)
    out[..., :h, h:] = -ts
    out[..., h:, :h] = -ts.transpose(-1, -2)
    out[..., h:, h:] = si
    return out


def _faces(k):
    """Harmonic west and south faces (0 at the walls) and the diagonal of the cell-centred operator."""
    Kw, Ks = torch.zeros_like(k), torch.zeros_like(k)
    Kw[:, :, 1:] = 2 * k[:, :, 1:] * k[:, :, :-1] / (k[:, :, 1:] + k[:, :, :-1])
    Ks[:, 1:] = 2 * k[:, 1:] * k[:, :-1] / (k[:, 1:] + k[:, :-1])
    D = Kw + Ks
    D[:, :, :-1] += Kw[:, :, 1:]
    D[:, :-1] += Ks[:, 1:]
    D[:, :, 0] += 2 * k[:, :, 0]
    D[:, :, -1] += 2 * k[:, :, -1]
    D[:, 0] += 2 * k[:, 0]
    D[:, -1] += 2 * k[:, -1]
    return Kw, Ks, D


def _source(case):
    n = case["n"]
    if case["dim"] == 1:
        return torch.full((n - 1,), 1.0 / n ** 2, dtype=F64, device=DEV)
    x = (torch.arange(n, dtype=F64, device=DEV) + 0.5) / n
    return 10.0 * torch.exp(-50.0 * ((x[None, :] - 0.5) ** 2 + (x[:, None] - 0.5) ** 2)) / n ** 2


def _solve(case, X, rhs_of=None):
    """The solutions of A(u) w = h^2 f for the rows of X by block elimination over the grid rows, and
    (with rhs_of: w -> another right-hand side) those for that one too."""
    n, out, two = case["n"], [], []
    f = _source(case)
    if case["dim"] == 1:
        K = torch.exp(_fields(case, X))
        c, y = [torch.zeros_like(K[:, 0])], [torch.zeros_like(K[:, 0])]
        for i in range(n - 1):                                  # Thomas elimination
            den = K[:, i] + K[:, i + 1] - K[:, i] * c[-1]
            c.append(K[:, i + 1] / den)
            y.append((f[i] + K[:, i] * y[-1]) / den)
        w = [y[-1]]
        for i in range(n - 2, 0, -1):
            w.insert(0, y[i] + c[i] * w[0])
        return torch.stack(w, 1), None
    step = max(1, int(6e9 / (8 * n ** 3)))
    for at in range(0, X.shape[0], step):
        Kw, Ks, D = _faces(torch.exp(_fields(case, X[at:at + step])))
        G = []
        for j in range(n):
            A = torch.diag_embed(D[:, j]) - torch.diag_embed(Kw[:, j, 1:], 1) - torch.diag_embed(Kw[:, j, 1:], -1)
            G.append(_inverse(A if j == 0 else A - Ks[:, j, :, None] * G[-1] * Ks[:, j, None, :]))

        def substitute(b):
            y = [b[:, 0]]
            for j in range(1, n):
                y.append(b[:, j] + Ks[:, j] * (G[j - 1] @ y[-1][..., None])[..., 0])
            w = [None] * n
            for j in range(n - 1, -1, -1):
                r = y[j] if j == n - 1 else y[j] + Ks[:, j + 1] * w[j + 1]
                w[j] = (G[j] @ r[..., None])[..., 0]
            return torch.stack(w, 1)
        w = substitute(f.expand(D.shape[0], n, n))
        out.append(w)
        if rhs_of is not None:
            two.append(substitute(rhs_of(w)))
    return torch.cat(out), torch.cat(two) if two else None


def _weights(case, obs):
    """Cells and weights of the bilinear interpolation at the observation points (all at least half a
    cell away from the walls)."""
    n = case["n"]
    s = obs * n - 0.5
    i0 = torch.floor(s).long()
    fx, fy = (s - i0).T
    i, j = i0.T
    return [(j * n + i, (1 - fy) * (1 - fx)), (j * n + i + 1, (1 - fy) * fx), ((j + 1) * n + i, fy * (1 - fx)), ((j + 1) * n + i + 1, fy * fx)]


def _observe(case, w, obs):
    if case["dim"] == 1:
        full = torch.nn.functional.pad(w, (1, 1))
        i = torch.clamp(torch.floor(obs * case["n"]).long(), max=case["n"] - 1)
        fx = obs * case["n"] - i
        return (1 - fx) * full[:, i] + fx * full[:, i + 1]
    flat = w.reshape(w.shape[0], -1)
    return sum(wt * flat[:, c] for c, wt in _weights(case, obs))


def _potential(case, X, obs, data):
    r = _observe(case, _solve(case, X)[0], obs) - data
    return (r * r).sum(1) / (2 * case["sigma"] ** 2)


def _gradient(case, X, obs, data):
    n, s2 = case["n"], case["sigma"] ** 2

    def misfit(w):
        g = torch.zeros(w.shape[0], n * n, dtype=F64, device=DEV)
        r = (_observe(case, w, obs) - data) / s2
        for c, wt in _weights(case, obs):
            g.index_add_(1, c, r * wt)
        return g.view(-1, n, n)
    w, a = _solve(case, X, misfit)
    r = _observe(case, w, obs) - data
    k = torch.exp(_fields(case, X))
    Kw, Ks, _ = _faces(k)
    g = torch.zeros_like(k)
    px = (a[:, :, 1:] - a[:, :, :-1]) * (w[:, :, 1:] - w[:, :, :-1]) * Kw[:, :, 1:] / (k[:, :, 1:] + k[:, :, :-1])
    g[:, :, 1:] -= px * k[:, :, :-1]
    g[:, :, :-1] -= px * k[:, :, 1:]
    py = (a[:, 1:] - a[:, :-1]) * (w[:, 1:] - w[:, :-1]) * Ks[:, 1:] / (k[:, 1:] + k[:, :-1])
    g[:, 1:] -= py * k[:, :-1]
    g[:, :-1] -= py * k[:, 1:]
    wall = 2 * k * a * w
    g[:, :, 0] -= wall[:, :, 0]
    g[:, :, -1] -= wall[:, :, -1]
    g[:, 0] -= wall[:, 0]
    g[:, -1] -= wall[:, -1]
    B = _basis(case)
    return (r * r).sum(1) / (2 * s2), (B.T @ g.transpose(-1, -2) @ B).reshape(X.shape[0], -1)


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on uint64 arrays holding 32-bit words."""
    mask, sh = np.uint64(0xFFFFFFFF), np.uint64(32)
    c = [np.array(v, dtype=np.uint64) for v in np.broadcast_arrays(c0, c1, c2, c3)]
    k = [seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF]
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> sh) ^ c[1] ^ np.uint64(k[0]), p1 & mask, (p0 >> sh) ^ c[3] ^ np.uint64(k[1]), p0 & mask]
        k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
    return c


def _uniform(a, b):
    return ((((a >> np.uint64(5)) << np.uint64(26)) | (b >> np.uint64(6))).astype(np.float64) + 0.5) * 2.0 ** -53


def _move(case, seed, X, Phi, obs, data, mix, S, lam, t, steps):
    """`steps` moves of every particle from (X, Phi), as ``_moved`` returns them."""
    N, d = X.shape
    indep = case["kernel"] == "gm_indep"
    b = 1.0 if indep else BETA
    gam = math.sqrt(1 - b * b)
    w, m, l = (torch.from_numpy(np.asarray(v)).to(DEV) for v in mix)
    lam_t, St, key = torch.from_numpy(lam).to(DEV), torch.from_numpy(S).to(DEV), _seed64(seed)
    K, l0, cum = len(w), torch.from_numpy(lam[S]).to(DEV), torch.cumsum(w, 0)
    ids = np.arange(N, dtype=np.uint64)

    def log_ratio(to, fr):
        e = to[:, St] - gam * fr[:, St]
        return torch.logsumexp(torch.stack([torch.log(w[j]) + (0.5 * torch.log(l0 / l[j]) - (e - (1 - gam) * m[j]) ** 2 / (2 * b * b * l[j])
                                            + e * e / (2 * b * b * l0)).sum(1) for j in range(K)], 1), 1)
    taken = 0
    for step in range(steps):
        u = _philox(0, ids, step, 2, key)
        comp = torch.clamp(torch.searchsorted(cum, torch.from_numpy(_uniform(u[0], u[1])).to(DEV), right=True), max=K - 1)
        z4 = _philox(np.arange(d // 2, dtype=np.uint64)[None, :], ids[:, None], step, 3, key)
        r = torch.sqrt(-2 * torch.log(torch.from_numpy(_uniform(z4[0], z4[1])).to(DEV)))
        a = 2 * math.pi * torch.from_numpy(_uniform(z4[2], z4[3])).to(DEV)
        z = torch.stack((r * torch.cos(a), r * torch.sin(a)), -1).view(N, d)
        V = gam * X + b * lam_t.sqrt() * z
        V[:, St] = gam * X[:, St] + (1 - gam) * m[comp] + b * l[comp].sqrt() * z[:, St]
        pv = _potential(case, V, obs, data)
        la = torch.zeros_like(pv) if indep else t * (Phi - pv) + log_ratio(X, V) - log_ratio(V, X)
        u = _philox(0, ids, step, 4, key)
        acc = (la >= 0) | (torch.log(torch.from_numpy(_uniform(u[0], u[1])).to(DEV)) < la)
        X, Phi = torch.where(acc[:, None], V, X), torch.where(acc, pv, Phi)
        taken += int(acc.sum())
    return {"X": X, "Phi": Phi, "rate": taken / (N * steps), "log_alpha": None if indep else la, "accepted": acc.to(torch.uint8), "phi_proposed": pv}


def _em(case, seed, X, S, lam):
    """EM of the mixture (diagonal or full covariances) on the modes S; with the outputs of ``_fitted``."""
    xs, l0, N, K = X[:, torch.from_numpy(S).to(DEV)], torch.from_numpy(lam[S]).to(DEV), X.shape[0], case["components"]
    full = case.get("full_cov", False)
    pooled = torch.maximum(xs.var(0, unbiased=False), VAR_FLOOR * l0)
    picks = []
    for k in range(K):
        c = (int(_philox(k, 0, 0, 6, _seed64(seed))[0]) * N) >> 32
        while c in picks:
            c = (c + 1) % N
        picks.append(c)
    w, m = torch.full((K,), 1.0 / K, dtype=F64, device=DEV), xs[picks].clone()
    C = torch.diag(pooled).repeat(K, 1, 1) if full else pooled.repeat(K, 1)

    def densities():
        dev = xs[None] - m[:, None]
        if full:
            L = torch.linalg.cholesky(C)
            y = torch.linalg.solve_triangular(L, dev.transpose(1, 2), upper=False)
            q, det = (y * y).sum(1), 2 * torch.log(torch.diagonal(L, dim1=1, dim2=2)).sum(1)
        else:
            q, det = (dev * dev / C[:, None]).sum(2), torch.log(C).sum(1)
        lp = torch.log(w)[:, None] - 0.5 * (len(S) * math.log(2 * math.pi) + det)[:, None] - 0.5 * q
        return lp, torch.logsumexp(lp, 0)
    for _ in range(EM_ITERS):
        lp, lse = densities()
        g = torch.exp(lp - lse)
        nj = g.sum(1)
        m = g @ xs / nj[:, None]
        dev = xs[None] - m[:, None]
        if full:
            C = (g[..., None] * dev).transpose(1, 2) @ dev / nj[:, None, None] + torch.diag(VAR_FLOOR * l0)
        else:
            C = torch.maximum((g[..., None] * dev * dev).sum(1) / nj[:, None], VAR_FLOOR * l0)
        w = nj / N
        low = nj < 2.0
        if bool(low.any()):
            m[low] = xs[int(torch.argmin(g.max(0).values))]
            C[low] = torch.diag(pooled) if full else pooled
            w[low] = 1.0 / N
        w = w / w.sum()
    out = {"w": w, "m": m, "lam": torch.diagonal(C, dim1=1, dim2=2) if full else C, "loglik": float(densities()[1].sum())}
    return dict(out, cov=C) if full else out


def _reweight(seed, X, Phi):
    """Reweighting from t = 0 and systematic resampling."""
    phi = Phi.cpu().numpy()
    N = len(phi)

    def ess(h):
        e = np.exp(-h * (phi - phi.min()))
        return e.sum() ** 2 / (e * e).sum()
    lo, hi = 0.0, 1.0
    if ess(1.0) >= ESS * N:
        lo = 1.0
    else:
        for _ in range(64):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if ess(mid) >= ESS * N else (lo, mid)
    lw = -lo * phi
    lse = lw.max() + np.log(np.exp(lw - lw.max()).sum())
    lw = lw - lse
    q = [int(v) for v in np.floor(np.exp(lw - (lw.max() + np.log(np.exp(lw - lw.max()).sum()))) * 2.0 ** 48)]
    q[int(np.argmax(lw))] += (1 << 48) - sum(q)
    u = _philox(0, 0, 0, 5, _seed64(seed))
    u48, idx, run_, i = (int(u[0]) << 16) | (int(u[1]) >> 16), [], q[0], 0
    for k in range(N):
        while N * run_ <= (k << 48) + u48:
            i += 1
            run_ += q[i]
        idx.append(i)
    at = torch.tensor(idx, device=DEV)
    head = {"h": float(lo), "ess": float(ess(lo)), "log_z": float(lse - np.log(N))}
    return head, torch.from_numpy(lw).to(DEV), at.to(torch.int32), X[at], Phi[at]


def _cheap(case):
    """Whether the block elimination of a case's solves ends in a few seconds."""
    solves = case["particles"] * case.get("steps", 1) + case["particles"]
    return case["dim"] == 1 or solves * float(case["n"]) ** 4 < 1.5e12


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        nothing = dict.fromkeys(("X", "Phi", "rate", "log_alpha", "accepted", "phi_proposed"))
        return [(exact(dict(p, kind="move"), seed + 7919 * (p["index"] + 1)) if p["n"] <= 128 else None) or nothing for p in _parts(case)]
    if kind not in ("fit", "reweight", "moments") and not _cheap(case):
        return None
    obs, data, X, lam, S = _problem(case, seed)
    if kind == "forward":
        w = _solve(case, X)[0]
        r = _observe(case, w, obs) - data
        return {"Phi": (r * r).sum(1) / (2 * case["sigma"] ** 2), "w": w.reshape(X.shape[0], -1)}
    if kind == "gradient":
        return dict(zip(("Phi", "gradient"), _gradient(case, X, obs, data)))
    if kind == "fit":
        return _em(case, seed, X, S, lam)
    if kind == "moments":
        mean = X.mean(0)
        var, grid, sq = ((X - mean) ** 2).mean(0), _fields(case, mean[None])[0], 0.0
        for at in range(0, X.shape[0], 512):
            sq = sq + ((_fields(case, X[at:at + 512]) - grid) ** 2).sum(0)
        return {"mean": mean, "var": var, "mean_grid": grid.reshape(-1), "var_grid": (sq / X.shape[0]).reshape(-1)}
    if kind == "reweight":
        Phi = 400.0 * torch.rand(X.shape[0], dtype=F64, device=DEV, generator=_gen(seed, 2)) ** 2
        head, lw, idx, X, Phi = _reweight(seed, X, Phi)
        return dict(head, logw=lw, indices=idx, X=X, Phi=Phi)
    Phi = _potential(case, X, obs, data)
    none = case["kernel"] == "pcn"
    if kind == "move":
        mix = (np.ones(1), np.zeros((1, len(S))), lam[S][None]) if none else _mixture(case, seed, lam, S)
        return _move(case, seed, X, Phi, obs, data, mix, S, lam, 0.01, case["steps"])
    head, _, _, X, Phi = _reweight(seed, X, Phi)
    fit = None if none else _em(case, seed, X, S, lam)
    mix = (np.ones(1), np.zeros((1, len(S))), lam[S][None]) if none else tuple(fit[k].cpu().numpy() for k in ("w", "m", "lam"))
    return dict(head, **(fit or {}), **_move(case, seed, X, Phi, obs, data, mix, S, lam, head["h"], case["steps"]))
