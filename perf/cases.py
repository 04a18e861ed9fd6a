"""Performance cases of the library: the work its users have it do, through the public binding.

A pass is one call (or the few calls a user's program makes together) of
`paper_1709_09763_gb300.native`: bulk likelihood evaluations on each mesh level, the sampler's two
update kinds, the evaluation of many small problems at once, and one gradient pass of the
surrogate network. Sizes are those of `workloads.py`, the tests and `bench.py`.

`exact` restates the likelihood in 64 bits with torch alone: the Karhunen-Loeve field, the 5-point
stencil of P1 elements on the diagonally split unit square, conjugate gradients to 1e-13, P1
interpolation and the Gaussian misfit.
"""
import functools
import math

import numpy as np
import torch

from paper_1709_09763_gb300 import native

# textbook work of the solve: ~11 iterations of multigrid-preconditioned CG, 2 refinement passes
FLOPS_PER_NODE = 11 * 55 + 2 * 100


def _solve(name, inv_h, J, K, **kw):
    case = dict(kind="solve", inv_h=inv_h, J=J, K=K, corr_len=0.1, cov="sep_exp", source="one", bc="dirichlet",
                obs=7, precision="mixed", host=False)
    case.update(kw)
    return dict(case, name=name) if name else case


def listed():
    return [
        # the cv^LU predictor's likelihoods: 100 particles on the coarsest level, host arrays in and out
        _solve("predictor_h8", 8, 100, 32, host=True),
        # single-level SMC in FP64 (smc_fp64_h16): one evaluation of its 1000 particles
        _solve("fp64_h16", 16, 1000, 16, corr_len=0.3, precision="fp64"),
        # the benchmark's hierarchy (mls2mc_mixed_h8_64): one launch on an inner and on the finest level
        _solve("mls2mc_h32", 32, 4000, 32),
        _solve("mls2mc_h64", 64, 4000, 32),
        # Example 5.1 (Matern prior, nine sources, 25 interpolated observations)
        _solve("example_5_1_h64", 64, 2500, 10, corr_len=0.65, cov="matern", source="nine", obs=5),
        # Example 5.3 (flow cell, Matern prior)
        _solve("flow_cell_h64", 64, 1000, 64, cov="matern", bc="flow_cell"),
        # the surrogate workload's finest level (da_mixed_h8_128): the exact solves of one Markov step
        _solve("surrogate_h128", 128, 8000, 64),
        # the large workload's finest level (large_mixed_h16_256): the survivors of one screened step
        _solve("large_h256", 256, 1001, 128, corr_len=0.05, obs=12),
        # a tempering update (increment, resampling, five pCN steps), host particles in and out
        dict(name="tempering_h32", kind="tempering", inv_h=32, J=1000, K=32, corr_len=0.1, n_mcmc=5),
        # a bridging step 1/32 -> 1/64 with its Markov steps on both levels
        dict(name="bridging_h32_64", kind="bridging", inv_h=32, J=1000, K=32, corr_len=0.1, n_mcmc=5),
        # many small problems (the batched workload at its small end): one graph replay for all
        dict(name="batch_small", kind="batch", problems=64, j_low=16, j_high=256, finest=64, draws=7),
        # one gradient pass of the surrogate network at the default minibatch
        dict(name="surrogate_grads", kind="grads", K=64, n_obs=49, batch=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 7 + ["tempering", "bridging", "batch", "grads"])
    if kind == "solve":
        inv_h = rng.choice([8, 16, 32, 64, 128, 256])
        # counts up to the workloads' 16384, less where that would outlast the largest listed case
        J = _log_int(rng, 100, {128: 6000, 256: 900}.get(inv_h, 16384))
        form = rng.choice(["plain", "plain", "plain", "nine", "flow", "fp64"])
        case = _solve(None, inv_h, J, _log_int(rng, 8, 256 if inv_h < 256 else 128),
                      corr_len=rng.choice([0.05, 0.1, 0.2, 0.3, 0.65]), obs=rng.choice([5, 7, 12]))
        if form in ("nine", "flow"):
            case.update(cov="matern", K=_log_int(rng, 8, 64), corr_len=rng.choice([0.1, 0.3, 0.65]))
            case.update(dict(source="nine") if form == "nine" else dict(bc="flow_cell"))
            if form == "flow" and inv_h >= 128:
                case["J"] = min(case["J"], 600 if inv_h == 256 else 2500)
        elif form == "fp64" and inv_h <= 32:
            case.update(precision="fp64", J=min(case["J"], 4000))
        return case
    if kind in ("tempering", "bridging"):
        return dict(kind=kind, inv_h=rng.choice([8, 16, 32]), J=_log_int(rng, 250, 1500), K=_log_int(rng, 8, 64),
                    corr_len=rng.choice([0.1, 0.3]), n_mcmc=rng.randint(1, 5))
    if kind == "batch":
        return dict(kind="batch", problems=rng.randint(16, 64), j_low=16, j_high=_log_int(rng, 64, 512),
                    finest=rng.choice([32, 64]), draws=rng.randrange(10 ** 6))
    return dict(kind="grads", K=_log_int(rng, 8, 128), n_obs=rng.choice([25, 49, 144]), batch=_log_int(rng, 512, 8192))


# ---- what a program has in hand before the call -------------------------------------------------
def _obs_grid(n):
    return np.array([((i + 1) / (n + 1), (j + 1) / (n + 1)) for j in range(n) for i in range(n)])


def _normals(shape, seed):
    return np.random.default_rng(seed).standard_normal(shape)


@functools.lru_cache(maxsize=64)
def _data(K, corr_len, cov, source, bc, obs, seed):
    """Synthetic data of a problem: the 64-bit response of a prior draw on 1/32, 1 % noise."""
    theta = torch.from_numpy(_normals((1, K), seed)).cuda()
    G = _response(dict(inv_h=32, K=K, corr_len=corr_len, cov=cov, source=source, bc=bc, obs=obs), theta)[0].cpu().numpy()
    sigma = 0.01 * float(np.abs(G).max())
    return G + sigma * _normals(G.shape, seed + 1), sigma


def _handle(inv_h, case, **kw):
    cov, source, bc = case.get("cov", "sep_exp"), case.get("source", "one"), case.get("bc", "dirichlet")
    obs = case.get("obs", 7)
    y, sigma = _data(case["K"], case["corr_len"], cov, source, bc, obs, case.get("data_seed", 11))
    prec = native.SMC_FP64 if case.get("precision") == "fp64" else native.SMC_MIXED
    return native.Handle(inv_h, case["K"], _obs_grid(obs), y, sigma, corr_len=case["corr_len"], precision=prec, cov=cov,
                         source=source, bc=bc, **kw)


def _batch_problems(case):
    rng = np.random.default_rng(case["draws"])
    out = []
    for p in range(case["problems"]):
        inv_h = int(rng.choice([h for h in (16, 32, 64) if h <= case["finest"]]))
        K = int(rng.choice([16, 32, 64]))
        J = int(round(math.exp(rng.uniform(math.log(case["j_low"]), math.log(case["j_high"])))))
        out.append(dict(inv_h=inv_h, K=K, J=J, corr_len=0.3 if K == 16 else 0.1, data_seed=100 + p % 8))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        h = _handle([case["inv_h"]], case)
        theta = _normals((case["J"], case["K"]), seed)
        if case["host"]:
            return dict(kind="host", h=h, theta=theta)
        theta = torch.from_numpy(theta).cuda()
        G = torch.empty((case["J"], case["obs"] ** 2), dtype=torch.float64, device="cuda")
        return dict(kind=kind, h=h, theta=theta, G=G, Phi=torch.empty_like(G[:, 0]).contiguous())
    if kind in ("tempering", "bridging"):
        N = case["inv_h"]
        h = _handle([N, 2 * N] if kind == "bridging" else [N], case, J=case["J"], n_mcmc=case["n_mcmc"], seed=seed)
        return dict(kind=kind, h=h, theta=_normals((case["J"], case["K"]), seed), n_mcmc=case["n_mcmc"])
    if kind == "batch":
        probs = _batch_problems(case)
        handles = [_handle([p["inv_h"]], p) for p in probs]
        thetas = [torch.from_numpy(_normals((p["J"], p["K"]), seed * 1000 + i)).cuda() for i, p in enumerate(probs)]
        J = [p["J"] for p in probs]
        Phi = torch.empty(sum(J), dtype=torch.float64, device="cuda")
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        return dict(kind=kind, batch=native.Batch(handles), handles=handles, thetas=thetas, J=J, Phi=Phi, stream=stream,
                    phi_ptrs=[p.data_ptr() for p in Phi.split(J)], theta_ptrs=[t.data_ptr() for t in thetas])
    h = native.Handle([8], case["K"], np.full((case["n_obs"], 2), 0.5), np.zeros(case["n_obs"]), 1.0, corr_len=0.1,
                      precision=native.SMC_MIXED)
    params, mu_sd, theta, G = _network(case, seed)
    h.surrogate_set(0, params, mu_sd)
    return dict(kind=kind, h=h, theta=theta, G=G)


def run(state):
    kind = state["kind"]
    h = state.get("h")
    if kind == "solve":
        theta, G, Phi = state["theta"], state["G"], state["Phi"]
        h.eval_likelihood_device(0, theta.shape[0], theta.data_ptr(), G.data_ptr(), Phi.data_ptr())
        return dict(G=G, Phi=Phi)
    if kind == "host":
        G, Phi = h.eval_likelihood(0, state["theta"])
        return dict(G=G, Phi=Phi)
    if kind in ("tempering", "bridging"):
        h.set_particles(state["theta"])
        if kind == "tempering":
            info = h.tempering_update(0, 0.0, state["n_mcmc"])
        else:
            info = h.bridging_update(0, 1.0, 0.0, state["n_mcmc"])
        theta, phi = h.particles()
        return dict(theta=theta, phi=phi, n_unique=info["n_unique"],
                    **{k: float(info[k]) for k in ("beta", "zeta", "delta", "cv", "log_z_inc", "accept_rate")})
    if kind == "batch":
        state["batch"].eval([0] * len(state["J"]), state["J"], state["theta_ptrs"], state["phi_ptrs"],
                            stream=state["stream"].cuda_stream)
        return state["Phi"]
    grads, loss = h.surrogate_grads(0, state["theta"], state["G"])
    return dict(grads=grads, loss=float(loss))


# ---- what a pass cannot do without ---------------------------------------------------------------
def _solve_work(inv_h, J, K, n_obs):
    E, nodes = 2 * inv_h ** 2, (inv_h - 1) ** 2
    return dict(bytes=8.0 * J * (K + n_obs + 1) + 4.0 * K * E, flops=J * (2.0 * K * E + nodes * FLOPS_PER_NODE))


def work(case):
    kind = case["kind"]
    if kind == "solve":
        return _solve_work(case["inv_h"], case["J"], case["K"], case["obs"] ** 2)
    if kind in ("tempering", "bridging"):
        # Phi of the particles, resampling, and each Markov step's solve of every proposal
        total = dict(bytes=8.0 * case["J"] * (2 * case["K"] + 1), flops=0.0)
        for inv_h in (case["inv_h"], 2 * case["inv_h"])[:1 + (kind == "bridging")]:
            total["flops"] += (1 + case["n_mcmc"]) * _solve_work(inv_h, case["J"], case["K"], 49)["flops"]
        return total
    if kind == "batch":
        parts = [_solve_work(p["inv_h"], p["J"], p["K"], 0) for p in _batch_problems(case)]
        return dict(bytes=sum(p["bytes"] for p in parts), flops=sum(p["flops"] for p in parts))
    B, d = case["batch"], [case["K"], 256, 256, 256, 256, case["n_obs"]]
    params = sum(a * b + b for a, b in zip(d, d[1:]))
    return dict(bytes=8.0 * B * (d[0] + d[-1]) + 8.0 * params,
                flops=2.0 * B * (3 * sum(a * b for a, b in zip(d, d[1:])) - d[0] * d[1]))


# ---- the same results in 64 bits ------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind in ("tempering", "bridging"):
        return None   # depends on the library's random draws
    if kind == "solve":
        theta = torch.from_numpy(_normals((case["J"], case["K"]), seed)).cuda()
        y, sigma = _data(case["K"], case["corr_len"], case["cov"], case["source"], case["bc"], case["obs"], 11)
        G = _response(case, theta)
        return dict(G=G, Phi=_misfit(G, y, sigma))
    if kind == "batch":
        out = []
        for i, p in enumerate(_batch_problems(case)):
            full = dict(cov="sep_exp", source="one", bc="dirichlet", obs=7, **p)
            y, sigma = _data(p["K"], p["corr_len"], "sep_exp", "one", "dirichlet", 7, p["data_seed"])
            theta = torch.from_numpy(_normals((p["J"], p["K"]), seed * 1000 + i)).cuda()
            out.append(_misfit(_response(full, theta), y, sigma))
        return torch.cat(out)
    return _network_gradients(case, seed)


def _misfit(G, y, sigma):
    return 0.5 * (((torch.from_numpy(y).to(G.device) - G) / sigma) ** 2).sum(1)


def _modes_1d(corr_len, n):
    """Frequencies and eigenvalues of exp(-|s - t| / corr_len) on [0, 1]: mode m in x = omega / 2 of
    (m pi / 2, (m + 1) pi / 2), even (cosine) for even m."""
    c = 1.0 / corr_len
    m = np.arange(n)
    lo, hi = m * math.pi / 2, (m + 1) * math.pi / 2
    even = m % 2 == 0
    f = lambda x: np.where(even, 2 * x * np.sin(x) - c * np.cos(x), 2 * x * np.cos(x) + c * np.sin(x))  # noqa: E731
    s = np.sign(f(lo + 1e-13 * (hi - lo)))
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        left = np.sign(f(mid)) == s
        lo, hi = np.where(left, mid, lo), np.where(left, hi, mid)
    w = lo + hi
    return w, 2 * c / (w * w + c * c), even


def _separable_basis(corr_len, K, x, y):
    w, lam, even = _modes_1d(corr_len, K)
    norm = np.sqrt(0.5 + np.where(even, 1, -1) * np.sin(w) / (2 * w))
    phi = lambda s: np.where(even[:, None], np.cos(np.outer(w, s - 0.5)), np.sin(np.outer(w, s - 0.5))) / norm[:, None]  # noqa: E731
    m, n = np.meshgrid(np.arange(K), np.arange(K), indexing="ij")
    m, n = m.ravel(), n.ravel()
    order = np.lexsort((m, np.maximum(m, n), -(lam[m] * lam[n])))[:K]
    px, py = phi(np.unique(x)), phi(np.unique(y))
    ix, iy = np.unique(x, return_inverse=True)[1], np.unique(y, return_inverse=True)[1]
    return np.stack([np.sqrt(lam[a] * lam[b]) * px[a][ix] * py[b][iy] for a, b in zip(m[order], n[order])])


def _matern_basis(corr_len, K, x, y, M=32):
    """Nystrom pairs of the Matern 3/2 covariance on an M x M midpoint grid (K <= 64), one quarter of
    the grid per reflection parity; x <-> y pairs of mixed parity are mirror images."""
    def cov(ax, ay, bx, by):
        z = math.sqrt(6.0) * np.hypot(ax[:, None] - bx[None], ay[:, None] - by[None]) / corr_len
        return (1 + z) * np.exp(-z)

    m = M // 2
    c = (np.arange(m) + 0.5) / M
    qx, qy = (a.ravel() for a in np.meshgrid(c, c, indexing="ij"))

    def folded(f, sx, sy):
        return f(qx, qy) + sx * f(1 - qx, qy) + sy * f(qx, 1 - qy) + sx * sy * f(1 - qx, 1 - qy)

    swap = np.arange(m * m).reshape(m, m).T.ravel()
    eye = np.eye(m * m)
    found = []
    for sector, sx, sy, par in ((0, 1, 1, 1), (0, 1, 1, -1), (1, 1, -1, 0), (3, -1, -1, 1), (3, -1, -1, -1)):
        A = folded(lambda bx, by: cov(qx, qy, bx, by), sx, sy) / M ** 2
        if par:
            B = (eye + par * eye[swap])[:, [i for i in range(m * m) if swap[i] > i or (par > 0 and swap[i] == i)]]
            B = B / np.linalg.norm(B, axis=0)
            lam, V = np.linalg.eigh(B.T @ A @ B)
            V = B @ V
        else:
            lam, V = np.linalg.eigh(A)
        g = folded(lambda bx, by: np.exp(0.7 * bx + 1.3 * by), sx, sy)
        for k in range(lam.size - 1, max(lam.size - 1 - K, -1), -1):
            u = V[:, k] * (M / 2) * (1 if V[:, k] @ g > 0 else -1)
            found.append((lam[k], (sector, -par), sx, sy, u))
            if sector == 1:
                found.append((lam[k], (2, 0), -1, 1, u[swap]))
    found.sort(key=lambda t: -t[0])
    ordered, i = [], 0
    while len(ordered) < K:   # equal eigenvalues (to 1e-9): by sector
        j = i + 1
        while j < len(found) and found[j - 1][0] - found[j][0] <= 1e-9 * found[i][0]:
            j += 1
        ordered += sorted(found[i:j], key=lambda t: t[1])
        i = j
    ordered = ordered[:K]
    dev = "cuda"
    tx, ty, hx, hy = (torch.from_numpy(a).to(dev) for a in (x, y, qx, qy))
    out = torch.empty((K, x.size), dtype=torch.float64, device=dev)
    for a in range(0, x.size, 16384):
        def kern(bx, by):
            z = math.sqrt(6.0) * torch.hypot(tx[a:a + 16384, None] - bx[None], ty[a:a + 16384, None] - by[None]) / corr_len
            return (1 + z) * torch.exp(-z)
        parts = [kern(hx, hy), kern(1 - hx, hy), kern(hx, 1 - hy), kern(1 - hx, 1 - hy)]
        for sx, sy in ((1, 1), (1, -1), (-1, 1), (-1, -1)):
            ks = [k for k, t in enumerate(ordered) if (t[2], t[3]) == (sx, sy)]
            if ks:
                F = parts[0] + sx * parts[1] + sy * parts[2] + sx * sy * parts[3]
                U = torch.from_numpy(np.stack([ordered[k][4] / math.sqrt(ordered[k][0]) for k in ks], 1)).to(dev)
                out[ks, a:a + 16384] = (F @ U / M ** 2).T
    return out


@functools.lru_cache(maxsize=2)
def _basis(cov, corr_len, K, N):
    """sqrt(lambda_k) phi_k at the centroids of the lower and the upper triangles: [K][2][N][N] (t, j, i)."""
    i = np.arange(N)
    lo = ((i + 2 / 3) / N, (i + 1 / 3) / N)
    up = ((i + 1 / 3) / N, (i + 2 / 3) / N)
    x = np.concatenate([np.tile(a[0], N) for a in (lo, up)])
    y = np.concatenate([np.repeat(a[1], N) for a in (lo, up)])
    psi = _matern_basis(corr_len, K, x, y) if cov == "matern" else torch.from_numpy(_separable_basis(corr_len, K, x, y)).cuda()
    return psi.reshape(K, 2, N, N)


def _nine_sources(N):
    """Load vector on the (N + 1)^2 nodes by the edge-midpoint rule: h^2 / 6 times f at the midpoints of
    a node's six edges."""
    def f(x, y):
        g = lambda s: sum(np.exp(-(s - 0.25 * n) ** 2 / 0.002) for n in (1, 2, 3)) / math.sqrt(0.002 * math.pi)  # noqa: E731
        return g(x) * g(y)
    s = np.arange(N + 1) / N
    x, y = s[None, :], s[:, None]
    d = 0.5 / N
    return sum(f(x + a * d, y + b * d) for a, b in ((1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1))) / (6 * N * N)


def _response(case, theta):
    """Observations of the PDE solutions of theta [J][K], in 64 bits, a bounded number of particles at a time."""
    N = case["inv_h"]
    chunk = max(1, 3 * 10 ** 8 // (N + 1) ** 2)
    return torch.cat([_response_of(case, t) for t in theta.split(chunk)])


def _response_of(case, theta):
    N, flow, dev = case["inv_h"], case["bc"] == "flow_cell", theta.device
    J = theta.shape[0]
    psi = _basis(case["cov"], case["corr_len"], case["K"], N)
    kap = torch.exp(theta @ psi.reshape(case["K"], -1)).reshape(J, 2, N, N)
    # edge weights: half the sum of the two triangles at an edge
    aE = torch.zeros((J, N + 1, N), dtype=torch.float64, device=dev)
    aE[:, :N] += 0.5 * kap[:, 0]
    aE[:, 1:] += 0.5 * kap[:, 1]
    aN = torch.zeros((J, N, N + 1), dtype=torch.float64, device=dev)
    aN[:, :, 1:] += 0.5 * kap[:, 0]
    aN[:, :, :N] += 0.5 * kap[:, 1]
    del kap
    free = torch.zeros((N + 1, N + 1), dtype=torch.float64, device=dev)
    if flow:
        free[:, 1:N] = 1
    else:
        free[1:N, 1:N] = 1

    def apply(v):
        out = torch.zeros_like(v)
        e = aE * (v[:, :, :-1] - v[:, :, 1:])
        out[:, :, :-1] += e
        out[:, :, 1:] -= e
        e = aN * (v[:, :-1] - v[:, 1:])
        out[:, :-1] += e
        out[:, 1:] -= e
        return out * free

    x = torch.zeros((J, N + 1, N + 1), dtype=torch.float64, device=dev)
    if flow:
        x[:, :, N] = 1
        r = -apply(x)
    else:
        load = np.full((N + 1, N + 1), 1.0 / N ** 2) if case["source"] == "one" else _nine_sources(N)
        r = (torch.from_numpy(load).to(dev) * free).expand(J, -1, -1).clone()
    diag = torch.zeros_like(x)
    diag[:, :, :-1] += aE
    diag[:, :, 1:] += aE
    diag[:, :-1] += aN
    diag[:, 1:] += aN
    z = r / diag
    p = z.clone()
    rz = (r * z).sum((1, 2), keepdim=True)
    stop = 1e-26 * (r * r).sum((1, 2), keepdim=True)
    for it in range(20 * N + 200):
        q = apply(p)
        alpha = rz / (p * q).sum((1, 2), keepdim=True).clamp_min(1e-300)
        x += alpha * p
        r -= alpha * q
        torch.div(r, diag, out=z)
        new = (r * z).sum((1, 2), keepdim=True)
        p.mul_(new / rz.clamp_min(1e-300)).add_(z)
        rz = new
        if it % 25 == 24 and bool(((r * r).sum((1, 2), keepdim=True) <= stop).all()):
            break
    xy = _obs_grid(case["obs"]) * N
    ij = np.minimum(xy.astype(int), N - 1)
    a, b = (xy - ij).T
    i, j = (torch.from_numpy(v).to(dev) for v in ij.T)
    lower = b <= a
    w = [1 - np.maximum(a, b), np.where(lower, a - b, 0), np.where(lower, 0, b - a), np.minimum(a, b)]
    w = [torch.from_numpy(v).to(dev) for v in w]
    return w[0] * x[:, j, i] + w[1] * x[:, j, i + 1] + w[2] * x[:, j + 1, i] + w[3] * x[:, j + 1, i + 1]


# ---- the surrogate network -----------------------------------------------------------------------
def _dims(case):
    return [(case["K"] + 7) // 8 * 8, 256, 256, 256, 256, (case["n_obs"] + 15) // 16 * 16]


def _network(case, seed):
    """He-normal weights (padding rows and columns zero), standardisation and a minibatch of pairs."""
    rng = np.random.default_rng(seed)
    d, K, n_obs = _dims(case), case["K"], case["n_obs"]
    flat = []
    for l in range(5):
        W = rng.standard_normal((d[l + 1], d[l])) * math.sqrt(2.0 / (K if l == 0 else 256))
        b = 0.05 * rng.standard_normal(d[l + 1])
        if l == 0:
            W[:, K:] = 0
        if l == 4:
            W[n_obs:], b[n_obs:] = 0, 0
        flat += [W.ravel(), b]
    theta = rng.standard_normal((case["batch"], K))
    mix = rng.standard_normal((K, n_obs)) / math.sqrt(K)
    mu = np.concatenate([np.full(n_obs, 0.05), np.zeros(d[5] - n_obs)])
    sd = np.concatenate([np.full(n_obs, 0.02), np.ones(d[5] - n_obs)])
    G = mu[:n_obs] + sd[:n_obs] * np.tanh(theta @ mix)
    return np.concatenate(flat).astype(np.float32), np.concatenate([mu, sd]).astype(np.float32), theta, G


def _network_gradients(case, seed):
    d, n_obs = _dims(case), case["n_obs"]
    params, mu_sd, theta, G = _network(case, seed)
    p = torch.from_numpy(params).double().cuda().requires_grad_()
    mu, sd = (torch.from_numpy(v[:n_obs]).double().cuda() for v in (mu_sd[:d[5]], mu_sd[d[5]:]))
    x = torch.zeros((case["batch"], d[0]), dtype=torch.float64, device="cuda")
    x[:, :case["K"]] = torch.from_numpy(theta)
    off = 0
    for l in range(5):
        W = p[off:off + d[l + 1] * d[l]].reshape(d[l + 1], d[l])
        off += W.numel()
        x = x @ W.T + p[off:off + d[l + 1]]
        off += d[l + 1]
        if l < 4:
            x = torch.nn.functional.gelu(x)
    loss = ((x[:, :n_obs] - (torch.from_numpy(G).cuda() - mu) / sd) ** 2).mean()
    loss.backward()
    return dict(grads=p.grad, loss=float(loss))
