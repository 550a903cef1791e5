"""The work a user of this solver has it do, as timed cases through its public entry points.

Four kinds of call, over the sizes, precisions, losses and maps in use:

  fit      a whole training call: create a solver, hand over the data, iterate, read the
           weights back (the set-up of features and cached factors is part of it);
  iterate  further iterations of a solver that already holds its data and factors;
  score    scores of query rows against a trained model that stays resident;
  sweep    iterations of several solvers side by side (one per bandwidth, one lambda per
           output column), the model-selection loop.

A case is a dict of plain values; prepare() draws its inputs from the seed on the GPU.
exact() gives the same results in float64 with plain torch.
"""
import math

import numpy as np
import torch

import paper_1409_0940_gb300 as rff

PHILOX = 11          # seed of the feature draw (a user fixes it once for a model)
MULTICLASS = dict(data="multiclass", d=440, m=147, loss="squared", reg="l2", lam=1e-5, map="fourier")


def _case(kind, **kw):
    c = dict(kind=kind, prec="split_bf16", map="fourier", data="multiclass", loss="squared", reg="l2", lam=1e-5,
             rho=1.0, n=2000, d=16, m=1, D=512, R=1, C=1, iters=10, q=0, host=False, fraction=1.0, degree=2,
             groups=0)
    c.update(kw)
    return c


def listed():
    return [
        # an online service asks for one row at a time, from host memory; a 147-class model
        _case("score", name="score-one-row", q=1, host=True, n=2048, D=16384, R=4, C=4, iters=2, **MULTICLASS),
        # the same service with micro-batches that are not a multiple of any tile
        _case("score", name="score-1000-rows", q=1000, n=2048, D=16384, R=4, C=4, iters=2, **MULTICLASS),
        # offline labelling of a whole data set at full FP32 precision
        _case("score", name="score-50k-rows-fp32", q=50_001, prec="fp32", data="sparse01", d=784, m=10, loss="hinge",
              lam=1e-6, n=2048, D=8192, C=2, iters=2),
        # a small regression from numpy arrays, run to convergence: launches and latency
        _case("fit", name="fit-ridge-2000", prec="fp32", data="ridge", n=2000, d=16, D=512, lam=1e-4, iters=200,
              host=True),
        # an ordinary binary classifier with sizes that divide by nothing
        _case("fit", name="fit-binary-20k", data="binary", loss="hinge", n=20_011, d=33, D=3000, R=2, C=3, iters=50),
        # an ordinary multiclass fit from start to weights, factors included
        _case("fit", name="fit-multiclass-50k", n=50_000, D=8192, R=2, C=2, iters=20, **MULTICLASS),
        # sparse rows from the host (CSR), many thin row blocks: the n_i x n_i projection
        _case("fit", name="fit-sparse-20k", data="sparse01", host=True, loss="hinge", lam=1e-6, n=20_000, d=784, m=10,
              D=32768, R=32, C=8, iters=10),
        # a polynomial-kernel classifier (TensorSketch)
        _case("fit", name="fit-polynomial-10k", prec="cached_z", map="tensorsketch", degree=3, loss="hinge", n=10_000,
              d=128, m=10, D=8192, R=2, C=4, iters=20),
        # the long middle of a training run at the benchmark's size, features regenerated
        _case("iterate", name="iterate-multiclass-200k", n=200_000, D=16384, R=4, C=4, iters=8, **MULTICLASS),
        # the same step at full FP32 precision, on a sample
        _case("iterate", name="iterate-multiclass-20k-fp32", prec="fp32", n=20_000, D=8192, R=2, C=2, iters=4,
              **MULTICLASS),
        # features kept in memory, multinomial logistic loss
        _case("iterate", name="iterate-cached-40k", prec="cached_z", n=40_000, D=8192, R=2, C=2, iters=10,
              **dict(MULTICLASS, loss="multinomial")),
        # a (bandwidth, lambda) grid: four data sets of falling size, eight lambdas each
        _case("sweep", name="sweep-4x8", data="binary", loss="logistic", n=80_000, d=128, m=8, D=8192, groups=4,
              iters=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["score", "score", "fit", "fit", "iterate", "sweep"])
    if kind == "sweep":
        return _case("sweep", data="binary", loss="logistic", groups=rng.randint(2, 5), m=rng.randint(2, 16),
                     n=_log_int(rng, 8000, 80_000), d=_log_int(rng, 16, 256), D=_log_int(rng, 1024, 8192),
                     iters=rng.randint(3, 12), lam=10 ** rng.uniform(-6, -4))
    fmap = rng.choice(["fourier", "fourier", "fourier", "laplace", "tensorsketch"])
    prec = {"fourier": rng.choice(["split_bf16", "split_bf16", "fp32", "cached_z"]),
            "laplace": rng.choice(["fp32", "cached_z"]), "tensorsketch": "cached_z"}[fmap]
    data = "histograms" if fmap == "laplace" else rng.choice(["multiclass", "sparse01", "binary", "ridge"])
    m = 1 if data in ("binary", "ridge") else _log_int(rng, 2, 147)
    loss = {"ridge": rng.choice(["squared", "l1"]), "binary": rng.choice(["hinge", "logistic", "squared"])}.get(
        data, rng.choice(["squared", "hinge", "multinomial", "crammer_singer"]))
    c = _case(kind, data=data, map=fmap, prec=prec, m=m, loss=loss, reg=rng.choice(["l2", "l2", "l1"]),
              lam=10 ** rng.uniform(-6, -4), d=_log_int(rng, 8, 784), D=_log_int(rng, 512, 16384),
              n=_log_int(rng, 1500, 60_000), R=rng.randint(1, 4), C=rng.randint(1, 4), host=rng.random() < 0.3,
              degree=rng.randint(2, 3))
    if fmap == "tensorsketch":
        c["d"] = min(c["d"], 256)
        c["D"] = min(c["D"], 4096 * c["C"])
    if kind == "score":
        c.update(n=rng.randint(1500, 3000), iters=2, q=_log_int(rng, 1, 50_000))
        if fmap == "tensorsketch":
            c["q"] = min(c["q"], 4096)
        return c
    if rng.random() < 0.2:
        c["fraction"] = rng.choice([0.25, 0.5, 0.75])
    c["iters"] = _log_int(rng, 5, 100 if kind == "fit" else 20)
    if fmap == "tensorsketch":
        c["n"] = min(c["n"], 10_000)
    # no dearer than the listed ones: smaller data, then fewer iterations
    limit = 1.5e12 if prec == "fp32" else 8e12
    while work(c)["flops"] > limit and (c["n"] > 1500 or c["iters"] > 5):
        c["n"], c["iters"] = max(1500, c["n"] * 3 // 4), max(5, c["iters"] * 3 // 4)
    return c


# --------------------------------------------------------------------------- inputs
def _rows(case, n, g, dev, part):
    """n rows of the case's kind of data (X float32, labels or targets)."""
    d, m = case["d"], case["m"]
    norm = lambda *s: torch.randn(*s, generator=g, device=dev)   # noqa: E731
    unif = lambda *s: torch.rand(*s, generator=g, device=dev)    # noqa: E731
    kind = case["data"]
    if kind == "ridge":          # a smooth function of uniform inputs, with noise
        X, u = unif(n, d), part["u"]
        return X, (torch.sin(2 * math.pi * (X @ u)) + 0.1 * norm(n)).reshape(n, 1)
    if kind == "binary":         # two overlapping Gaussians
        y = torch.where(unif(n) < 0.5, 1.0, -1.0)
        return y[:, None] * part["mu"] + norm(n, d), y.reshape(n, 1).repeat(1, m)
    lab = torch.randint(0, m, (n,), generator=g, device=dev)
    if kind == "multiclass":     # a Gaussian mixture, standardised
        X = (part["means"][lab] + 2.0 * norm(n, d)) / math.sqrt(5.0)
    elif kind == "sparse01":     # intensities in [0, 1], about a fifth of them not zero
        keep = part["support"][lab] & (unif(n, d) < 0.57)
        X = torch.where(keep, (part["level"][lab] + 0.25 * norm(n, d)).clamp(0, 1), 0.0)
    else:                        # histograms: rows that are nonnegative and sum to 1
        X = part["weights"][lab] * -torch.log(unif(n, d).clamp_min(1e-6))
        X = X / X.sum(1, keepdim=True)
    Y = torch.full((n, m), -1.0, device=dev)
    Y[torch.arange(n, device=dev), lab] = 1.0
    return X, Y


def _inputs(case, seed):
    """(list of (X, Y) per solver, queries or None), float32 on the GPU."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(int(seed) + 1)
    d, m = case["d"], case["m"]
    part = {"u": torch.randn(d, generator=g, device=dev) / math.sqrt(d),
            "mu": 2.0 * torch.randn(d, generator=g, device=dev) / math.sqrt(d),
            "means": torch.randn(m, d, generator=g, device=dev),
            "support": torch.rand(m, d, generator=g, device=dev) < 0.35,
            "level": torch.rand(m, d, generator=g, device=dev)}
    part["weights"] = torch.where(torch.rand(m, d, generator=g, device=dev) < 0.2, 5.0, 0.2)
    sets = [tuple(t.float().contiguous() for t in _rows(case, n, g, dev, part)) for n, _, _, _ in _members(case)]
    q = _rows(case, case["q"], g, dev, part)[0].float().contiguous() if case["q"] else None
    return sets, q


def _sigma(case):
    d = case["d"]
    return {"ridge": 1.0, "binary": math.sqrt(d), "multiclass": math.sqrt(d) / 2, "sparse01": 9.0 * math.sqrt(d / 784),
            "histograms": 8.0 * math.sqrt(d / 440)}[case["data"]] * (2.0 if case["map"] == "tensorsketch" else 1.0)


def _members(case):
    """(n, D, sigma factor, grid) of each solver of the case."""
    if case["kind"] != "sweep":
        return [(case["n"], case["D"], 1.0, (case["R"], case["C"]))]
    out = []
    for k in range(case["groups"]):
        n, D = max(2000, case["n"] >> k), max(512, case["D"] >> (case["groups"] - 1 - k))
        out.append((n, D, 0.5 * 2.0 ** (0.5 * k), (-(-n // 50_000), -(-D // 2048))))
    return out


def _lambdas(case):
    return [case["lam"] * 4.0 ** k for k in range(case["m"])] if case["kind"] == "sweep" else None


def _solvers(case):
    made = []
    for n, D, f, (R, C) in _members(case):
        s = rff.Solver(loss=case["loss"], reg=case["reg"], lam=case["lam"], sigma=f * _sigma(case), rho=case["rho"],
                       D=D, R=R, C=C, seed=PHILOX, m=case["m"], prec=case["prec"], feature_map=case["map"],
                       degree=case["degree"], coef0=1.0)
        if case["kind"] == "sweep":
            s.set_lambdas(_lambdas(case))
        if case["fraction"] < 1.0:
            s.set_block_fraction(case["fraction"])
        made.append(s)
    return made


def prepare(case, seed):
    sets, q = _inputs(case, seed)
    state = {"case": case}
    if case["kind"] == "fit":
        X, Y = sets[0]
        if case["host"] and case["data"] == "sparse01":
            sp = X.cpu().to_sparse_csr()
            state["csr"] = (sp.crow_indices().numpy(), sp.col_indices().numpy().astype(np.int32), sp.values().numpy())
            state["Y"] = Y.cpu().numpy()
        else:
            state["X"], state["Y"] = (X.cpu().numpy(), Y.cpu().numpy()) if case["host"] else (X, Y)
        return state
    solvers = _solvers(case)
    for s, (X, Y) in zip(solvers, sets):
        s.set_data(X, Y)
    if case["kind"] == "sweep":
        rff.rff_sweep_run([s.h for s in solvers], 2)
    else:
        solvers[0].solve(case["iters"] if case["kind"] == "score" else 1, stats=False)
    state["solvers"] = solvers
    state["out"] = [torch.empty(s.D, s.m, device="cuda") for s in solvers]
    if case["kind"] == "score":
        state["q"] = q.cpu().numpy() if case["host"] else q
        shape = (case["q"], case["m"])
        state["scores"] = np.empty(shape, np.float32) if case["host"] else torch.empty(shape, device="cuda")
    return state


def _trained(W, stats):
    # (not the residuals: once a run has converged they are the rounding of its last step)
    return {"W": W, "objective": stats["objective"]}


def run(state):
    case = state["case"]
    if case["kind"] == "score":
        return state["solvers"][0].predict(state["q"], state["scores"])
    if case["kind"] == "iterate":
        s = state["solvers"][0]
        stats = s.solve(case["iters"])
        return _trained(s.weights(state["out"][0]), stats)
    if case["kind"] == "sweep":
        rff.rff_sweep_run([s.h for s in state["solvers"]], case["iters"])
        return [s.weights(o) for s, o in zip(state["solvers"], state["out"])]
    s = _solvers(case)[0]
    if "csr" in state:
        s.set_data_csr(*state["csr"], state["Y"], case["d"])
    else:
        s.set_data(state["X"], state["Y"])
    stats = s.solve(case["iters"])
    W = s.weights() if case["host"] else s.weights(torch.empty(s.D, s.m, device="cuda"))
    s.close()
    return _trained(W, stats)


# --------------------------------------------------------------------------- work
def work(case):
    """Algorithmic bytes (data in, weights or scores out) and flops (each product once)."""
    byts = flops = 0.0
    d, m = case["d"], case["m"]
    for n, D, _, (R, C) in _members(case):
        form = 2.0 * d * D if case["map"] != "tensorsketch" else 2.0 * (case["degree"] - 1) * D * (d + 1)
        if case["kind"] == "score":
            q = case["q"]
            byts += 4.0 * (q * d + d * D + D * m + q * m)
            flops += q * (form + 2.0 * D * m)
            continue
        ni, sj = n / R, D / C
        side = min(ni, sj)
        project = 2.0 * R * C * side * side * m
        stored = case["prec"] == "cached_z"
        iters = case["iters"]
        active = case["fraction"]
        flops += iters * active * (project + 2 * n * ((0 if stored else form) + 2.0 * D * m))
        byts += 4.0 * (n * (d + m) + D * m)
        if stored:   # each of an iteration's two products reads Z (its 32 bits a value)
            byts += 4.0 * 2 * iters * active * n * D
        if case["kind"] == "fit":   # features, Gram matrices (one triangle) and factors
            flops += n * form + R * C * (max(ni, sj) * side * side + side ** 3)
    return {"bytes": byts, "flops": flops}


def tolerance(case):
    # measured against exact(): FP32 up to 1.8e-6; the split precisions up to 1.5e-5 in scores,
    # 2.5e-5 in weights and 2.4e-4 in the small remaining objective of a hinge loss
    if case["prec"] == "fp32":
        return {"rel": 1e-5}
    return {"rel": 6e-5} if case["kind"] == "score" else {"rel": 1e-3}


# --------------------------------------------------------------------------- float64
def _philox(c0, c1, c2, seed):
    """Philox4x32-10 words at counters (c0, c1, c2, 0), int64 tensors of 32-bit values."""
    M = 0xFFFFFFFF
    c0, c1 = torch.broadcast_tensors(c0, c1)
    c = [c0, c1, torch.full_like(c0, c2), torch.zeros_like(c0)]
    k0, k1 = seed & M, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57   # wraps mod 2^64: the low bits and the masked high ones hold
        c = [((p1 >> 32) & M) ^ c[1] ^ k0, p1 & M, ((p0 >> 32) & M) ^ c[3] ^ k1, p0 & M]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c


def _unit(w):
    return ((w >> 8).double() + 0.5) / 2 ** 24


def _features(case, X, D, C, sigma):
    """Z of the rows X in float64."""
    dev, d = X.device, case["d"]
    if case["map"] == "tensorsketch":
        Xa = torch.cat([X / sigma, torch.ones(X.shape[0], 1, dtype=torch.float64, device=dev)], 1)
        blocks = []
        for j, S in enumerate(_sizes(D, C)):
            F = None
            e = torch.arange(case["degree"] * (d + 1), device=dev)
            w = _philox(torch.full_like(e, j), e, 7, PHILOX)
            h = ((w[0] * S) >> 32).reshape(case["degree"], d + 1)
            sgn = (1.0 - 2.0 * (w[1] >> 31).double()).reshape(case["degree"], d + 1)
            for p in range(case["degree"]):
                cs = torch.zeros(X.shape[0], S, dtype=torch.float64, device=dev).index_add_(1, h[p], Xa * sgn[p])
                F = torch.fft.rfft(cs) if F is None else F * torch.fft.rfft(cs)
            blocks.append(math.sqrt(S / D) * torch.fft.irfft(F, n=S))
        return torch.cat(blocks, 1)
    k = torch.arange(D, device=dev)[None, :]
    w = _philox(k, torch.arange(-(-d // 4), device=dev)[:, None], 0, PHILOX)
    g = []
    for a, b in ((w[0], w[1]), (w[2], w[3])):
        r, t = torch.sqrt(-2 * torch.log(_unit(a))), 2 * math.pi * _unit(b)
        g += [r * torch.cos(t), r * torch.sin(t)]
    g = torch.stack(g, 1).reshape(-1, D)[:d]
    if case["map"] == "laplace":
        return torch.exp(-X @ (1.0 / (2 * sigma * sigma * g * g)).float().double()) / math.sqrt(D)
    b = (_unit(_philox(k[0], torch.zeros_like(k[0]), 1, PHILOX)[0]) * math.pi).float().double()
    Z = X @ (g / sigma).float().double()
    return Z.add_(b).cos_().mul_(math.sqrt(2.0 / D))


def _sizes(total, parts):
    return [total // parts + (1 if p < total % parts else 0) for p in range(parts)]


def _loss(case, Y, o):
    loss = case["loss"]
    if loss == "squared":
        return ((Y - o) ** 2).sum()
    if loss == "hinge":
        return (1 - Y * o).clamp_min(0).sum()
    if loss == "l1":
        return (Y - o).abs().sum()
    if loss == "logistic":
        return torch.nn.functional.softplus(-Y * o).sum()
    oc = o.gather(1, Y.argmax(1, keepdim=True))
    if loss == "multinomial":
        return (torch.logsumexp(o, 1, keepdim=True) - oc).sum()
    return (o - oc + (1 - (Y > 0).double())).amax(1).sum()


def _prox(case, v, Y, t):
    loss = case["loss"]
    if loss == "squared":
        return (v + 2 * t * Y) / (1 + 2 * t)
    if loss == "hinge":
        u = Y * v
        return torch.where(u > 1, v, torch.where(u < 1 - t, v + t * Y, Y))
    if loss == "l1":
        return Y + torch.sign(v - Y) * ((v - Y).abs() - t).clamp_min(0)
    if loss == "logistic":   # p - a = t / (1 + e^p), p = y o, by bisection
        lo, hi = Y * v, Y * v + t
        a = lo.clone()
        for _ in range(60):
            mid = (lo + hi) / 2
            below = mid - a - t * torch.sigmoid(-mid) < 0
            lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
        return Y * (lo + hi) / 2
    E = torch.nn.functional.one_hot(Y.argmax(1), Y.shape[1]).double()
    if loss == "crammer_singer":   # o = v - t (a - e_c), a the projection of e_c + (Delta + v) / t on the simplex
        u = E + (1 - E + v) / t
        s = u.sort(1, descending=True).values
        j = torch.arange(1, s.shape[1] + 1, device=v.device)
        tau = (s.cumsum(1) - 1) / j
        r = (s > tau).sum(1, keepdim=True)
        return v - t * ((u - tau.gather(1, r - 1)).clamp_min(0) - E)
    o = v.clone()   # multinomial: Newton steps with the diagonal-plus-rank-one Hessian
    for _ in range(30):
        p = torch.softmax(o, 1)
        g = o - v + t * (p - E)
        Dg, Dp = g / (1 + t * p), p / (1 + t * p)
        step = Dg + t * Dp * ((p * Dg).sum(1, keepdim=True) / (1 - t * (p * Dp).sum(1, keepdim=True)))
        o = o - step * (1.0 / step.norm(dim=1, keepdim=True).clamp_min(1.0))
    return o


def _admm(case, X, Y, n, D, sigma, R, C, iters, fit_stats=True):
    """Wbar, and the objective, after `iters` iterations in float64."""
    Z = _features(case, X, D, C, sigma)
    dev, m, t = X.device, case["m"], 1.0 / case["rho"]
    lam = torch.tensor(_lambdas(case) or [case["lam"]] * m, dtype=torch.float64, device=dev)
    tau = n * lam / case["rho"]
    rows, cols = _sizes(n, R), _sizes(D, C)
    r0 = [sum(rows[:i]) for i in range(R + 1)]
    c0 = [sum(cols[:j]) for j in range(C + 1)]
    inv = {}
    for i in range(R):
        for j in range(C):
            B = Z[r0[i]:r0[i + 1], c0[j]:c0[j + 1]]
            H = B.T @ B if cols[j] <= rows[i] else B @ B.T
            H.diagonal().add_(1.0)
            inv[i, j] = torch.cholesky_inverse(torch.linalg.cholesky(H))
    zero = lambda *s: torch.zeros(*s, dtype=torch.float64, device=dev)   # noqa: E731
    Obar, nu, Wbar, mu = zero(n, m), zero(n, m), zero(D, m), zero(D, m)
    Op, Wij, muij = zero(C, n, m), zero(R, D, m), zero(R, D, m)
    U = zero(n, m)   # Obar_ij + nu_i - O'_ij, the same for every column block
    for k in range(iters):
        active = [[True] * C for _ in range(R)]
        if case["fraction"] < 1.0:
            e = torch.arange(R * C)
            w = _philox(e, torch.full_like(e, k), 2, PHILOX)[0]
            active = ((w >> 8) < int(case["fraction"] * 2 ** 24)).reshape(R, C).tolist()
        O = _prox(case, Obar - nu, Y, t)
        V = Wbar - mu
        W = V / (1 + 2 * tau) if case["reg"] == "l2" else torch.sign(V) * (V.abs() - tau).clamp_min(0)
        for i in range(R):
            rs = slice(r0[i], r0[i + 1])
            for j in range(C):
                if not active[i][j]:
                    continue
                cs = slice(c0[j], c0[j + 1])
                B = Z[rs, cs]
                c, v = Wbar[cs] - muij[i, cs], Op[j, rs] + U[rs]
                if cols[j] <= rows[i]:
                    Wij[i, cs] = inv[i, j] @ (c + B.T @ v)
                else:
                    Wij[i, cs] = c + B.T @ (inv[i, j] @ (v - B @ c))
                Op[j, rs] = B @ Wij[i, cs]
        new = (W + Wij.sum(0)) / (R + 1)
        S = Op.sum(0)
        nbar = (S + C * O) / (C + 1)
        Wbar, Obar = new, nbar
        mu = mu + W - Wbar
        muij = muij + (Wij - Wbar)
        nu = nu + O - Obar
        U = (O - S) / (C + 1) + nu
    if not fit_stats:
        return Wbar, {}
    size = Wbar ** 2 if case["reg"] == "l2" else Wbar.abs()
    return Wbar, {"objective": float(_loss(case, Y, Z @ Wbar) + n * (lam * size).sum())}


def exact(case, seed):
    members = _members(case)
    before = {"fit": 0, "iterate": 1, "sweep": 2, "score": 0}[case["kind"]]
    # float64 work of the factors and iterations (the features once, stored)
    cost = sum(2.0 * n * case["d"] * D + R * C * 4.0 * max(n / R, D / C) * min(n / R, D / C) ** 2 +
               (case["iters"] + before) * 4.0 * n * D * case["m"] for n, D, _, (R, C) in members)
    if cost > 1.2e13:
        return None
    sets, q = _inputs(case, seed)
    got = []
    for (X, Y), (n, D, f, (R, C)) in zip(sets, members):
        got.append(_admm(case, X.double(), Y.double(), n, D, f * _sigma(case), R, C, case["iters"] + before,
                         case["kind"] in ("fit", "iterate")))
    if case["kind"] == "sweep":
        return [W for W, _ in got]
    W, stats = got[0]
    if case["kind"] != "score":
        return _trained(W.cpu().numpy() if case["host"] and case["kind"] == "fit" else W, stats)
    n, D, f, (R, C) = members[0]
    out = torch.cat([_features(case, b.double(), D, C, f * _sigma(case)) @ W for b in q.split(16384)])
    return out.cpu().numpy() if case["host"] else out
