"""What the framework's users have it do, as cases that can be timed.

Each case goes through the package's public entry points on inputs drawn from
a seed.  Kinds of case:

  solve   AMFR-W2 prices of `count` instances of one shape (N axes, level, psi
          or a full grid, FP64 or mixed), or of uneven shapes, through
          solve_batch (host parameters in, host prices out), Batch.run
          (parameters resident, prices into a device array), solve_noalloc, or
          Problem.step / combine / grid_values on a problem kept in time
  gemm    the tensor-core GEMM C = A B^T (BF16 in, FP32 out)
  predict the surrogate ensemble on raw feature rows
  grad    the loss gradient of one surrogate member on one training batch

The parameters follow the package's seeded workloads (workloads.py) and the
paper's market data table.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2408_00559_gb300 import _lib as L
from paper_2408_00559_gb300 import workloads as W

# the paper's market data (Table marketData, Sec. 6), as bench.py uses it
MKT_T = [0.0, 0.5, 1.0, 1.5, 2.0, 2.5]
MKT_F0 = [0.0112, 0.0118, 0.0122, 0.0126, 0.013, 0.0135]
MKT_ALPHA = [0.0, 0.2366, 0.2145, 0.2221, 0.2068, 0.1932]


def _solve(name, **kw):
    c = {"name": name, "kind": "solve", "data": "synthetic", "entry": "solve_batch", "N": 4, "level": 5, "psi": 0,
         "full": False, "precision": "fp64", "bc": "neumann", "payoff": "swaption", "steps": 40, "count": 1}
    c.update(kw)
    return c


def listed():
    return [
        # one caplet on the d=2 full 65x65 grid: the smallest product, priced on request
        _solve("caplet_full65", N=2, level=6, full=True, payoff="caplet", steps=20),
        # one d=4 level-5 swaption on request: 121 small grids
        _solve("swaption_d4_single"),
        # a problem kept on the device and advanced in time a few steps at a
        # time, its component values read back; the earlier Dirichlet faces
        _solve("stepped_d4_dirichlet", level=7, bc="dirichlet", entry="stepped", steps=10),
        # a book of d=4 swaptions revalued in FP64 from resident parameters
        _solve("book_d4_fp64", count=1024, entry="batch"),
        # an uneven book (4, 6, 8 axes, levels 4 to 6) in mixed precision: the
        # batched benchmark workload
        _solve("book_uneven_mixed", N=0, level=0, precision="mixed", count=256, entry="batch"),
        # labels for the surrogate's training set: d=6 family instances, host in and out
        _solve("labels_d6_mixed", data="family", N=6, level=6, precision="mixed", count=512),
        # d=6 modified combination, grids of up to 4096 nodes, mixed precision
        _solve("modified_d6_mixed", N=6, level=6, psi=1, precision="mixed", count=2, entry="batch"),
        # a row of the paper's d=4 sparse-grid table: grids of up to 4096 nodes
        # and lines of up to 4096 rows
        _solve("paper_d4_level12", data="paper", level=12, steps=8),
        # the surrogate's hidden layer on a full prediction chunk
        {"name": "gemm_hidden", "kind": "gemm", "M": 65536, "N": 256, "K": 256},
        # a small ragged product
        {"name": "gemm_small", "kind": "gemm", "M": 1000, "N": 48, "K": 80},
        # price queries answered by the surrogate ensemble
        {"name": "surrogate_queries", "kind": "predict", "members": 4, "rows": 65536},
        # forward and backward pass of one training batch
        {"name": "surrogate_grad", "kind": "grad", "rows": 1024},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single", "single", "stepped", "book", "book", "uneven", "labels", "modified", "paper",
                       "gemm", "predict", "grad"])
    prec = rng.choice(["fp64", "mixed"])
    c = None
    if kind == "single":
        N = rng.randint(2, 6)
        full = N <= 3 and rng.random() < 0.5
        level = rng.randint(4, 7 if N == 2 else 4) if full else rng.randint(3, 6 if N > 4 else 8)
        c = _solve("", N=N, level=level, full=full, precision=prec, payoff=rng.choice(["caplet", "swaption"]),
                   steps=rng.randint(8, 64), bc=rng.choice(["neumann", "neumann", "dirichlet"]),
                   entry=rng.choice(["solve_batch", "solve_batch", "noalloc"]))
    elif kind == "stepped":
        c = _solve("", N=rng.randint(2, 5), level=rng.randint(3, 8), precision=prec, entry="stepped",
                   steps=rng.randint(1, 20), bc=rng.choice(["neumann", "dirichlet"]))
    elif kind == "book":
        N = rng.randint(3, 8)
        top = {3: 1024, 4: 1024, 5: 256, 6: 96, 7: 24, 8: 8}[N] * (4 if prec == "mixed" and N > 4 else 1)
        c = _solve("", N=N, level=rng.randint(3, 6), precision=prec, count=_log_int(rng, 2, top),
                   steps=rng.randint(10, 40), entry=rng.choice(["batch", "solve_batch"]))
        if N == 4 and c["level"] == 6:
            c["count"] = (c["count"] + 1) // 2
    elif kind == "uneven":
        c = _solve("", N=0, level=0, precision=prec, entry="batch",
                   count=_log_int(rng, 3, 256 if prec == "mixed" else 48))
    elif kind == "labels":
        c = _solve("", data="family", N=6, level=rng.randint(4, 6), precision="mixed", count=_log_int(rng, 16, 512))
    elif kind == "modified":
        N = rng.randint(3, 6)
        c = _solve("", N=N, level=rng.randint(3, 5 if N == 6 and prec == "fp64" else 6), psi=1, precision=prec,
                   entry="batch", count=rng.randint(1, 2), steps=rng.randint(8, 24))
    elif kind == "paper":
        N = rng.choice([3, 4])
        c = _solve("", data="paper", N=N, level=rng.randint(8, 11), steps=_log_int(rng, 4, 48 if N == 3 else 8))
    elif kind == "gemm":
        c = {"kind": "gemm", "M": _log_int(rng, 64, 65536), "N": rng.choice([16, 48, 128, 240, 256, 512]),
             "K": 16 * _log_int(rng, 1, 32)}
        if c["N"] == 512:
            c["M"] = (c["M"] + 1) // 2
    elif kind == "predict":
        c = {"kind": "predict", "members": rng.randint(2, 5), "rows": _log_int(rng, 100, 65536)}
    else:
        c = {"kind": "grad", "rows": 16 * rng.randint(1, 64)}
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs
def _paper_instance(N, level, steps, rng):
    nr = N - 1
    T = np.array(MKT_T[1:1 + nr])
    th = W.THETA_W2
    return dict(N=N, payoff="swaption", n_steps=steps, alpha=np.array(MKT_ALPHA[1:1 + nr]),
                phi=np.full(nr, rng.uniform(0.2, 0.4)), tau=np.full(nr, 0.5), F0=np.array(MKT_F0[1:1 + nr]),
                Fmax=np.full(nr, 0.04), Vmax=3.5, rho=np.exp(-0.1 * np.abs(T[:, None] - T[None, :])),
                sigma=rng.uniform(0.2, 0.4), beta=1.0, V0=1.0, K=rng.uniform(0.010, 0.012), T=MKT_T[1], theta=th,
                nu=(N - 1) * th, discount=1.0 / (1.0 + 0.5 * MKT_F0[0]), level=level, psi=0, full=False,
                precision="fp64")


def _instances(case, seed):
    n, steps = case["count"], case["steps"]
    base = (seed % 1000003) * 4096
    if case["data"] == "paper":
        rng = np.random.default_rng(base)
        return [_paper_instance(case["N"], case["level"], steps, rng) for _ in range(n)]
    if case["data"] == "family":
        return W.c5_instances(n, start=base, level=case["level"], steps=steps, precision=case["precision"],
                              box="configured_strikes")
    out = []
    for i in range(n):
        N = case["N"] or (4, 6, 8)[i % 3]
        level = case["level"] or (4, 5, 6)[(i // 3) % 3]
        x = W.small_instance(N, level, psi=case["psi"], steps=steps, seed=base + i, precision=case["precision"],
                             full=case["full"], payoff=case["payoff"])
        x["bc"] = case["bc"]
        out.append(x)
    return out


def _weights(rng):
    """FP32 parameters of one member, He-initialised like the library's own."""
    p = np.zeros(L.SURROGATE_PARAMS, dtype=np.float32)
    scale = {"W1": math.sqrt(2.0 / 8), "W2": math.sqrt(2.0 / 256), "W3": math.sqrt(2.0 / 256),
             "w4": math.sqrt(1.0 / 256), "b1": 0.1, "b2": 0.1, "b3": 0.1, "b4": 0.1}
    for name, (o, size) in L.surrogate_layout().items():
        p[o:o + size] = rng.standard_normal(size) * scale[name]
    w1 = p[:256 * 16].reshape(256, 16)
    w1[:, 8:] = 0.0  # the input's padding
    return p


def _surrogate_set(case, seed):
    """Training rows, their labels, query rows and member weights."""
    rng = np.random.default_rng(seed)
    train = W.c5_features(1024, start=seed % 1000003, box="configured_strikes")
    f = train
    prices = 0.05 * f[:, 0] * np.sqrt(f[:, 4]) * np.exp(0.5 * f[:, 1] - 0.3 * f[:, 6]) * np.exp(-20.0 * (f[:, 3] - 0.02))
    prices *= np.exp(0.05 * rng.standard_normal(len(prices)))
    q = np.empty((case["rows"], 8))
    B = W.C5_BOXES["configured_strikes"]
    for c, key in enumerate(("alpha", "sigma", "beta", "K", "T", "lam", "phi", "phi")):
        q[:, c] = rng.uniform(*B[key], size=len(q))
    q[:, 3] = rng.choice(np.unique(train[:, 3]), size=len(q))
    weights = [_weights(rng) for _ in range(case["members"])]
    return train, prices, q, weights


def _gemm_operands(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn(case["M"], case["K"], device="cuda", generator=g).to(torch.bfloat16)
    b = torch.randn(case["N"], case["K"], device="cuda", generator=g).to(torch.bfloat16)
    return a, b / math.sqrt(case["K"])


def _grad_rows(case, seed):
    rng = np.random.default_rng(seed)
    x = rng.uniform(-1.0, 1.0, size=(case["rows"], 8)).astype(np.float32)
    t = rng.standard_normal(case["rows"]).astype(np.float32)
    return x, t, _weights(rng)


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "solve":
        s["insts"] = _instances(case, seed)
        if case["entry"] == "batch":
            s["batch"] = L.Batch(s["insts"])
        elif case["entry"] == "stepped":
            s["problem"] = L.Problem(s["insts"][0])
        s["prices"] = torch.zeros(case["count"], dtype=torch.float64, device="cuda")
    elif case["kind"] == "gemm":
        s["a"], s["b"] = _gemm_operands(case, seed)
        s["c"] = torch.zeros(case["M"], case["N"], device="cuda")
    elif case["kind"] == "predict":
        train, prices, s["queries"], weights = _surrogate_set(case, seed)
        s["net"] = L.Surrogate(case["members"], seed=seed % 1000)
        s["net"].fit([W.c5_instance_from(f, box="configured_strikes") for f in train], prices, epochs=1)
        for m, p in enumerate(weights):
            s["net"].params(m, p)
    else:
        s["x"], s["t"], p = _grad_rows(case, seed)
        s["net"] = L.Surrogate(1, seed=1)
        s["net"].params(0, p)
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "gemm":
        L.tc_gemm_bf16(s["a"], s["b"], s["c"])
        return s["c"]
    if case["kind"] == "predict":
        mean, spread, ok = s["net"].predict_features(s["queries"])
        return {"mean": mean, "spread": spread, "in_box": ok}
    if case["kind"] == "grad":
        g, loss = s["net"].grad(0, s["x"], s["t"])
        return {"grad": g, "loss": np.float32(loss)}  # (the C entry point's float)
    if case["entry"] == "batch":
        s["batch"].run(s["prices"].data_ptr())
        return s["prices"]
    if case["entry"] == "noalloc":
        L.solve_noalloc(s["insts"], s["prices"].data_ptr())
        return s["prices"]
    if case["entry"] == "stepped":
        p = s["problem"]
        p.step(case["steps"])
        return {"price": p.combine(), "values": p.grid_values()}
    return L.solve_batch(s["insts"])


# ------------------------------------------------------- work of one pass
def _levels(N, level, psi, full):
    """(levels, coefficient) of every component grid in the library's order."""
    if full:
        return [((level,) * N, 1.0)]
    out = []

    def rec(prefix, m, coef):
        if len(prefix) == N - 1:
            out.append((tuple(psi + v for v in (*prefix, m)), coef))
            return
        for v in range(m + 1):
            rec((*prefix, v), m - v, coef)

    for q in range(min(N - 1, level) + 1):
        rec((), level - q, (-1.0) ** q * math.comb(N - 1, q))
    return out


def _grid_flops(lv, steps):
    """Operations of the method on one component grid (a multiply-add counts
    two): per step 4 evaluations of F (Sketch 1: second differences on every
    axis, cross differences and drift off the upper faces), 4N Thomas solves
    with known factors, and the stage algebra."""
    N = len(lv)
    off = [1.0 - 0.5 ** v for v in lv]  # share of nodes off an axis's upper face
    f = 3 * N + 1 + 4 * (N - 1)
    f += sum(off[i] * (2 * i + 4) for i in range(1, N - 1))
    f += sum(off[i] * off[k] * (6 if k < N - 1 else 5) for i, k in itertools.combinations(range(N), 2))
    thomas = 4 * sum(5 - 4 * 0.5 ** v for v in lv)
    return 2.0 ** sum(lv) * (4 * f + thomas + 24) * steps


_FLOPS = {}


def work(case):
    if case["kind"] == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2 * K * (M + N) + 4 * M * N, "flops": 2 * M * N * K}
    layers = 2 * (8 * 256 + 2 * 256 * 256 + 256)
    if case["kind"] == "predict":
        n = case["rows"]
        return {"bytes": n * (64 + 17) + 4 * case["members"] * L.SURROGATE_PARAMS,
                "flops": n * (case["members"] * layers + 2 * 165)}
    if case["kind"] == "grad":
        return {"bytes": 36 * case["rows"] + 8 * L.SURROGATE_PARAMS, "flops": 3 * layers * case["rows"]}
    flops = nbytes = 0.0
    for i in range(case["count"]):
        N = case["N"] or (4, 6, 8)[i % 3]
        level = case["level"] or (4, 5, 6)[(i // 3) % 3]
        key = (N, level, case["psi"], case["full"], case["steps"])
        if key not in _FLOPS:
            grids = _levels(*key[:4])
            _FLOPS[key] = (sum(_grid_flops(lv, case["steps"]) for lv, _ in grids),
                           sum(16 * 2 ** sum(lv) + 8 for lv, _ in grids))
        flops += _FLOPS[key][0]
        nbytes += 8 * (5 * N + N * N + 10) + (_FLOPS[key][1] if case["entry"] == "stepped" else 0)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------- the same results in 64 bits
def _axis(t, axis, s):
    """The rows j = 1..M of an axis of M + 1 rows, displaced by s; the row
    beyond the upper face is the mirror of the one below it."""
    n = t.shape[axis]
    if s == 0:
        return t.narrow(axis, 1, n - 1)
    if s < 0:
        return t.narrow(axis, 0, n - 1)
    return torch.cat([t.narrow(axis, 2, n - 2), t.narrow(axis, n - 2, 1)], axis)


def _solve_grid(insts, lv, dev):
    """Values interpolated at the spot [B] of one component grid for instances
    of one shape: tensors are [instance, vector, axis 0, ..., axis N-1]."""
    x0 = insts[0]
    N, steps, B = x0["N"], x0["n_steps"], len(insts)
    nr = N - 1
    M = [1 << v for v in lv]
    n_in = int(np.prod(M))

    def par(get):
        return torch.tensor([float(get(x)) for x in insts], dtype=torch.float64, device=dev).reshape([B] + [1] * (N + 1))

    def along(vals, axis, outer):  # vals: [B, rows] -> broadcastable
        shape = [B, 1] + [1] * N
        shape[2 + axis] = M[axis] + (1 if outer else 0)
        return vals.reshape(shape)

    h = [par(lambda x, i=i: (x["Fmax"][i] if i < nr else x["Vmax"]) / M[i]) for i in range(N)]
    full = [along(h[i].reshape(B, 1) * torch.arange(0, M[i] + 1, device=dev, dtype=torch.float64), i, True) for i in range(N)]
    inner = [_axis(full[i], 2 + i, 0) for i in range(N)]
    V2 = inner[nr] ** 2
    beta, sigma = par(lambda x: x["beta"]), par(lambda x: x["sigma"])
    al = [par(lambda x, i=i: x["alpha"][i]) for i in range(nr)]
    tau = [par(lambda x, i=i: x["tau"][i]) for i in range(nr)]
    rho = [[par(lambda x, i=i, k=k: x["rho"][i][k]) for k in range(nr)] for i in range(nr)]
    pw = [al[i] * inner[i] ** beta for i in range(nr)]
    d = [0.5 * rho[i][i] * pw[i] ** 2 * V2 / h[i] ** 2 for i in range(nr)] + [0.5 * sigma ** 2 * V2 / h[nr] ** 2]
    mix = {}
    for i, k in itertools.combinations(range(N), 2):
        if M[i] > 1 and M[k] > 1:
            mix[i, k] = (rho[i][k] * pw[i] * pw[k] if k < nr else sigma * par(lambda x, i=i: x["phi"][i]) * pw[i]) \
                * V2 / (4 * h[i] * h[k])
    drift = {}
    for i in range(1, nr):
        if M[i] > 1:
            S = sum(rho[i][r] * pw[r] * tau[r] / (1 + tau[r] * inner[r]) for r in range(1, i + 1))
            drift[i] = pw[i] * S * V2 / (2 * h[i])
    # payoff on every node, Outer ones included
    K = par(lambda x: x["K"])
    if x0["payoff"] == "caplet":
        G = (full[0] - K).clamp(min=0)
    else:
        P, G = 1.0, 0.0
        for i in range(nr):
            P = P / (1 + tau[i] * full[i])
            G = G + tau[i] * (full[i] - K) * P
        G = G.clamp(min=0)
    G = G.expand([B, 1] + [m + 1 for m in M])

    def F(E):
        core = E
        for a in range(N):
            core = _axis(core, 2 + a, 0)

        def at(T, skip):
            for a in range(N):
                if a not in skip:
                    T = _axis(T, 2 + a, 0)
            return T
        out = 0.0
        for i in range(N):
            p, m = _axis(E, 2 + i, 1), _axis(E, 2 + i, -1)
            out = out + d[i] * at(p - 2 * _axis(E, 2 + i, 0) + m, (i,))
            if i in drift:
                out = out + drift[i] * at(p - m, (i,))
            for k in range(i + 1, N):
                if (i, k) in mix:
                    q = p - m
                    out = out + mix[i, k] * at(_axis(q, 2 + k, 1) - _axis(q, 2 + k, -1), (i, k))
        return out

    pad = [1, 0] * N
    dt = par(lambda x: x["T"] / x["n_steps"])
    th, nudt = par(lambda x: x["theta"]), par(lambda x: x["nu"]) * dt

    def F0(X):
        return F(torch.nn.functional.pad(X, pad))

    FG = F(G)

    def S(X):
        for a in range(N):
            nd = nudt * d[a]
            if M[a] == 1:
                X = X / (1 + 2 * nd)
                continue
            nd = nd.expand([B, 1] + list(nd.shape[2:])).expand(-1, -1, *[max(s, 1) for s in nd.shape[2:]])
            rows = [t.unsqueeze(2 + a) for t in X.unbind(2 + a)]
            nds = [t.unsqueeze(2 + a) for t in nd.unbind(2 + a)] if nd.shape[2 + a] > 1 else [nd] * M[a]
            gam, y = [], []
            for j in range(M[a]):
                lo = 0.0 if j == 0 else (-nds[j] if j < M[a] - 1 else -2 * nds[j])
                piv = 1 + 2 * nds[j] - (lo * gam[-1] if j else 0.0)
                gam.append(-nds[j] / piv)
                y.append((rows[j] - (lo * y[-1] if j else 0.0)) / piv)
            for j in range(M[a] - 2, -1, -1):
                y[j] = y[j] - gam[j] * y[j + 1]
            X = torch.cat(y, 2 + a)
        return X

    def stage(r):
        k = S(r)
        return S(2 * r - k + th * dt * F0(k))

    def step(Z):
        r = dt * (FG + F0(Z))
        K1 = stage(r)
        K2 = stage(r + (2.0 / 3.0) * dt * F0(K1) - (4.0 / 3.0) * K1)
        return Z + 1.25 * K1 + 0.75 * K2

    Z = torch.zeros([B, 1] + M, dtype=torch.float64, device=dev)
    if n_in <= 64 and n_in <= 2 * steps:
        # the step is affine and the same every time: its matrix once, then products
        eye = torch.eye(n_in, dtype=torch.float64, device=dev).reshape([1, n_in] + M)
        c = step(Z).reshape(B, 1, n_in)
        R = step(eye.expand([B] + [-1] * (N + 1))).reshape(B, n_in, n_in) - c
        z = Z.reshape(B, 1, n_in)
        for _ in range(steps):
            z = torch.bmm(z, R) + c
        Z = z.reshape([B, 1] + M)
    else:
        for _ in range(steps):
            Z = step(Z)
    U = torch.nn.functional.pad(Z, pad) + G
    for a in range(N):
        w = torch.zeros(B, M[a] + 1, dtype=torch.float64, device=dev)
        for b, x in enumerate(insts):
            s = (x["F0"][a] / x["Fmax"][a] if a < nr else x["V0"] / x["Vmax"]) * M[a]
            j = min(max(int(math.floor(s)), 0), M[a] - 1)
            w[b, j], w[b, j + 1] = 1 - (s - j), s - j
        U = (U * along(w, a, True)).sum(2 + a, keepdim=True)
    return U.reshape(B)


def _exact_cost(case):
    """Rough tensor operations of _solve_grid over the case's grids."""
    ops = 0.0
    for lv, _ in _levels(case["N"], case["level"], case["psi"], case["full"]):
        act = sum(v > 0 for v in lv)
        one = 4 * (10 * case["N"] + 6 * act * act + sum(6 << v if v else 1 for v in lv))
        n_in = 1 << sum(lv)
        once = n_in <= min(64, 2 * case["steps"])
        ops += one * (2 if once else case["steps"]) * (1 + 1e-6 * case["count"] * n_in * (n_in if once else 1))
        ops += 2 * case["steps"]
    return ops


def _exact_solve(case, seed):
    if case["data"] == "paper" or case["N"] == 0 or case["bc"] != "neumann" or _exact_cost(case) > 4e6:
        return None
    # few instances are launch-bound on a GPU: the host is quicker
    dev = "cuda" if case["count"] > 8 else "cpu"
    torch.set_num_threads(1 if dev == "cpu" else torch.get_num_threads())
    insts = _instances(case, seed)
    if case["entry"] == "stepped":
        dt = insts[0]["T"] / insts[0]["n_steps"]
        insts = [dict(x, n_steps=case["steps"], T=dt * case["steps"]) for x in insts]
    values, coefs = [], []
    for lv, coef in _levels(case["N"], case["level"], case["psi"], case["full"]):
        values.append(_solve_grid(insts, lv, dev))
        coefs.append(coef)
    u = torch.stack(values, 1)
    prices = (u * torch.tensor(coefs, dtype=torch.float64, device=dev)).sum(1)
    prices = prices * torch.tensor([x.get("discount", 1.0) for x in insts], dtype=torch.float64, device=dev)
    if case["entry"] == "stepped":
        return {"price": float(prices[0]), "values": u[0].cpu().numpy()}
    return prices.cpu().numpy()


def _split(p):
    return {k: torch.tensor(p[o:o + n], dtype=torch.float64) for k, (o, n) in L.surrogate_layout().items()}


def _forward(p, x):
    z, h = [], [x]
    for k in (1, 2, 3):
        w = p["W%d" % k].reshape(256, -1)[:, :h[-1].shape[1]]
        z.append(h[-1] @ w.T + p["b%d" % k])
        h.append(0.5 * z[-1] * (1 + torch.erf(z[-1] / math.sqrt(2.0))))
    return h[-1] @ p["w4"] + p["b4"], z, h


def _exact_predict(case, seed):
    train, prices, q, weights = _surrogate_set(case, seed)
    # the family's features as the library reads them back from an instance
    train = train.copy()
    train[:, 5] = -np.log(np.exp(-train[:, 5]))
    lo, hi = train.min(0), train.max(0)
    span = np.where(hi > lo, hi - lo, 1.0)

    def norm(f):
        z = np.where(hi > lo, 2 * (f - lo) / span - 1, np.where(f == lo, 0.0, 2.0))
        return z

    def cubic(z):
        z = z.astype(np.float32).astype(np.float64)
        cols = [np.ones(len(z))]
        for deg in (1, 2, 3):
            cols += [np.prod(z[:, list(ix)], axis=1) for ix in itertools.combinations_with_replacement(range(8), deg)]
        return np.stack(cols, 1)

    y = np.log(prices)
    A = cubic(norm(train))
    H = A.T @ A
    coef = np.linalg.solve(H + np.eye(len(H)) * (1e-12 * np.trace(H) / len(H) + 1e-300), A.T @ y)
    res = y - A @ coef
    mu, sd = res.mean(), math.sqrt(max(res.var(), 1e-300))
    zq = norm(q)
    ok = np.all((zq >= -1 - 1e-9) & (zq <= 1 + 1e-9), axis=1)
    x = torch.tensor(zq.astype(np.float32).astype(np.float64), device="cuda")
    outs = torch.stack([_forward({k: v.cuda() for k, v in _split(p).items()}, x)[0] for p in weights])
    g = cubic(zq) @ coef + mu + sd * outs.mean(0).cpu().numpy()
    spread = outs.std(0, unbiased=True).cpu().numpy() * sd * np.exp(g)
    return {"mean": np.exp(g), "spread": spread, "in_box": ok}


def _exact_grad(case, seed):
    x, t, p = _grad_rows(case, seed)
    p = _split(p)
    x = torch.tensor(x.astype(np.float64))
    y, z, h = _forward(p, x)
    r = y - torch.tensor(t.astype(np.float64))
    g = {}
    dy = r / len(r)
    g["w4"], g["b4"] = h[3].T @ dy, dy.sum().reshape(1)
    up = dy[:, None] * p["w4"]
    for k in (3, 2, 1):
        zk = z[k - 1]
        dz = up * (0.5 * (1 + torch.erf(zk / math.sqrt(2.0))) + zk * torch.exp(-0.5 * zk ** 2) / math.sqrt(2 * math.pi))
        w = dz.T @ h[k - 1]
        g["W%d" % k] = torch.nn.functional.pad(w, (0, 8)) if k == 1 else w
        g["b%d" % k] = dz.sum(0)
        up = dz @ p["W%d" % k].reshape(256, -1)
    out = np.zeros(L.SURROGATE_PARAMS)
    for k, (o, n) in L.surrogate_layout().items():
        out[o:o + n] = g[k].reshape(-1).numpy()
    return {"grad": out, "loss": 0.5 * float((r * r).mean())}


def exact(case, seed):
    if case["kind"] == "solve":
        return _exact_solve(case, seed)
    if case["kind"] == "predict":
        return _exact_predict(case, seed)
    if case["kind"] == "grad":
        return _exact_grad(case, seed)
    a, b = _gemm_operands(case, seed)
    return a.double() @ b.double().T
