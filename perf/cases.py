"""Timed cases of the GaBP SVM solver: the calls a program makes, over the sizes it makes them with.

A case is a dict of plain values.  ``prepare`` makes its inputs from a seed (and, where a program keeps one,
the solver handle), ``run`` is one pass through the public entry points of ``paper_0810_1648_gb300.gabp``,
``work`` counts what such a pass cannot do without, and ``exact`` gives the same outputs in 64 bits (the
linear solve that the belief propagation converges to, and FP64 kernel sums), without the package's code.

Kinds of pass:

* ``train``     a solver made from new data, solved, asked for the means and for decision values, closed;
* ``retrain``   a kept solver refitted with a data set and solved again;
* ``batch``     a C x gamma grid over several data sets solved together;
* ``serve``     a continuous-batching server that is given requests and stepped until all are done;
* ``decide``    decision values of a trained solver for new rows;
* ``decide_noalloc``  the same from a program's own arrays, without a solver.
"""
import math
import random

import numpy as np
import torch

from paper_0810_1648_gb300 import gabp, workloads

Q_MODES = {"f32": gabp.Q_F32, "bf16": gabp.Q_BF16, "recompute": gabp.Q_RECOMPUTE}
GRID_C = (0.1, 1.0, 10.0, 100.0)
GRID_GAMMA = (0.1, 0.5, 1.0, 2.0)   # times 1 / m
TO_TOLERANCE_ROUNDS = 20            # rounds counted by work() for a solve to a tolerance


def listed():
    return [
        # The smallest training call: 1000 x 10 FP64 host data (two Gaussian classes), to 1e-6, with the
        # decision values of a small test set.  Launches and host work count.
        dict(name="train_small_host64", kind="train", data="two_gaussians", n=1000, m=10, gm=1.0, C=1.0, q="f32",
             iters=200, tol=1e-6, host=True, fp64=True, t=200),
        # An ordinary training call on device data, odd sizes and many features (the shape of a speech set
        # that Section 5 of the paper times).
        dict(name="train_mid_wide", kind="train", data="mixture", n=6238, m=617, gm=1.0, C=1.0, q="f32",
             iters=200, tol=1e-6, t=1559),
        # The plain form at its large size: a kept solver, new data, 100 synchronous rounds.
        dict(name="retrain_large_100", kind="retrain", data="mixture", n=20000, m=128, gm=1.0, C=10.0, q="f32",
             iters=100, tol=0.0),
        # Kernel ridge regression with the four-stage schedule, few features.
        dict(name="retrain_krr_staged", kind="retrain", data="mixture", n=12960, m=25, gm=1.0, C=1.0, q="f32",
             iters=200, tol=1e-6, krr=True, stages=4),
        # The largest: the precision form (BF16 Q and messages, refined to the FP32 matrix).
        dict(name="retrain_precision", kind="retrain", data="mixture", n=100000, m=64, gm=0.5, C=1.0, q="bf16",
             msg_bf16=True, refine=10, iters=200, tol=1e-6),
        # The precision form that does not store Q.
        dict(name="retrain_recompute", kind="retrain", data="mixture", n=30011, m=100, gm=1.0, C=1.0,
             q="recompute", msg_bf16=True, refine=10, iters=200, tol=1e-6),
        # A narrow kernel on rows ordered by cluster: the tile-sparse option.
        dict(name="retrain_tile_sparse", kind="retrain", data="clustered", n=20000, m=64, gm=9.6, C=1.0, q="f32",
             iters=200, tol=1e-6, tau=1e-3),
        # A parameter grid over few data sets: the plain form, synchronous.
        dict(name="batch_grid_plain", kind="batch", datasets=6, sizes=3, n_lo=200, n_hi=4000, q="f32", iters=200,
             tol=1e-6),
        # The whole grid search: 512 uneven problems, BF16 refined, four stages.
        dict(name="batch_grid_bf16_staged", kind="batch", datasets=32, sizes=100, n_lo=200, n_hi=4000, q="bf16",
             msg_bf16=True, refine=10, stages=4, iters=200, tol=1e-6),
        # A burst of training requests from host memory through the server.
        dict(name="serve_burst", kind="serve", requests=24, sizes=7, n_lo=500, n_hi=12000, m_lo=16, m_hi=512,
             q="f32", stages=4, iters=200, tol=1e-6),
        # Prediction of a large test set with a large model.
        dict(name="decide_large", kind="decide", data="mixture", n=20000, m=128, gm=1.0, C=10.0, t=10000),
        # Prediction of a few rows in a serving loop that cannot allocate.
        dict(name="decide_few_noalloc", kind="decide_noalloc", data="mixture", n=2000, m=32, gm=1.0, C=1.0, t=64),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["train", "train", "retrain", "retrain", "retrain", "batch", "serve", "decide",
                       "decide_noalloc"])
    C = round(_log(rng, 0.1, 100.0), 3)
    gm = round(_log(rng, 0.1, 2.0), 3)
    if kind == "train":
        return dict(kind=kind, data=rng.choice(["mixture", "two_gaussians"]), n=int(_log(rng, 200, 12000)),
                    m=int(_log(rng, 4, 800)), gm=gm, C=C, q=rng.choice(["f32", "f32", "bf16"]), refine=10,
                    iters=200, tol=1e-6, host=rng.random() < 0.5, fp64=rng.random() < 0.3,
                    stages=rng.choice([1, 1, 4]), t=int(_log(rng, 50, 5000)))
    if kind == "retrain":
        q = rng.choice(["f32", "f32", "bf16", "recompute"])
        case = dict(kind=kind, data="mixture", n=int(_log(rng, 2000, 40000)), m=int(_log(rng, 8, 300)), gm=gm, C=C,
                    q=q, iters=200, tol=1e-6, stages=rng.choice([1, 1, 2, 4]))
        if q == "f32" and rng.random() < 0.5:
            case.update(iters=100, tol=0.0, stages=1)
        if q == "f32" and rng.random() < 0.3:
            case.update(krr=True)
        if q != "f32":
            case.update(refine=10, msg_bf16=rng.random() < 0.7)
        if q == "f32" and rng.random() < 0.3:
            case.update(data="clustered", gm=round(_log(rng, 4.0, 10.0), 3), tau=1e-3, m=64)
        return case
    if kind == "batch":
        q = rng.choice(["f32", "bf16"])
        case = dict(kind=kind, datasets=rng.randint(2, 12), sizes=rng.randint(1000, 9999), n_lo=200, n_hi=4000, q=q,
                    stages=rng.choice([1, 4]), iters=200, tol=1e-6)
        if q == "bf16":
            case.update(msg_bf16=True, refine=10)
        return case
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(4, 32), sizes=rng.randint(1000, 9999), n_lo=500,
                    n_hi=int(_log(rng, 2000, 12000)), m_lo=16, m_hi=512, q="f32", stages=rng.choice([1, 4]), iters=200,
                    tol=1e-6)
    if kind == "decide":
        return dict(kind=kind, data="mixture", n=int(_log(rng, 300, 25000)), m=int(_log(rng, 4, 500)), gm=gm, C=C,
                    t=int(_log(rng, 1, 20000)))
    n = int(_log(rng, 100, 10000))
    t = int(_log(rng, 1, 4000))
    return dict(kind=kind, data="mixture", n=n, m=int(_log(rng, 4, 300)), gm=gm, C=C,
                t=max(1, min(t, (1 << 19) // (n // 128 + 2))))


# ---------------------------------------------------------------- inputs
def _gen(seed, *more):
    g = torch.Generator(device="cuda")
    h = seed
    for v in more:
        h = (h * 1000003 + int(v) + 12345) % (1 << 62)
    g.manual_seed(h)
    return g


def _rows(data, n, m, g):
    """Features (n x m, FP32) and labels +-1: two classes, each one Gaussian (``two_gaussians``, means +-1/2) or
    three components with means N(0, I) and spread 0.7, rows shuffled, or ordered by component (``clustered``)."""
    def randn(*shape):
        return torch.randn(*shape, generator=g, device="cuda")
    y = torch.ones(n, device="cuda")
    y[n - n // 2:] = -1.0
    if data == "two_gaussians":
        X = randn(n, m) + 0.5 * y[:, None]
        p = torch.randperm(n, generator=g, device="cuda")
    else:
        means = randn(2, 3, m)
        cls = (y < 0).long()
        comp = torch.randint(0, 3, (n,), generator=g, device="cuda")
        X = means[cls, comp] + 0.7 * randn(n, m)
        p = (torch.argsort(cls * 3 + comp, stable=True) if data == "clustered"
             else torch.randperm(n, generator=g, device="cuda"))
    return X[p].contiguous(), y[p].contiguous()


def _targets(X, g):
    """Regression targets sin(<w, x>) + 0.1 N(0, 1), w ~ N(0, I / m)."""
    w = torch.randn(X.shape[1], generator=g, device="cuda") / math.sqrt(X.shape[1])
    return torch.sin((X * w).sum(dim=1)) + 0.1 * torch.randn(X.shape[0], generator=g, device="cuda")


def _test_rows(X, t, g):
    i = torch.randint(0, X.shape[0], (t,), generator=g, device="cuda")
    return X[i] + 0.5 * torch.randn(t, X.shape[1], generator=g, device="cuda")


def _inputs(case, seed):
    """{X, y, Xt, gamma} on the GPU (FP32 values), also for the cases that hand them over from the host."""
    g = _gen(seed, case["n"], case["m"])
    X, y = _rows(case["data"], case["n"], case["m"], g)
    if case.get("krr"):
        y = _targets(X, g)
    Xt = _test_rows(X, case["t"], g) if case.get("t") else None
    return X, y, Xt, case["gm"] / case["m"]


def _grid_sizes(case):
    """(n, m) of every data set of a batch, or of every request: of the case, not of the seed."""
    r = random.Random(case["sizes"])
    if case["kind"] == "batch":
        return [(int(round(_log(r, case["n_lo"], case["n_hi"]))), r.choice([8, 32, 128, 256]))
                for _ in range(case["datasets"])]
    return [(int(round(_log(r, case["n_lo"], case["n_hi"]))), int(round(_log(r, case["m_lo"], case["m_hi"]))))
            for _ in range(case["requests"])]


def _problems(case, seed):
    """[(X, y, gamma, C)] of a batch (a grid over each data set) or of a server's requests, on the GPU."""
    out = []
    r = random.Random(case["sizes"] + 1)
    for d, (n, m) in enumerate(_grid_sizes(case)):
        X, y = _rows("mixture", n, m, _gen(seed, n, m, d))
        if case["kind"] == "batch":
            out += [(X, y, gm / m, C) for C in GRID_C for gm in GRID_GAMMA]
        else:
            out.append((X, y, 1.0 / m, _log(r, 0.1, 100.0)))
    return out


def _options(case):
    o = dict(q_mode=Q_MODES[case.get("q", "f32")])
    if case.get("q", "f32") != "f32":
        o["refine"] = case.get("refine", 0)
        o["msg_bf16"] = 1 if case.get("msg_bf16") else 0
    if case.get("stages", 1) > 1:
        o["stages"] = case["stages"]
    if case.get("krr"):
        o["task"] = gabp.TASK_KRR
    if case.get("tau"):
        o["sparse_tau"] = case["tau"]
    return o


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, kind=kind)
    if kind == "batch":
        s["problems"] = [workloads.Problem(*p) for p in _problems(case, seed)]
        return s
    if kind == "serve":
        s["problems"] = [(X.cpu().numpy(), y.cpu().numpy(), g, C) for X, y, g, C in _problems(case, seed)]
        return s
    X, y, Xt, gamma = _inputs(case, seed)
    if case.get("host"):
        dt = np.float64 if case.get("fp64") else np.float32
        X, y = X.cpu().numpy().astype(dt), y.cpu().numpy()
        Xt = Xt.cpu().numpy().astype(dt) if Xt is not None else None
    elif case.get("fp64"):
        X, Xt = X.double(), Xt.double() if Xt is not None else None
    s.update(X=X, y=y, Xt=Xt, gamma=gamma)
    if kind == "retrain":
        s["svm"] = gabp.GabpSVM(X, y, gamma, case["C"], **_options(case))
    elif kind == "decide":
        s["svm"] = gabp.GabpSVM(X, y, gamma, case["C"])
        s["svm"].solve(40, 1e-6)
    elif kind == "decide_noalloc":
        # weights as a solver leaves them: positive, of the size of 1 / (row sum)
        s["alpha"] = _weights(case, seed)
        s["out"] = torch.empty(case["t"], device="cuda")
    return s


def _weights(case, seed):
    g = _gen(seed, 99)
    return (0.5 + torch.rand(case["n"], generator=g, device="cuda")) / case["n"]


# ------------------------------------------------------------------- one pass
def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "train":
        svm = gabp.GabpSVM(s["X"], s["y"], s["gamma"], case["C"], **_options(case))
        alpha, _, _ = svm.solve(case["iters"], case["tol"])
        out = {"alpha": alpha, "mean": svm.mean(), "decision": svm.decision(s["Xt"])}
        svm.close()
        return out
    if kind == "retrain":
        svm = s["svm"]
        svm.refit(s["X"], s["y"], s["gamma"], case["C"])
        alpha, _, _ = svm.solve(case["iters"], case["tol"])
        return {"alpha": alpha, "mean": svm.mean()}
    if kind == "batch":
        alphas, results, _ = gabp.batch_solve(s["problems"], case["iters"], case["tol"], means=True,
                                              **_options(case))
        return {"alpha": torch.cat(alphas), "mean": torch.cat([r["mu"] for r in results])}
    if kind == "serve":
        srv = gabp.Server(iters=case["iters"], tol=case["tol"], max_members=32, chunk=4, **_options(case))
        tickets = [srv.submit(X, y, g, C) for X, y, g, C in s["problems"]]
        left = len(tickets)
        got = {}
        while left:
            srv.step()
            for t in srv.completed():
                got[t] = srv.poll(t)[0]
                left -= 1
        srv.close()
        return [got[t] for t in tickets]
    if kind == "decide":
        return s["svm"].decision(s["Xt"])
    gabp.decision_noalloc(s["X"], s["y"], s["alpha"], s["Xt"], s["gamma"], 1.0 / case["n"], s["out"])
    return s["out"]


# --------------------------------------------------------- what a pass needs
def work(case):
    """Bytes: inputs read once and outputs written once.  Flops: the Gram products of the upper triangle (2 m a
    pair), one multiply-add for each directed edge and round, and 2 m + 2 for each decision pair."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        sizes = _grid_sizes(case)
        grid = len(GRID_C) * len(GRID_GAMMA) if kind == "batch" else 1
        return {"bytes": sum(4 * (n * m + n) + grid * 8 * n for n, m in sizes),
                "flops": sum(float(n) * n * (m + grid * 2 * TO_TOLERANCE_ROUNDS) for n, m in sizes)}
    n, m, t = case["n"], case["m"], case.get("t", 0)
    el = 8 if case.get("fp64") else 4
    if kind in ("decide", "decide_noalloc"):
        return {"bytes": 4 * (n * m + 2 * n + t * m + t), "flops": float(n) * t * (2 * m + 2)}
    rounds = case["iters"] if case["tol"] <= 0 else TO_TOLERANCE_ROUNDS
    return {"bytes": el * (n * m + t * m) + 4 * (3 * n + t),
            "flops": float(n) * n * (m + 2 * rounds) + float(n) * t * (2 * m + 2)}


# ------------------------------------------------------------------ in 64 bits
def _kernel(A, B, gamma):
    d2 = (A * A).sum(dim=1)[:, None] + (B * B).sum(dim=1)[None, :] - 2.0 * (A @ B.T)
    return d2.clamp_min_(0.0).mul_(-gamma).exp_()


def _solve64(X, y, gamma, C, krr=False, tau=0.0):
    """Q^-1 b in FP64 by conjugate gradients: Q_ij = y_i y_j (K + 1/n^2), Q_ii = max(1 + 1/n^2 + 1/C, 1.1 sum
    |Q_ij|) (SVM, b = 1); K, max(1 + C, ...) and b = y (ridge C); off-diagonal 128 x 128 tiles whose largest
    entry is at most tau count as 0 (the diagonal is that of the whole matrix)."""
    X, y = X.double(), y.double()
    n = X.shape[0]
    lam2 = 0.0 if krr else 1.0 / n / n
    b = y if krr else torch.ones_like(y)
    s = torch.ones_like(y) if krr else y
    Q = torch.empty(n, n, dtype=torch.float64, device="cuda")
    R = torch.empty(n, dtype=torch.float64, device="cuda")
    step = 128 * max(1, min(16, (1 << 28) // (n * 128)))
    for i in range(0, n, step):
        e = min(n, i + step)
        K = _kernel(X[i:e], X, gamma).add_(lam2)
        r = torch.arange(i, e, device="cuda")
        K[r - i, r] = 0.0
        R[i:e] = K.sum(dim=1)
        if tau:
            nt = (n + 127) // 128
            pad = torch.zeros(((e - i + 127) // 128) * 128, nt * 128, dtype=torch.float64, device="cuda")
            pad[:e - i, :n] = K
            t = pad.view(-1, 128, nt, 128)
            keep = t.amax(dim=(1, 3)) > tau
            keep[torch.arange(keep.shape[0], device="cuda"), i // 128 + torch.arange(keep.shape[0], device="cuda")] = True
            K = (t * keep[:, None, :, None]).reshape(pad.shape)[:e - i, :n]
        Q[i:e] = K.mul_(s[i:e, None]).mul_(s[None, :])
        del K
    D = torch.maximum(1.0 + lam2 + (C if krr else 1.0 / C) + torch.zeros_like(R), 1.1 * R)
    x = b / D
    r = b - (Q @ x + D * x)
    z = r / D
    p, rz = z.clone(), r @ z
    stop = 1e-14 * float(b.norm())
    for k in range(400):
        Ap = Q @ p + D * p
        a = rz / (p @ Ap)
        x += a * p
        r -= a * Ap
        if k % 8 == 7 and float(r.norm()) < stop:
            break
        z = r / D
        rz, old = r @ z, rz
        p = z + (rz / old) * p
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        mu = [(_solve64(X, y, g, C), C) for X, y, g, C in _problems(case, seed)]
        if kind == "serve":
            return [m.clamp(0.0, C) for m, C in mu]
        return {"alpha": torch.cat([m.clamp(0.0, C) for m, C in mu]), "mean": torch.cat([m for m, _ in mu])}
    X, y, Xt, gamma = _inputs(case, seed)
    if kind == "decide_noalloc":
        w = _weights(case, seed).double() * y.double()
        return (_kernel(Xt.double(), X.double(), gamma) + 1.0 / case["n"] ** 2) @ w
    mu = _solve64(X, y, gamma, case["C"], bool(case.get("krr")), case.get("tau", 0.0))
    alpha = mu if case.get("krr") else mu.clamp(0.0, case["C"])
    if Xt is not None:
        w, f = alpha * y.double(), []
        for i in range(0, Xt.shape[0], 2000):
            f.append((_kernel(Xt[i:i + 2000].double(), X.double(), gamma) + 1.0 / case["n"] ** 2) @ w)
        f = torch.cat(f)
    if kind == "decide":
        return f
    return {"alpha": alpha, "mean": mu, "decision": f} if kind == "train" else {"alpha": alpha, "mean": mu}
