"""What the speed of this library is measured on.

Twelve cases of the work its users have it do, through the entry points of
``paper_2106_09382_gb300.concord``, and ``draw`` for more of the same ranges.
The kinds, and what each stands for in use:

    solve      X (device, n x p) -> Omega: ``State.solve_device``, the library's
               main call, from tables of a hundred variables (latency) to
               genome-sized ones (p = 20000), in both precisions
    host       the same from and to numpy arrays: ``State.solve_host``
    path       a warm-started lambda path on a Gram: ``State.set_S``, ``path``
    batch      stability selection: many row subsets of one table, a lambda
               path on each in one launch: ``Batch.gram``, ``Batch.path``
    joint      two related populations: ``Joint.set_S``, ``Joint.run``
    hypergrad  one step of tuning lambda on held-out rows, with the gradient
               of the data: ``solve_device``, ``heldout``, ``adjoint``,
               ``adjoint_data``
    gram       S = Z^T Z / n alone: ``concord_gram`` in its four arithmetics

Data: n rows of N(0, Omega0^-1) for a sparse diagonally dominant Omega0 of the
designs of ``synth`` (AR(1) with extra edges, power law, random graph,
diagonal blocks), each column with a scale and an offset of its own, as tables
come.  Mixed-precision results are taken in FP32 and FP64 ones in FP64.
"""
import math

import numpy as np
import torch

from paper_2106_09382_gb300 import concord as C
from paper_2106_09382_gb300 import synth

PRECISION = {"fp64": C.FP64, "mixed": C.MIXED}
GRAM = {"fp64": C.GRAM_FP64, "fp32": C.GRAM_FP32, "tf32x3": C.GRAM_TF32X3,
        "bf16x3": C.GRAM_BF16X3}
PREP = {"none": C.PREP_NONE, "center": C.PREP_CENTER, "standardize": C.PREP_STANDARDIZE}
TORCH = {"f32": torch.float32, "f64": torch.float64}


def listed():
    return [
        # the smallest whole solve: a hundred variables, a plain FP64 answer
        dict(name="solve_fp64_p100", kind="solve", precision="fp64", graph="random", p=100, n=200,
             data="f64", lam=0.3, tol=1e-6),
        # an ordinary table with FP32 data
        dict(name="solve_mixed_p1000", kind="solve", precision="mixed", graph="ar1", p=1000, n=500,
             data="f32", lam=0.25, tol=1e-5),
        # the benchmark workload: p = 5000, n = 2000, FP64 data
        dict(name="solve_mixed_p5000", kind="solve", precision="mixed", graph="ar1", p=5000, n=2000,
             data="f64", lam=0.2, tol=1e-5),
        # its FP64 counterpart at the odd size (a bye vertex in every colour)
        dict(name="solve_fp64_p4999", kind="solve", precision="fp64", graph="ar1", p=4999, n=2000,
             data="f64", lam=0.2, tol=1e-5),
        # the large sparse solve, FP32 data
        dict(name="solve_mixed_p20000", kind="solve", precision="mixed", graph="power", p=20000,
             n=5000, data="f32", lam=0.15, tol=1e-5),
        # a numpy caller: host X in, dense host Omega out, FP64
        dict(name="host_fp64_p999", kind="host", precision="fp64", graph="ar1", p=999, n=700,
             data="f64", lam=0.25, tol=1e-6),
        # a regularisation path of 32 lambdas, from no edge to a third of all pairs
        dict(name="path_mixed_p1000", kind="path", precision="mixed", graph="power", p=1000, n=800,
             lambdas=32, lam_last=0.05, tol=1e-5),
        # stability selection: 24 uneven subsamples, 8 lambdas
        dict(name="batch_mixed_p500", kind="batch", precision="mixed", graph="power", p=500, n=800,
             problems=24, lambdas=8, lam_last=0.3, tol=1e-5),
        # two populations, 500 rows each
        dict(name="joint_mixed_p1000", kind="joint", precision="mixed", graph="ar1", p=1000, n=500,
             lam=0.2, lam2=0.05, tol=1e-5),
        # tuning lambda: the differentiable-solve workload
        dict(name="hypergrad_mixed_p2000", kind="hypergrad", precision="mixed", graph="blocks",
             p=2000, n=1000, n_val=500, data="f32", lam_frac=0.3, tol=1e-5),
        # an FP64 Gram of ragged sizes
        dict(name="gram_fp64_p2049", kind="gram", mode="fp64", prep="center", graph="random",
             p=2049, n=1203, data="f32"),
        # a large tensor-core Gram
        dict(name="gram_tf32x3_p12000", kind="gram", mode="tf32x3", prep="standardize",
             graph="power", p=12000, n=5000, data="f32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _noise(p, n):
    """Twice the largest sample correlation of independent columns: the scale of
    the lambdas that separate edges from noise."""
    return 2.0 * math.sqrt(2.0 * math.log(p) / n)


def draw(rng):
    kind = rng.choice(["solve"] * 5 + ["host", "path", "batch", "joint", "hypergrad"] + ["gram"] * 2)
    graph = rng.choice(["ar1", "power", "random"])
    if kind == "solve":
        precision = rng.choice(["fp64", "mixed", "mixed"])
        p = _log(rng, 60, 5000 if precision == "fp64" else 12000)
        n = max(50, _log(rng, p // 4 + 40, min(2 * p + 100, 3000)))
        c = dict(kind=kind, precision=precision, graph=graph, p=p, n=n,
                 data=rng.choice(["f32", "f64"]), tol=rng.choice([1e-5, 1e-6]))
        c["lam"] = round(_noise(p, n) * rng.uniform(0.95, 1.3), 4)
        return c
    if kind == "host":
        p = _log(rng, 60, 1500)
        n = _log(rng, p // 2 + 40, 2 * p + 100)
        return dict(kind=kind, precision="fp64", graph=graph, p=p, n=n, data="f64", tol=1e-6,
                    lam=round(_noise(p, n) * rng.uniform(0.95, 1.3), 4))
    if kind == "path":
        p = _log(rng, 100, 1000)
        return dict(kind=kind, precision="mixed", graph=graph, p=p, n=_log(rng, 0.8 * p, 2 * p),
                    lambdas=rng.randint(8, 32), lam_last=round(rng.uniform(0.08, 0.4), 3), tol=1e-5)
    if kind == "batch":
        p = _log(rng, 60, 500)
        return dict(kind=kind, precision="mixed", graph=graph, p=p, n=rng.randint(500, 1000),
                    problems=rng.randint(4, 24), lambdas=rng.randint(3, 8),
                    lam_last=round(rng.uniform(0.35, 0.6), 3), tol=1e-5)
    if kind == "joint":
        p = _log(rng, 60, 1000)
        n = _log(rng, p // 2 + 40, 2 * p)
        return dict(kind=kind, precision=rng.choice(["fp64", "mixed"]), graph="ar1", p=p, n=n,
                    lam=round(0.5 * _noise(p, n) * rng.uniform(0.9, 1.3), 4),
                    lam2=round(rng.uniform(0.01, 0.1), 3), tol=1e-5)
    if kind == "hypergrad":
        p = _log(rng, 100, 2000)
        n = _log(rng, p // 2 + 40, p + 40)
        return dict(kind=kind, precision=rng.choice(["fp64", "mixed"]),
                    graph=rng.choice(["blocks", "ar1"]), p=p, n=n, n_val=n // 2,
                    data=rng.choice(["f32", "f64"]), lam_frac=round(rng.uniform(0.3, 0.5), 3),
                    tol=1e-5)
    mode = rng.choice(["fp64", "fp64", "fp32", "tf32x3", "bf16x3"])
    p = _log(rng, 33, 5000 if mode == "fp64" else 8000)
    return dict(kind=kind, mode=mode, prep=rng.choice(["none", "center", "standardize"]),
                graph=graph, p=p, n=_log(rng, 20, 5000), data=rng.choice(["f32", "f64"]))


# ------------------------------------------------------------------ inputs
def _precision_matrix(graph, p, seed):
    """Edges (i < j), values and diagonal of a diagonally dominant Omega0."""
    rng = np.random.default_rng(seed)
    if graph == "power":
        return synth.power_law(p, 2, 0.2, 0.5, 0.5, seed)
    if graph == "ar1":
        i, j, v = np.arange(p - 1), np.arange(1, p), np.full(p - 1, -2.0 / 3.0)
        diag = np.full(p, 5.0 / 3.0)
        diag[[0, -1]] = 4.0 / 3.0
        k = round(0.01 * (p - 1))
        m = 8 * k + 8
    else:
        i, j, v = np.zeros(0, int), np.zeros(0, int), np.zeros(0)
        diag = np.full(p, 0.5)
        # two or three edges per vertex; ten within a block of a hundred
        k = p * (5 if graph == "blocks" else 3) if p > 60 else p
        m = 2 * k
    a = rng.integers(0, p, m)
    if graph == "blocks":
        size = max(2, p // 20)
        b = np.minimum(a // size * size + rng.integers(0, size, m), p - 1)
    else:
        b = rng.integers(0, p, m)
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    far = hi - lo > (1 if graph == "ar1" else 0)
    at = np.unique(lo[far] * p + hi[far])
    at = np.sort(rng.permutation(at)[:k])
    e = rng.uniform(0.3, 0.6, at.size) * np.where(rng.random(at.size) < 0.5, -1.0, 1.0)
    np.add.at(diag, at // p, np.abs(e))
    np.add.at(diag, at % p, np.abs(e))
    if graph != "ar1":
        return at // p, at % p, e, diag
    return np.concatenate([i, at // p]), np.concatenate([j, at % p]), np.concatenate([v, e]), diag


def _table(Om0, n, seed, dtype):
    """n rows of N(0, Omega0^-1) on the GPU, columns with scales and offsets."""
    X = synth.sample_sparse(*Om0, n, seed)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 17)
    p = X.shape[1]
    X *= torch.exp(0.5 * torch.randn(p, generator=g, dtype=torch.float64, device="cuda"))
    X += torch.randn(p, generator=g, dtype=torch.float64, device="cuda")
    return X.to(dtype).contiguous()


def _standardized(X, prep="standardize"):
    Z = X.double()
    if prep != "none":
        Z = Z - Z.mean(0)
    if prep == "standardize":
        Z = Z / Z.square().mean(0).sqrt()
    return Z


def _gram(X, prep="standardize"):
    Z = _standardized(X, prep)
    S = Z.t() @ Z / Z.shape[0]
    return (S + S.t()) / 2


def _lambda_max(S):
    r = S.diagonal().rsqrt()
    return float(((S - torch.diag(S.diagonal())).abs() * (r[:, None] + r[None, :])).max())


def _inputs(case, seed):
    """The arrays of a case, with no handle of the library."""
    p, n, kind = case["p"], case["n"], case["kind"]
    Om0 = _precision_matrix(case["graph"], p, seed)
    if kind in ("solve", "host", "gram"):
        return {"X": _table(Om0, n, seed, TORCH[case["data"]])}
    if kind == "path":
        S = _gram(_table(Om0, n, seed, torch.float64))
        lam = _lambda_max(S) * np.geomspace(1.0, case["lam_last"], case["lambdas"])
        return {"S": S, "lam": lam}
    if kind == "batch":
        X = _table(Om0, n, seed, torch.float64)
        rng = np.random.default_rng(seed + 5)
        sizes = rng.integers(n // 4, n + 1, case["problems"])
        rows = [np.sort(rng.choice(n, int(m), replace=False)).astype(np.int32) for m in sizes]
        lam = _lambda_max(_gram(X)) * np.geomspace(1.0, case["lam_last"], case["lambdas"])
        return {"X": X, "rows": [torch.as_tensor(r, device="cuda") for r in rows], "lam": lam}
    if kind == "joint":
        # a second population: the same band and other extra edges
        Om1 = _precision_matrix(case["graph"], p, seed + 1)
        return {"S": [_gram(_table(Om0, n, seed, torch.float64)),
                      _gram(_table(Om1, n, seed + 1, torch.float64))]}
    X = _table(Om0, n + case["n_val"], seed, TORCH[case["data"]])
    X, Xv = X[:n].contiguous(), X[n:].contiguous()
    return {"X": X, "Sv": _gram(Xv), "lam": case["lam_frac"] * _lambda_max(_gram(X))}


def prepare(case, seed):
    s = _inputs(case, seed)
    p, n, kind = case["p"], case["n"], case["kind"]
    s["case"], s["stream"] = case, torch.cuda.Stream()
    if kind != "gram":
        precision = PRECISION[case["precision"]]
        s["out"] = torch.float64 if case["precision"] == "fp64" else torch.float32
        if kind == "joint":
            s["handle"] = C.Joint(p, precision)
        elif kind == "batch":
            s["handle"] = C.Batch([p] * case["problems"], precision, n_cap=n)
        else:
            s["handle"] = C.State(p, precision, n_cap=0 if kind == "path" else n)
        s["handle"].set_stream(s["stream"])
    if kind in ("solve", "joint"):
        s["Omega"] = [torch.empty((p, p), dtype=s["out"], device="cuda")
                      for _ in range(2 if kind == "joint" else 1)]
    elif kind == "path":
        s["Omega"] = torch.empty((case["lambdas"], p, p), dtype=s["out"], device="cuda")
    elif kind == "host":
        s["X"] = s["X"].cpu().numpy()
        s["Omega"] = np.empty((p, p))
    torch.cuda.synchronize()
    return s


def run(s):
    with torch.cuda.stream(s["stream"]):
        return _RUN[s["case"]["kind"]](s, s["case"])


def _run_solve(s, c):
    s["handle"].solve_device(s["X"], c["lam"], tol=c["tol"], Omega_out=s["Omega"][0])
    return {"Omega": s["Omega"][0]}


def _run_host(s, c):
    s["handle"].solve_host(s["X"], c["lam"], tol=c["tol"], Omega_out=s["Omega"])
    return {"Omega": s["Omega"]}


def _run_path(s, c):
    s["handle"].set_S(s["S"])
    s["handle"].path(s["lam"], tol=c["tol"], omega_out=s["Omega"])
    return {"Omega": s["Omega"]}


def _run_batch(s, c):
    bt = s["handle"]
    for b, rows in enumerate(s["rows"]):
        bt.gram(b, s["X"], rows)
    bt.path(s["lam"], tol=c["tol"])
    return {"Omega": [bt.get_omega(b, s["out"]) for b in range(len(bt))]}


def _run_joint(s, c):
    jt = s["handle"]
    for m in (0, 1):
        jt.set_S(m, s["S"][m])
    jt.run(c["lam"], c["lam2"], tol=c["tol"])
    return {"Omega": [jt.get_omega(m, s["Omega"][m]) for m in (0, 1)]}


def _run_hypergrad(s, c):
    st = s["handle"]
    st.solve_device(s["X"], s["lam"], tol=c["tol"])
    loss = st.heldout(s["Sv"])
    info = st.adjoint(None)
    return {"Omega": st.get_omega(s["out"]), "loss": loss, "dlambda": info.dlambda,
            "dX": st.adjoint_data(s["X"])}


def _run_gram(s, c):
    return {"S": C.concord_gram(s["X"], PREP[c["prep"]], GRAM[c["mode"]])}


_RUN = {"solve": _run_solve, "host": _run_host, "path": _run_path, "batch": _run_batch,
        "joint": _run_joint, "hypergrad": _run_hypergrad, "gram": _run_gram}


def work(case):
    """Inputs in, results out, and the products that no method does without: the
    Gram's where it starts from data."""
    p, n, kind = case["p"], case["n"], case["kind"]
    x = n * p * (4 if case.get("data") == "f32" else 8)
    om = p * p * (8 if case.get("precision") == "fp64" else 4)
    gram = float(n) * p * (p + 1)
    if kind in ("solve", "host"):
        return {"bytes": x + om, "flops": gram}
    if kind == "path":
        return {"bytes": p * p * 8 + case["lambdas"] * om, "flops": 2 * case["lambdas"] * p * p}
    if kind == "batch":
        m = case["problems"]
        return {"bytes": x + m * om, "flops": 0.625 * m * gram}  # subsets hold 5/8 of the rows
    if kind == "joint":
        return {"bytes": 2 * (p * p * 8 + om), "flops": 4 * p * p}
    if kind == "hypergrad":  # X read and dX written; the held-out Gram read
        return {"bytes": 2 * x + p * p * 8 + om, "flops": gram}
    return {"bytes": x + p * p * (8 if case["mode"] == "fp64" else 4), "flops": gram}


# ------------------------------------------------- the same in plain FP64 torch
def _colours(p):
    """The circle method: (pairs, 2) index tensors, one per colour step."""
    pe = p + p % 2
    ring = np.arange(1, pe)
    for c in range(pe - 1):
        r = np.roll(ring, c)
        row = np.concatenate([[0], r])
        a, b = row[: pe // 2], row[::-1][: pe // 2]
        keep = (a < p) & (b < p)
        yield torch.as_tensor(np.stack([a[keep], b[keep]]), device="cuda")


def _soft(x, t):
    return torch.sign(x) * (x.abs() - t).clamp_min(0)


def _kkt(S, Om, lam):
    W = Om @ S
    G = W + W.t()
    r = torch.where(Om != 0, (G + lam * torch.sign(Om)).abs(), (G.abs() - lam).clamp_min(0))
    r.fill_diagonal_(0)
    return max(float(r.max()), float((W.diagonal() - 1 / Om.diagonal()).abs().max()))


def _descend(S, lam, tol, colours):
    """Coordinate descent of Eq. 1 from the identity in colour order until the
    subgradient conditions hold to tol."""
    p = S.shape[0]
    d = S.diagonal().clone()
    Om, W = torch.eye(p, dtype=S.dtype, device=S.device), S.clone()
    for _ in range(1000):
        for ij in colours:
            i, j = ij
            w, s = Om[i, j], d[i] + d[j]
            new = _soft(s * w - W[i, j] - W[j, i], lam) / s
            k = torch.nonzero(new != w).flatten()
            if k.numel():
                i, j, dw = i[k], j[k], (new - w)[k]
                Om[i, j] += dw
                Om[j, i] += dw
                W[i] += dw[:, None] * S[j]
                W[j] += dw[:, None] * S[i]
        w = Om.diagonal().clone()
        b = W.diagonal() - w * d
        new = (-b + (b * b + 4 * d).sqrt()) / (2 * d)
        Om.diagonal().copy_(new)
        W += (new - w)[:, None] * S
        if _kkt(S, Om, lam) <= tol:
            break
    return Om


def _descend_joint(S, lam, lam2, tol, colours):
    p = S[0].shape[0]
    d = [s.diagonal().clone() for s in S]
    Om = [torch.eye(p, dtype=S[0].dtype, device="cuda") for _ in S]
    W = [s.clone() for s in S]

    def split(x, y, fused):
        """x, y for either sign of the fusion term, else the fused value."""
        up, down = x[0] > y[0], x[1] < y[1]
        return (torch.where(up, x[0], torch.where(down, x[1], fused)),
                torch.where(up, y[0], torch.where(down, y[1], fused)))

    def root(b, s):
        return (-b + (b * b + 4 * s).sqrt()) / (2 * s)

    for _ in range(1000):
        for ij in colours:
            i, j = ij
            w = [o[i, j] for o in Om]
            c = [e[i] + e[j] for e in d]
            g = [W[m][i, j] + W[m][j, i] - c[m] * w[m] for m in (0, 1)]
            new = split([_soft(-(g[0] + t * lam2), lam) / c[0] for t in (1, -1)],
                        [_soft(-(g[1] - t * lam2), lam) / c[1] for t in (1, -1)],
                        _soft(-(g[0] + g[1]), 2 * lam) / (c[0] + c[1]))
            for m in (0, 1):
                k = torch.nonzero(new[m] != w[m]).flatten()
                if k.numel():
                    a, b, dw = i[k], j[k], (new[m] - w[m])[k]
                    Om[m][a, b] += dw
                    Om[m][b, a] += dw
                    W[m][a] += dw[:, None] * S[m][b]
                    W[m][b] += dw[:, None] * S[m][a]
        w = [o.diagonal().clone() for o in Om]
        b = [W[m].diagonal() - w[m] * d[m] for m in (0, 1)]
        s, h = d[0] + d[1], b[0] + b[1]
        new = split([root(b[0] + t * lam2, d[0]) for t in (1, -1)],
                    [root(b[1] - t * lam2, d[1]) for t in (1, -1)],
                    (-h + (h * h + 8 * s).sqrt()) / (2 * s))
        for m in (0, 1):
            Om[m].diagonal().copy_(new[m])
            W[m] += (new[m] - w[m])[:, None] * S[m]
        G = [Om[m] @ S[m] for m in (0, 1)]
        G = [x + x.t() for x in G]
        sub = [G[m] + lam * torch.sign(Om[m]) for m in (0, 1)]
        zero = [o == 0 for o in Om]
        same, low = Om[0] == Om[1], lam * zero[0].double()
        u = torch.where(same, ((sub[1] - sub[0]) / 2).clamp(-lam2, lam2),
                        lam2 * torch.sign(Om[0] - Om[1]))
        r = torch.maximum(((sub[0] + u).abs() - low).clamp_min(0),
                          ((sub[1] - u).abs() - lam * zero[1].double()).clamp_min(0))
        r.fill_diagonal_(0)
        e = [G[m].diagonal() / 2 - 1 / Om[m].diagonal() for m in (0, 1)]
        ud = torch.where(same.diagonal(), ((e[1] - e[0]) / 2).clamp(-lam2, lam2),
                         lam2 * torch.sign(Om[0].diagonal() - Om[1].diagonal()))
        far = torch.maximum((e[0] + ud).abs(), (e[1] - ud).abs())
        if max(float(r.max()), float(far.max())) <= tol:
            break
    return Om


def _adjoint(S, Om, Sv, tol=1e-12):
    """Held-out loss, dL/dlambda and dL/dS on the active set of Om, by conjugate
    gradients on masked dense products."""
    on = Om != 0
    Wv = Om @ Sv
    loss = float(-Om.diagonal().log().sum() + 0.5 * (Wv * Om).sum())
    b = (Wv + Wv.t()) * on
    b.diagonal().copy_(Wv.diagonal() - 1 / Om.diagonal())
    diag2 = 1 / Om.diagonal().square()

    def hess(V):
        VS = V @ S
        R = (VS + VS.t()) * on
        R.diagonal().copy_(VS.diagonal() + V.diagonal() * diag2)
        return R

    def dot(A, B):  # over the diagonal and the upper pairs
        return float(((A * B).sum() + (A * B).diagonal().sum()) / 2)

    s = S.diagonal()
    pre = s[:, None] + s[None, :]
    pre.diagonal().copy_(s + diag2)
    a, r = torch.zeros_like(S), b.clone()
    z = r / pre
    q, rz, top = z.clone(), dot(r, z), dot(b, b)
    for _ in range(500):
        hq = hess(q)
        t = rz / dot(q, hq)
        a += t * q
        r -= t * hq
        if dot(r, r) <= tol * tol * top:
            break
        z = r / pre
        rz, old = dot(r, z), rz
        q = z + rz / old * q
    dlam = -float((a * torch.sign(Om)).triu(1).sum())
    return loss, dlam, -(Om @ a)


def exact(case, seed):
    """What run() returns, in FP64 by plain torch; None where that takes long."""
    p, kind = case["p"], case["kind"]
    if kind in ("path", "batch") or (p > 5000 and kind != "gram"):
        return None
    s = _inputs(case, seed)
    if kind == "gram":
        return {"S": _gram(s["X"], case["prep"])}
    colours = list(_colours(p))
    if kind == "joint":
        return {"Omega": _descend_joint(s["S"], case["lam"], case["lam2"], case["tol"], colours)}
    S = _gram(s["X"])
    if kind in ("solve", "host"):
        return {"Omega": _descend(S, case["lam"], case["tol"], colours)}
    Om = _descend(S, s["lam"], case["tol"], colours)
    loss, dlam, dS = _adjoint(S, Om, s["Sv"])
    X = s["X"].double().requires_grad_()
    Z = _standardized(X)
    (Z.t() @ Z / X.shape[0]).backward(dS)
    return {"Omega": Om, "loss": loss, "dlambda": dlam, "dX": X.grad}
