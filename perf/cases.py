"""The work a user of this library has it do, as measurable cases.

Four kinds of call, through the package's public functions, on device-resident
inputs of the shapes the package's workloads have (``synth``):

* ``online``   a trained model held on the device (``Model``) scores a few or
  many new rows: real-valued rows in mixed precision, binary rows in FP64;
* ``heldout``  ``svm_decision`` straight from the training rows and multipliers
  (the call after a training: score the held-out set, or single requests);
* ``train``    ``svm_train`` to the KKT tolerance, FP64 and mixed precision, with
  and without the shrinking policies of Table 3;
* ``batch``    ``svm_train_batch``: one-vs-one pairs or a C x gamma grid, with the
  launch shape a user keeps from one ``svm_batch_autotune``.

Inputs are drawn on the device from the seed alone. The multipliers of the
decision cases are drawn like those of trained models (a share of the rows are
support vectors, most of these at the bound C), so no training runs before a
decision is timed. The training server is left out: its engine kernel stays on
the device for half a second after the last job, which is what a device-wide
wait would then measure; it runs the kernel of the batch cases.
"""
from __future__ import annotations

import math

import torch

import paper_1406_5161_gb300 as svm

TAU = 1e-3
PRECISION = {"fp64": svm.SVM_FP64, "mixed": svm.SVM_MIXED_BF16}


# ------------------------------------------------------------------- cases
def listed():
    return [
        # one request scored in FP64: 8 rows against 20,000 support vectors
        {"name": "score_8_fp64", "kind": "heldout", "data": "covtype", "n": 20000, "m": 8,
         "sv": 1.0, "precision": "fp64"},
        # a micro-batch of requests, mixed precision, the benchmark model's 48,868 vectors
        {"name": "online_300_mixed", "kind": "online", "data": "covtype", "n": 48868, "m": 300,
         "sv": 1.0, "precision": "mixed"},
        # the benchmark's second half: 10,000 held-out rows after the 581,012-row training
        {"name": "heldout_covtype_fp64", "kind": "heldout", "data": "covtype", "n": 581012,
         "m": 10000, "sv": 0.0841, "precision": "fp64"},
        # held-out rows of the a9a-shaped problem: binary rows, distance tables
        {"name": "heldout_onehot_fp64", "kind": "heldout", "data": "onehot", "n": 32561,
         "m": 10000, "sv": 0.36, "precision": "fp64"},
        # bulk scoring, the tensor-core contraction at its benchmark size
        {"name": "bulk_mixed", "kind": "online", "data": "covtype", "n": 100000, "m": 100000,
         "sv": 1.0, "precision": "mixed"},
        # a small dense problem, plain SMO in FP64
        {"name": "train_gauss_fp64", "kind": "train", "data": "gauss", "n": 2000, "d": 20,
         "C": 1.0, "gamma": 0.05, "precision": "fp64", "policy": "Original"},
        # the a9a-shaped problem under the aggressive policy
        {"name": "train_onehot_fp64", "kind": "train", "data": "onehot", "n": 32561,
         "C": 1.0, "gamma": 0.05, "precision": "fp64", "policy": "Multi5pc"},
        # covtype-shaped rows: the largest problem here (streamed, re-layout, reconstruction)
        {"name": "train_covtype_fp64", "kind": "train", "data": "covtype", "n": 120000,
         "C": 4.0, "gamma": 0.1, "precision": "fp64", "policy": "Multi500"},
        # the same kind of problem in the precision pattern, a ragged size
        {"name": "train_covtype_mixed", "kind": "train", "data": "covtype", "n": 47001,
         "C": 4.0, "gamma": 0.1, "precision": "mixed", "policy": "Multi500"},
        # dense L2-normalised rows of a served job, precision pattern
        {"name": "train_dense_mixed", "kind": "train", "data": "unit", "n": 12000, "d": 100,
         "C": 5.0, "gamma": 0.01, "precision": "mixed", "policy": "Multi5pc"},
        # one-vs-one pairs of ten classes, 256 dense columns, two values of C
        {"name": "batch_ovo_mixed", "kind": "batch", "data": "ovo", "n": 20000, "d": 256,
         "jobs": 90, "precision": "mixed", "cluster_size": 2, "lanes_per_row": 16},
        # a C x gamma grid over one small dense problem in FP64
        {"name": "batch_grid_fp64", "kind": "batch", "data": "gauss", "n": 1500, "d": 20,
         "jobs": 45, "precision": "fp64", "cluster_size": 4, "lanes_per_row": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: kind, shape, precision and options over the ranges above."""
    kind = rng.choice(["online", "online", "heldout", "heldout", "train", "train", "train", "batch"])
    precision = rng.choice(["fp64", "mixed"])
    if kind == "online":
        # one row to a bulk job of at most 4e8 pairs
        data = "onehot" if precision == "fp64" else rng.choice(["covtype", "covtype", "gauss", "sparse"])
        n = _log(rng, 1000, 20000 if data == "onehot" else 100000)
        c = {"kind": kind, "data": data, "n": n, "m": _log(rng, 1, min(20000 if data == "sparse" else 100000, 400000000 // n)),
             "sv": 1.0, "precision": precision}
    elif kind == "heldout":
        data = rng.choice(["covtype", "onehot", "gauss"])
        c = {"kind": kind, "data": data, "n": _log(rng, 2000, 581012 if data == "covtype" else 32561),
             "m": _log(rng, 1, 10000), "sv": round(rng.uniform(0.05, 0.4), 3), "precision": precision}
        c["sv"] = min(c["sv"], round(48868 / c["n"], 4)) if data == "covtype" else c["sv"]
    elif kind == "train":
        data = rng.choice(["covtype", "onehot", "gauss", "unit", "sparse"])
        top = {"covtype": 60000, "onehot": 32561, "gauss": 6000, "unit": 12000, "sparse": 20000}[data]
        c = {"kind": kind, "data": data, "n": _log(rng, 500, top), "precision": precision,
             "policy": rng.choice(["Original", "Multi500", "Multi5pc", "Multi10pc", "Single5pc"]),
             "C": round(math.exp(rng.uniform(math.log(0.5), math.log(8.0))), 2),
             "gamma": {"covtype": 0.1, "onehot": 0.05, "gauss": 0.05}.get(data, 0.0)}
    else:
        data = rng.choice(["ovo", "gauss"])
        c = {"kind": kind, "data": data, "n": _log(rng, 3000, 20000) if data == "ovo" else _log(rng, 300, 1500),
             "jobs": rng.randint(4, 90 if data == "ovo" else 45), "precision": precision,
             "cluster_size": rng.choice([2, 4, 8]),
             "lanes_per_row": 16 if (data, precision) == ("ovo", "mixed") else rng.choice([1, 2, 4])}
        if data == "ovo" and precision == "fp64":
            c["n"], c["jobs"] = min(c["n"], 6000), min(c["jobs"], 45)
    if c["data"] == "gauss":
        c["d"] = rng.randint(5, 64)
    elif c["data"] == "unit":
        c["d"] = _log(rng, 20, 300)
    elif c["data"] == "sparse":
        c["d"] = _log(rng, 200, 2000)
    elif c["data"] == "ovo":
        c["d"] = rng.choice([64, 96, 128, 256]) if precision == "mixed" else rng.randint(16, 64)
    if c.get("gamma") == 0.0:
        c["gamma"] = round(1.0 / c["d"], 6)
    return c


# ------------------------------------------------------------------ inputs
def _csr(cols, vals, d):
    """Rows with the same number of stored entries: cols, vals of shape (n, k)."""
    n, k = cols.shape
    indptr = torch.arange(0, n * k + 1, k, dtype=torch.int64, device=cols.device)
    return svm.DeviceCSR(n, d, indptr, cols.to(torch.int32).reshape(-1).contiguous(),
                         vals.to(torch.float32).reshape(-1).contiguous())


def _dense(x):
    n, d = x.shape
    return _csr(torch.arange(d, device=x.device).expand(n, d), x, d)


def _balanced(n, g):
    return torch.where(torch.randperm(n, device="cuda", generator=g) < n // 2, 1, -1).to(torch.int8)


def _rows(case, total, g):
    """Feature rows and labels of the case's data family: (CSR of all rows, labels)."""
    dev, data = "cuda", case["data"]

    def randn(*shape):
        return torch.randn(*shape, device=dev, generator=g)

    if data == "covtype":   # 10 dense columns, one-hot blocks of 4 and 40; a tanh network labels
        dense, blocks, hidden = 10, (4, 40), 32
        d = dense + sum(blocks)
        cats = [torch.randint(0, b, (total,), device=dev, generator=g) for b in blocks]
        x = randn(total, dense)
        cols = torch.stack([torch.full((total,), c, device=dev) for c in range(dense)] +
                           [dense + cats[0], dense + blocks[0] + cats[1]], 1)
        w1, b1, w2 = randn(d, hidden) / math.sqrt(12), 0.5 * randn(hidden), randn(hidden)
        score = torch.tanh(x @ w1[:dense] + w1[cols[:, 10]] + w1[cols[:, 11]] + b1) @ w2
        y = torch.where(score > score.median(), 1, -1)
        return _csr(cols, torch.cat([x, torch.ones(total, 2, device=dev)], 1), d), y.to(torch.int8)
    if data == "onehot":    # 14 one-hot groups over 123 columns, Zipf categories, an RBF teacher
        sizes = [2, 3, 4, 5, 6, 7, 8, 8, 9, 9, 10, 12, 16, 24]
        cols, offset = [], 0
        for s in sizes:
            p = 1.0 / torch.arange(1, s + 1, device=dev, dtype=torch.float32) ** 1.1
            c = torch.multinomial(p, total + 200, replacement=True, generator=g)
            cols.append(offset + torch.randperm(s, device=dev, generator=g)[c])
            offset += s
        cols = torch.stack(cols, 1)
        hot = torch.zeros(total + 200, offset, device=dev).scatter_(1, cols, 1.0)
        score = torch.exp(-0.05 * (28 - 2 * hot[:total] @ hot[total:].T)) @ randn(200)
        y = torch.where(score > torch.sort(score).values[int(0.76 * total)], 1, -1)
        y = torch.where(torch.rand(total, device=dev, generator=g) < 0.05, -y, y)
        return _csr(cols[:total], torch.ones(total, len(sizes), device=dev), offset), y.to(torch.int8)
    if data in ("gauss", "unit"):   # two dense Gaussian classes; "unit": L2-normalised rows
        d = case["d"]
        y = _balanced(total, g)
        x = randn(total, d)
        x[:, : min(5, d)] += 0.5 * y[:, None]
        if data == "unit":
            x = x / x.norm(dim=1, keepdim=True)
        return _dense(x), y
    # "sparse": 0.5% of the columns, lognormal values, L2-normalised, columns leaning on the class
    d = case["d"]
    k = max(1, int(round(0.005 * d)))
    y = _balanced(total, g)
    lean = torch.rand(total, d, device=dev, generator=g)
    half = torch.arange(d, device=dev)[None, :] < d // 2
    cols = torch.topk(lean + 0.2 * (half == (y[:, None] > 0)), k, dim=1).indices.sort(1).values
    v = torch.exp(randn(total, k))
    return _csr(cols, v / v.norm(dim=1, keepdim=True), d), y


def _split(X, y, n):
    cut = int(X.indptr[n])
    A = svm.DeviceCSR(n, X.d, X.indptr[: n + 1].clone(), X.indices[:cut].clone(), X.values[:cut].clone())
    B = svm.DeviceCSR(X.n - n, X.d, X.indptr[n:] - cut, X.indices[cut:].clone(), X.values[cut:].clone())
    return A, y[:n].contiguous(), B


def _multipliers(case, n, C, g):
    """Like a trained model's: a share of the rows, 70% of these at the bound."""
    u = torch.rand(n, device="cuda", generator=g, dtype=torch.float64)
    a = C * torch.rand(n, device="cuda", generator=g, dtype=torch.float64).clamp_(min=1e-3)
    a = torch.where(torch.rand(n, device="cuda", generator=g) < 0.7, torch.full_like(a, C), a)
    a[u >= case["sv"]] = 0.0
    a[:2] = C
    return a


def _decision_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X, y = _rows(case, case["n"] + case["m"], g)
    X, y, Z = _split(X, y, case["n"])
    C, gamma = {"covtype": (4.0, 0.1), "onehot": (1.0, 0.05), "gauss": (1.0, 0.05)}.get(
        case["data"], (2.0, 1.0 / X.d))
    return X, y, _multipliers(case, case["n"], C, g), 0.25, gamma, Z


def prepare(case, seed):
    kind, prec = case["kind"], PRECISION[case["precision"]]
    if kind in ("online", "heldout"):
        X, y, alpha, b, gamma, Z = _decision_inputs(case, seed)
        if kind == "heldout":
            return {"kind": kind, "args": (X, y, alpha, b, gamma, Z), "precision": prec}
        return {"kind": kind, "model": svm.Model(X, y, alpha, b, gamma, precision=prec), "Z": Z}
    g = torch.Generator(device="cuda").manual_seed(seed)
    if kind == "train":
        X, y = _rows(case, case["n"], g)
        return {"kind": kind, "args": (X, y, case["C"], case["gamma"], TAU), "precision": prec,
                "shrink": svm.POLICIES[case["policy"]]}
    if case["data"] == "ovo":
        # ten classes, the largest three times the smallest
        weight = torch.linspace(0.5, 1.5, 10, device="cuda").cumsum(0)
        labels = torch.bucketize(torch.linspace(0, 9.999, case["n"], device="cuda"), weight)
        labels = labels[torch.randperm(case["n"], device="cuda", generator=g)].clamp_(max=9)
        means = 0.3 * torch.randn(10, case["d"], device="cuda", generator=g)
        X = _dense(means[labels] + torch.randn(case["n"], case["d"], device="cuda", generator=g))
        pairs = [(a, b) for a in range(10) for b in range(a + 1, 10)]
        jobs = []
        for k in range(case["jobs"]):
            a, b = pairs[k % len(pairs)]
            rows = torch.nonzero((labels == a) | (labels == b)).reshape(-1)
            jobs.append({"rows": rows.to(torch.int32), "y": torch.where(labels[rows] == a, 1, -1).to(torch.int8),
                         "C": (1.0, 10.0)[k // len(pairs)], "gamma": 2.0 / case["d"], "tau": TAU})
    else:
        X, y = _rows(case, case["n"], g)
        jobs = [{"y": y, "C": 0.5 * 1.5 ** (k % 9), "gamma": 0.02 * 1.4 ** (k // 9), "tau": TAU}
                for k in range(case["jobs"])]
    return {"kind": kind, "X": X, "jobs": jobs, "precision": prec, "cluster_size": case["cluster_size"],
            "lanes_per_row": case["lanes_per_row"]}


# --------------------------------------------------------------------- run
def run(state):
    if state["kind"] == "online":
        return state["model"].decision(state["Z"])
    if state["kind"] == "heldout":
        return svm.svm_decision(*state["args"], precision=state["precision"])
    if state["kind"] == "train":
        r = svm.svm_train(*state["args"], precision=state["precision"], shrink=state["shrink"])
        return {"alpha": r["alpha"], "b": r["b"], "iters": r["iters"], "objective": r["stats"]["objective"]}
    r = svm.svm_train_batch(state["X"], state["jobs"], precision=state["precision"],
                            cluster_size=state["cluster_size"], lanes_per_row=state["lanes_per_row"])
    out = r["results"]
    return {"alpha": torch.cat([j["alpha"] for j in out]),
            "b": torch.tensor([j["b"] for j in out], dtype=torch.float64),
            "objective": torch.tensor([j["objective"] for j in out], dtype=torch.float64),
            "iters": torch.tensor([j["iters"] for j in out])}


def work(case):
    """Inputs read once, results written once, and the arithmetic of the kernel
    values: every (query, support vector) pair of a decision; for a training, a
    kernel row for each of the about n / 8 rows that end as support vectors."""
    entries = {"covtype": 12, "onehot": 14, "sparse": max(1, int(round(0.005 * case.get("d", 0))))}.get(
        case["data"], case.get("d", 0))
    row = 8 * entries + 8
    pair = 2 * entries + 10
    n, m = case["n"], case.get("m", 0)
    if case["kind"] == "online":
        return {"bytes": (n + m) * row + 8 * n + 8 * m, "flops": n * m * pair}
    if case["kind"] == "heldout":
        return {"bytes": (n + m) * row + 9 * n + 8 * m, "flops": case["sv"] * n * m * pair}
    if case["kind"] == "train":
        return {"bytes": n * row + 9 * n, "flops": n * n / 8 * pair}
    per = n / 5 if case["data"] == "ovo" else n
    return {"bytes": n * row + 13 * per * case["jobs"], "flops": case["jobs"] * per * per / 8 * pair}


# ------------------------------------------------------------------- exact
def _as_dense(X):
    rows = torch.repeat_interleave(torch.arange(X.n, device="cuda"), X.indptr[1:] - X.indptr[:-1])
    out = torch.zeros(X.n, X.d, dtype=torch.float64, device="cuda")
    out[rows, X.indices.long()] = X.values.double()
    return out


def exact(case, seed):
    """Decision values in 64 bits; a training's result is one of many within
    the tolerance, so it has no such value."""
    if case["kind"] not in ("online", "heldout"):
        return None
    X, y, alpha, b, gamma, Z = _decision_inputs(case, seed)
    keep = alpha > 0
    xs, coef = _as_dense(X)[keep], (alpha * y.double())[keep]
    xn, zs = (xs * xs).sum(1), _as_dense(Z)
    out = torch.empty(Z.n, dtype=torch.float64, device="cuda")
    for s in range(0, Z.n, 2048):
        z = zs[s:s + 2048]
        d2 = ((z * z).sum(1)[:, None] + xn[None, :] - 2.0 * (z @ xs.T)).clamp_(min=0.0)
        out[s:s + 2048] = torch.exp(-gamma * d2) @ coef - b
    return out
