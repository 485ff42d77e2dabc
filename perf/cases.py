"""Performance cases: the fits a user of this framework runs, through its public entry points.

A pass is a whole fit as a program with a data set in hand makes it: a context built from host
arrays, fitted, its descriptors and screened ids read back, the context closed (``Sisso``); or,
for many problems at once, new values loaded into a kept ``Batch``, one run, its results read
back.  A data set is fitted once, so building the context is part of the call.

The sizes are those of the seeded workloads in ``paper_2410_01752_gb300/inputs.py`` (20 to
65 536 samples, 4 to 12 primaries, rung 2 and 3, 1 to 5 terms) and odd ones between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_01752_gb300 import (GRAMMAR_EQ2, GRAMMAR_NEW_X_PREV, MLP, PREC_FP32, PREC_FP64, PREC_MIXED_BF16,
                                    PREC_MIXED_FP16, Batch, Sisso)
from paper_2410_01752_gb300.inputs import OPS9

PRECISION = {"fp64": PREC_FP64, "fp32": PREC_FP32, "bf16": PREC_MIXED_BF16, "fp16": PREC_MIXED_FP16}
MAX_COST = 1.2e12          # candidate-samples of a drawn case: those of the largest listed one


# ---- the cases ------------------------------------------------------------------------
def _fit(name, N, d, k, D, x, rung=2, precision="fp32", learned=False):
    return {"name": name, "kind": "fit", "N": N, "d": d, "rung": rung, "k": k, "D": D, "x": x,
            "precision": precision, "learned": learned}


def _batch(name, tasks, n_lo, n_hi, d_lo, d_hi, k, D, x):
    return {"name": name, "kind": "batch", "tasks": tasks, "n_lo": n_lo, "n_hi": n_hi, "d_lo": d_lo, "d_hi": d_hi,
            "rung": 2, "k": k, "D": D, "x": x}


def listed():
    return [
        # the smallest problem: a first look at twenty measurements of four quantities
        _fit("fit_smallest", 20, 4, 10, 2, "uniform"),
        # the paper's small data sets (tens of samples, three terms), in full FP64
        _fit("fit_small_fp64", 50, 5, 20, 3, "uniform", precision="fp64"),
        # the everyday fit: about a thousand samples, rung 2, three terms; ragged sizes
        _fit("fit_rung2", 1013, 9, 50, 3, "wide"),
        # five-term descriptors: the exhaustive search over C(300, 5) subsets weighs most
        _fit("fit_five_terms", 1234, 10, 60, 5, "uniform"),
        # the same fit with the learned subset proposal in the place of the exhaustive search
        _fit("fit_five_terms_learned", 1234, 10, 60, 5, "uniform", learned=True),
        # rung 3 on a small laboratory data set: few samples, 1.6e7 candidates
        _fit("fit_rung3_small", 333, 6, 37, 3, "lognormal", rung=3),
        # the headline workload: 2.9e8 rung-3 candidates per step, four terms
        _fit("fit_rung3", 1000, 10, 100, 4, "lognormal", rung=3),
        # long collinear sensor data in FP32: 65 536 samples
        _fit("fit_long_fp32", 65536, 12, 200, 3, "collinear"),
        # the same through the mixed form (FP16 on the tensor cores, FP64 refits)
        _fit("fit_long_fp16", 65536, 12, 200, 3, "collinear", precision="fp16"),
        # a shorter, ragged log of fewer sensors, BF16
        _fit("fit_long_bf16", 20011, 9, 100, 3, "collinear", precision="bf16"),
        # many independent problems of uneven sizes in one launch
        _batch("batch_tasks", 512, 20, 2000, 4, 12, 50, 3, "wide"),
        # an ensemble on disjoint subsets of one data set: 30 models of 100 samples
        _batch("batch_ensemble", 30, 100, 100, 4, 4, 20, 4, "uniform"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sizes(d, rung):
    """|phi_l| for l = 0..rung: nine operators, NEW_X_PREV pairs from level 3 on."""
    phi = [d]
    for level in range(1, rung + 1):
        P, Q = phi[-1], phi[-2] if level >= 2 else 0
        pairs = Q * (P - Q) if level >= 3 else P * (P - 1) // 2 - Q * (Q - 1) // 2
        phi.append(P + 5 * pairs + 5 * (P - Q))
    return phi


def _cost(c):
    """Candidate-samples scored over all steps."""
    if c["kind"] == "batch":
        N, d = 0.5 * (c["n_lo"] + c["n_hi"]), 0.5 * (c["d_lo"] + c["d_hi"])
        return c["tasks"] * N * _sizes(math.ceil(d), 2)[-1] * c["D"]
    return float(c["N"]) * _sizes(c["d"], c["rung"])[-1] * c["D"]


def draw(rng):
    while True:
        kind = rng.choice(["rung2", "rung2", "rung2", "five", "rung3", "rung3", "long", "long", "batch"])
        if kind == "rung2":
            c = _fit("", _log_int(rng, 20, 4000), rng.randint(4, 12), _log_int(rng, 10, 60), rng.randint(1, 3),
                     rng.choice(["uniform", "wide", "lognormal"]), precision=rng.choice(["fp32", "fp32", "fp64"]))
        elif kind == "five":
            c = _fit("", _log_int(rng, 500, 2000), rng.randint(8, 12), rng.randint(20, 60), rng.randint(4, 5), "uniform")
            c["learned"] = c["D"] == 5 and rng.random() < 0.4
        elif kind == "rung3":
            c = _fit("", _log_int(rng, 50, 1000), rng.randint(3, 10), _log_int(rng, 10, 100), rng.randint(2, 4),
                     rng.choice(["lognormal", "uniform"]), rung=3)
        elif kind == "long":
            c = _fit("", _log_int(rng, 5000, 65536), rng.randint(7, 12), _log_int(rng, 20, 200), rng.randint(2, 3),
                     "collinear", precision=rng.choice(["fp32", "bf16", "fp16"]))
        else:
            n_lo = _log_int(rng, 20, 200)
            c = _batch("", _log_int(rng, 8, 512), n_lo, _log_int(rng, max(100, n_lo), 2000), 4, rng.randint(4, 12),
                       rng.randint(10, 50), rng.randint(2, 3), rng.choice(["uniform", "wide"]))
        if _cost(c) <= MAX_COST:
            del c["name"]
            return c


# ---- inputs ---------------------------------------------------------------------------
_TERMS = [lambda x: x[0] * x[1] / x[2], lambda x: np.sqrt(x[0]) * x[3], lambda x: (x[1] + x[2]) ** 2,
          lambda x: np.log(x[3]) / x[0], lambda x: x[2] * x[2] / x[1], lambda x: np.exp(x[0] / x[3]),
          lambda x: (x[0] - x[1]) * x[2], lambda x: 1.0 / (x[1] * x[3])]


def _problem(r, N, d, x, n_terms, noise):
    """A data set with planted terms: primaries uniform in [1, 5] or [0.5, 5], lognormal, or half
    of them correlated 0.999 with one another; noise relative to the clean signal's deviation."""
    if x == "collinear":
        h = d // 2
        X = r.uniform(1.0, 5.0, size=(N, d))
        g = r.normal(size=(N, 1))
        X[:, :h] = 3.0 + 0.5 * (np.sqrt(0.999) * g + np.sqrt(0.001) * r.normal(size=(N, h)))
        c = r.uniform(1.0, 5.0, size=3) * r.choice([-1.0, 1.0], size=3)
        clean = (c[0] * X[:, 0] * X[:, h] ** 2 + c[1] * X[:, 1] / np.sqrt(X[:, h + 1])
                 + c[2] * np.log(X[:, 2]) * X[:, h + 2])
    else:
        X = (r.lognormal(0.0, 0.5, size=(N, d)) if x == "lognormal" else
             r.uniform(0.5 if x == "wide" else 1.0, 5.0, size=(N, d)))
        p = r.permutation(d) if d >= 4 else np.array([0, 1, 2, 0])
        cols = [X[:, j] for j in p[:4]]
        terms = r.choice(len(_TERMS), size=n_terms, replace=False)
        c = r.uniform(1.0, 5.0, size=n_terms) * r.choice([-1.0, 1.0], size=n_terms)
        clean = sum(ci * _TERMS[t](cols) for ci, t in zip(c, terms))
    return np.ascontiguousarray(X), clean + r.normal(0.0, noise * max(clean.std(), 1e-12), size=N)


def _problems(case, seed):
    r = np.random.default_rng([seed, 2410, 1752])
    if case["kind"] == "fit":
        return [_problem(r, case["N"], case["d"], case["x"], 3, 0.01)]
    shapes = np.random.default_rng([case["tasks"], case["n_lo"], case["n_hi"], case["d_hi"]])
    sizes = [(int(shapes.integers(case["n_lo"], case["n_hi"] + 1)), int(shapes.integers(case["d_lo"], case["d_hi"] + 1)))
             for _ in range(case["tasks"])]          # the shapes are the case's, the values the seed's
    return [_problem(r, N, d, case["x"], int(r.integers(1, 4)), 0.005) for N, d in sizes]


def prepare(case, seed):
    problems = _problems(case, seed)
    state = {"case": case, "problems": problems}
    if case["kind"] == "batch":
        state["batch"] = Batch(problems, OPS9, case["rung"], case["k"], case["D"])
    elif case["learned"]:
        # a proposal network whose corrections are small against the greedy base, as trained ones are
        state["mlp"] = MLP(seed=1)
        state["mlp"].set_params(state["mlp"].params() * np.float32(0.05))
    return state


def _grammar(case):
    return GRAMMAR_NEW_X_PREV if case["rung"] >= 3 else GRAMMAR_EQ2


# ---- one pass -------------------------------------------------------------------------
def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        b.load(state["problems"])
        b.run()
        return _pack(b.results(), case["D"])
    X, y = state["problems"][0]
    with Sisso(X, y, OPS9, case["rung"], case["k"], case["D"], precision=PRECISION[case["precision"]],
               grammar=_grammar(case)) as s:
        if case["learned"]:
            s.set_proposal(state["mlp"], 0.01, certify=False)
        dims = s.fit()
        sis = [np.array(s.sis(t + 1), dtype=np.int64) for t in range(len(dims))]
    return {"ids": [np.array(m.ids, dtype=np.int64) for m in dims], "coef": [np.array(m.coef) for m in dims],
            "rmse": np.array([m.rmse for m in dims]), "r2": np.array([m.r2 for m in dims]), "sis": sis}


def _pack(results, D):
    """The tasks' models as arrays: ids and coefficients of dimension t in row t - 1, 0 beyond them."""
    n = len(results)
    out = {"status": np.zeros(n, dtype=np.int64), "ids": np.full((n, D, D), -1, dtype=np.int64),
           "coef": np.zeros((n, D, D + 1)), "rmse": np.zeros((n, D)), "r2": np.zeros((n, D))}
    for i, (status, dims) in enumerate(results):
        out["status"][i] = status
        for t, m in enumerate(dims):
            out["ids"][i, t, : t + 1] = m.ids
            out["coef"][i, t, : t + 2] = m.coef
            out["rmse"][i, t], out["r2"][i, t] = m.rmse, m.r2
    return out


# ---- what a pass cannot do without ----------------------------------------------------
def work(case):
    """Data in, models out; per candidate-sample one operation and a square once, one multiply-add
    with the target per step; the Gram of the screened features; per t-subset the update of its last
    pivot and its residual (8 operations: the rest is shared with other subsets)."""
    def one(N, d):
        cand = float(_sizes(d, case["rung"])[-1])
        flops = cand * N * (3.0 + 2.0 * case["D"]) + float(case["k"] * case["D"]) ** 2 * N
        for t in range(1, case["D"] + 1):
            frac = 0.01 if case.get("learned") and t == 5 else 1.0
            flops += math.comb(case["k"] * t, t) * frac * 8.0
        return 8.0 * N * (d + 1) + 8.0 * case["D"] * (case["k"] + 8), flops

    if case["kind"] == "batch":
        parts = [one(len(y), X.shape[1]) for X, y in _problems(case, 0)]
    else:
        parts = [one(case["N"], case["d"])]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ---- the same fits in plain torch, 64 bits --------------------------------------------
_BINARY = (torch.add, torch.sub, torch.mul, torch.div)
_UNARY = (torch.exp, torch.log, torch.sqrt, torch.square, torch.reciprocal)


def _pairs(P, Q, ordered, new_x_prev, dev):
    """Operand pairs of one binary operator, in lexicographic order."""
    if new_x_prev:
        lo, hi = torch.arange(Q, device=dev), torch.arange(Q, P, device=dev)
        a, b = torch.cartesian_prod(lo, hi).unbind(1)
        if ordered:
            c, e = torch.cartesian_prod(hi, lo).unbind(1)
            a, b = torch.cat([a, c]), torch.cat([b, e])
        return a, b
    if ordered:
        a, b = torch.cartesian_prod(torch.arange(P, device=dev), torch.arange(P, device=dev)).unbind(1)
        keep = (a != b) & ((a >= Q) | (b >= Q))
    else:
        a, b = torch.triu_indices(P, P, 1, device=dev).unbind(0)
        keep = b >= Q
    return a[keep], b[keep]


def _level(P, Q, new_x_prev, dev):
    """(operator, first operands, second operands or None) of one level's sections, in id order."""
    for o in range(4):
        yield (o, *_pairs(P, Q, o == 3, new_x_prev, dev))
    for o in range(5):
        yield 4 + o, torch.arange(Q, P, device=dev), None


def _values(V, op, a, b):
    if b is None:
        v = _UNARY[op - 4](V[a])
        return v, None
    x, z = V[a], V[b]
    return _BINARY[op](x, z), (x.abs() + z.abs()).amax(1) if op < 2 else None


def _stats(v, mag):
    """(valid, mean, deviation) per row: finite, at most 1e12, not constant, not cancelled."""
    mx = v.abs().amax(1)
    mean = v.mean(1)
    sd = (v - mean[:, None]).square().mean(1).sqrt()
    ok = torch.isfinite(v).all(1) & (mx <= 1e12) & (sd > 1e-6 * mx)
    return (ok if mag is None else ok & (mx > 1e-9 * mag)), mean, sd


class _Space64:
    """Values of phi_(L-1) and the sections of level L."""

    def __init__(self, X, rung, new_x_prev):
        dev = X.device
        self.V, self.ok = X.t().contiguous(), None
        self.ok = _stats(self.V, None)[0]
        sizes = [0, self.V.shape[0]]
        for level in range(1, rung):
            P, Q = sizes[-1], sizes[-2]
            rows, oks = [self.V], [self.ok]
            for op, a, b in _level(P, Q, False, dev):
                v, mag = _values(self.V, op, a, b)
                ok = _stats(v, mag)[0] & self.ok[a]
                rows.append(v)
                oks.append(ok if b is None else ok & self.ok[b])
            self.V, self.ok = torch.cat(rows), torch.cat(oks)
            sizes.append(self.V.shape[0])
        self.P = sizes[-1]
        self.top = list(_level(sizes[-1], sizes[-2], new_x_prev and rung >= 3, dev))
        self.base = np.cumsum([self.P] + [len(t[1]) for t in self.top])

    def rows(self, ids):
        out = []
        for i in ids:
            if i < self.P:
                out.append(self.V[i])
                continue
            s = int(np.searchsorted(self.base, i, side="right")) - 1
            op, a, b = self.top[s]
            q = slice(int(i - self.base[s]), int(i - self.base[s]) + 1)
            out.append(_values(self.V, op, a[q], None if b is None else b[q])[0][0])
        return torch.stack(out)

    def scores(self, t):
        """Pearson |rho| of every candidate with t, -1 where it is not valid."""
        tc = t - t.mean()
        scale = 1.0 / (t.numel() * tc.square().mean().sqrt())

        def score(v, mag, ok):
            good, mean, sd = _stats(v, mag)
            rho = ((v - mean[:, None]) @ tc).abs() * scale / sd
            return torch.where(good & ok, rho, -torch.ones_like(rho))

        out = [score(self.V, None, self.ok)]
        step = max(1, (1 << 26) // t.numel())
        for op, a, b in self.top:
            for lo in range(0, len(a), step):
                p, q = a[lo:lo + step], None if b is None else b[lo:lo + step]
                v, mag = _values(self.V, op, p, q)
                out.append(score(v, mag, self.ok[p] if q is None else self.ok[p] & self.ok[q]))
        return torch.cat(out)


def _screen(space, target, S, k):
    """The k best ids against target: ties within 1e-9 go to the lowest id, duplicates of accepted ones are passed over."""
    sc = space.scores(target)
    sc[torch.tensor(S, dtype=torch.long, device=sc.device)] = -1.0
    n = min(sc.numel(), max(4096, 64 * k))
    top = torch.topk(sc, n)
    left = sorted(((s, i) for s, i in zip(top.values.tolist(), top.indices.tolist()) if s >= 0), key=lambda p: (-p[0], p[1]))

    def standard(ids):
        v = space.rows(ids)
        v = v - v.mean(1, keepdim=True)
        return v / v.square().mean(1, keepdim=True).sqrt()

    refs = torch.empty((len(S) + k, target.numel()), dtype=torch.float64, device=target.device)
    if S:
        refs[: len(S)] = standard(S)
    acc = []
    while left and len(acc) < k:
        w = 0
        while w < len(left) and left[w][0] >= left[0][0] - 1e-9:
            w += 1
        at = min(range(w), key=lambda q: left[q][1])
        i = left.pop(at)[1]
        z = standard([i])
        r = refs[: len(S) + len(acc)]
        if len(r) and bool((torch.minimum((r - z).abs().amax(1), (r + z).abs().amax(1)) <= 1e-8).any()):
            continue
        refs[len(S) + len(acc)] = z[0]
        acc.append(i)
    return acc


def _best(V, y, S, t):
    """Ids of the lowest-RSS t-subset of the columns V (rows of S): exhaustive, ties to the smallest ids."""
    n, N = V.shape
    Z = V - V.mean(1, keepdim=True)
    Z = Z / Z.square().mean(1, keepdim=True).sqrt()
    yc = y - y.mean()
    G, b, syy = Z @ Z.t() / N, Z @ yc / N, yc.square().mean()
    sub = torch.combinations(torch.arange(n, device=V.device), t)
    L, w = [[None] * t for _ in range(t)], []
    good = torch.ones(len(sub), dtype=torch.bool, device=V.device)
    for i in range(t):
        for j in range(i + 1):
            s = G[sub[:, i], sub[:, j]] - sum(L[i][m] * L[j][m] for m in range(j))
            if i == j:
                good &= s > 1e-12
                L[i][i] = s.clamp_min(1e-300).sqrt()
            else:
                L[i][j] = s / L[j][j]
        w.append((b[sub[:, i]] - sum(L[i][m] * w[m] for m in range(i))) / L[i][i])
    rss = torch.where(good, syy - sum(x.square() for x in w), torch.inf)
    tied = sub[rss <= rss.min() + 1e-12 * syy].cpu().numpy()
    return min(tuple(sorted(S[p] for p in q)) for q in tied)


def _fit64(X, y, case):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    Xd, yd = torch.tensor(X, dtype=torch.float64, device=dev), torch.tensor(y, dtype=torch.float64, device=dev)
    space = _Space64(Xd, case["rung"], _grammar(case) == GRAMMAR_NEW_X_PREV)
    S, sis, dims, target = [], [], [], yd
    for t in range(1, case["D"] + 1):
        sis.append(_screen(space, target, S, case["k"]))
        S = S + sis[-1]
        if len(S) < t:
            break
        ids = _best(space.rows(S), yd, S, t)
        F = space.rows(ids).cpu().numpy()
        mean, sd = F.mean(1), F.std(1)
        c = np.linalg.lstsq(((F - mean[:, None]) / sd[:, None]).T, y - y.mean(), rcond=None)[0] / sd
        coef = np.concatenate([[y.mean() - c @ mean], c])
        res = y - coef[0] - c @ F
        dims.append((ids, coef, math.sqrt(np.mean(res ** 2)), 1.0 - np.sum(res ** 2) / np.sum((y - y.mean()) ** 2)))
        target = torch.tensor(res, device=dev)
        if dims[-1][2] <= 1e-10 * y.std():
            break
    return dims, sis[: len(dims)]


def exact(case, seed):
    """The fit in 64 bits; None where enumerating it in plain torch would take too long."""
    if max(case["k"] * t for t in range(1, case["D"] + 1)) ** case["D"] > 3e8 or case.get("learned"):
        return None
    if case["kind"] == "batch":
        if case["tasks"] > 32:
            return None
        out = {k: v for k, v in _pack([(0, [])] * case["tasks"], case["D"]).items()}
        for i, (X, y) in enumerate(_problems(case, seed)):
            for t, (ids, coef, rmse, r2) in enumerate(_fit64(X, y, case)[0]):
                out["ids"][i, t, : t + 1] = ids
                out["coef"][i, t, : t + 2] = coef
                out["rmse"][i, t], out["r2"][i, t] = rmse, r2
        return out
    if _cost(case) > 1.5e11:
        return None
    X, y = _problems(case, seed)[0]
    dims, sis = _fit64(X, y, case)
    return {"ids": [np.array(m[0], dtype=np.int64) for m in dims], "coef": [m[1] for m in dims],
            "rmse": np.array([m[2] for m in dims]), "r2": np.array([m[3] for m in dims]),
            "sis": [np.array(s, dtype=np.int64) for s in sis]}
