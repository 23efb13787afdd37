"""Timed cases: the work a user of the library has it do, through its public
Python binding and pipeline.

Every case builds its inputs from the seed alone (node sets in the unit cube or
unit ball, interior nodes first, then Dirichlet boundary nodes; a Gaussian or
plane-wave exact solution; for the full SVD and the projected solves with
measurement noise on the data), and returns everything the call computes.

Kinds:
  train      one Adam step of the stop network on one batch
  projected  lambda / rank choice and lift on a finished GKB run
  matvec     one product with A and one with its transpose
  solve      assemble (or matrix-free) -> GKB -> HKT / Ine-TSVD -> u
  many       several (c, k) solves on the same nodes at once
  batch      uneven instances in one batched GKB + HKT
  fullsvd    Tikhonov with GCV or TSVD through the full SVD
  evaluate   reconstruction on a field of points
  label      every Krylov vector at the test points + the error table
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_09798_gb300 import pipeline as P
from paper_2511_09798_gb300 import rbfkr as R

DEV = "cuda"
L2_BYTES = 126e6  # a matrix below this stays on the chip between the steps of a run

_ctx = None


def ctx():
    """One context for all solves, as a program that solves many problems keeps."""
    global _ctx
    if _ctx is None:
        _ctx = R.Context(0)
    return _ctx


# --------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------

def listed():
    return [
        # the smallest calls: one optimiser step of the stop network at the batch of its training program
        dict(name="train_512", kind="train", batch=512),
        # another parameter choice on a run already made: projected SVD, lambda grid, lift (l = 150 is the longest run)
        dict(name="hkt_l150", kind="projected", n=8000, steps=150, method="gcv"),
        # the operator applied once each way (residual checks, outer iterations), 512 MB matrix
        dict(name="matvec_8000", kind="matvec", n=8000, precision="fp64", storage="assembled", form="c"),
        # one small problem from nodes to u: launches and latency
        dict(name="solve_1000", kind="solve", domain="cube", n=1000, steps=40, precision="fp64", storage="assembled",
             method="hkt", form="c", c=0.3, k=2.0, m=2000),
        # an odd, middle-sized problem with the longer runs and the rank choice of the accuracy tables
        dict(name="tsvd_2161", kind="solve", domain="sphere", n=2161, steps=140, precision="fp64", storage="assembled",
             method="ine_tsvd", form="eps", c=0.25, k=3.0, m=2000),
        # FP32 matrix-free products on a ball too large to store comfortably in FP64
        dict(name="mixed_20000", kind="solve", domain="sphere", n=20000, steps=60, precision="mixed", storage="free",
             method="hkt", form="c", c=0.15, k=10.0, m=2000),
        # the six (c, k) problems of the cube at N = 8000, 100 steps each, at once: the headline workload
        dict(name="many6_8000", kind="many", n=8000, steps=100, count=6, m=2000),
        # a sweep of uneven instances through the batched path
        dict(name="batch_24", kind="batch", count=24, n_lo=2000, n_hi=8000, steps=40, sizes=7),
        # full-SVD Tikhonov with GCV, small and large
        dict(name="tikhonov_1000", kind="fullsvd", n=1000, method="tikhonov", c=0.3, k=2.0),
        dict(name="tikhonov_3001", kind="fullsvd", n=3001, method="tikhonov", c=0.2, k=3.0),
        # the field u on many points (plots, error maps)
        dict(name="field_20000", kind="evaluate", n=20000, m=20000, form="c", c=0.15),
        # labelling one training run: 150 Krylov vectors at 500 points, errors over (l, lambda)
        dict(name="label_8000", kind="label", n=8000, steps=150, m=500),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "projected", "matvec", "solve", "solve", "many", "batch", "fullsvd", "evaluate",
                       "label"])
    if kind == "train":
        return dict(kind=kind, batch=_log(rng, 64, 2048))
    if kind == "projected":
        n = _log(rng, 500, 16000)
        return dict(kind=kind, n=n, steps=rng.randint(15, 150),
                    method=rng.choice(["gcv", "gcv", "lcurve", "fixed_t", "ine_tsvd", "lsqr"]))
    if kind == "matvec":
        precision = rng.choice(["fp64", "fp64", "mixed"])
        storage = rng.choice(["assembled", "assembled", "free"])
        return dict(kind=kind, n=_log(rng, 500, 16000 if storage == "assembled" or precision == "mixed" else 8000),
                    precision=precision, storage=storage, form=rng.choice(["c", "eps"]))
    if kind == "solve":
        precision, storage = rng.choice([("fp64", "assembled")] * 4 + [("mixed", "free"), ("mixed", "assembled")])
        n = _log(rng, 343, 10000)
        top = 140 if precision == "fp64" else 40
        return dict(kind=kind, domain=rng.choice(["cube", "sphere"]), n=n, steps=rng.randint(15, top),
                    precision=precision, storage=storage, method=rng.choice(["hkt", "hkt", "ine_tsvd"]),
                    form=rng.choice(["c", "c", "eps"]), c=round(rng.uniform(0.1, 0.4), 3),
                    k=round(rng.uniform(1.0, 10.0), 2), m=_log(rng, 300, 4000))
    if kind == "many":
        return dict(kind=kind, n=_log(rng, 1000, 8000), steps=rng.randint(40, 100), count=rng.randint(2, 6),
                    m=_log(rng, 500, 4000))
    if kind == "batch":
        lo = rng.randint(500, 2000)
        return dict(kind=kind, count=rng.randint(8, 24), n_lo=lo, n_hi=rng.randint(2 * lo, 8000),
                    steps=rng.randint(15, 40), sizes=rng.randint(1, 10**6))
    if kind == "fullsvd":
        return dict(kind=kind, n=_log(rng, 343, 2600), method=rng.choice(["tikhonov", "tikhonov", "tsvd"]),
                    c=round(rng.uniform(0.15, 0.3), 3), k=round(rng.uniform(1.0, 5.0), 2))
    if kind == "evaluate":
        return dict(kind=kind, n=_log(rng, 1000, 20000), m=_log(rng, 500, 20000), form=rng.choice(["c", "eps"]),
                    c=round(rng.uniform(0.05, 1.0), 3))
    return dict(kind=kind, n=_log(rng, 2000, 12000), steps=rng.randint(50, 150), m=500)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _rng(*key):
    return np.random.Generator(np.random.PCG64(list(key)))


def _nodes(domain, n, rng):
    """n x 3 nodes, interior first; returns (X, n_interior)."""
    nb = int(round((0.3 if domain == "cube" else 0.2) * n))
    ni = n - nb
    if domain == "cube":
        inner = rng.uniform(1e-6, 1.0 - 1e-6, (ni, 3))
        outer = rng.uniform(0.0, 1.0, (nb, 3))
        face = rng.integers(0, 6, nb)
        outer[np.arange(nb), face // 2] = face % 2
    else:
        v = rng.normal(size=(ni, 3))
        inner = v / np.linalg.norm(v, axis=1, keepdims=True) * rng.uniform(0.0, 0.999, (ni, 1)) ** (1.0 / 3.0)
        i = np.arange(nb)
        z = 1.0 - (2.0 * i + 1.0) / nb
        phi = i * math.pi * (3.0 - math.sqrt(5.0))
        rho = np.sqrt(1.0 - z * z)
        outer = np.stack([rho * np.cos(phi), rho * np.sin(phi), z], 1)
    return np.concatenate([inner, outer]), ni


def _points(domain, m, rng):
    if domain == "cube":
        return rng.uniform(0.0, 1.0, (m, 3))
    v = rng.normal(size=(m, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True) * rng.uniform(0.0, 1.0, (m, 1)) ** (1.0 / 3.0)


class _Problem:
    """Node set, exact solution and data f = [source; boundary values] of one seed."""

    def __init__(self, domain, n, k, seed, m=0, wave=False, noise=0.0):
        rng = _rng(11, seed, n)
        self.X, self.ni = _nodes(domain, n, rng)
        self.points = _points(domain, m, rng) if m else None
        self.wave, self.k = wave, k
        d = rng.normal(size=3)
        self.d = d / np.linalg.norm(d)
        self.sigma = float(rng.uniform(0.5, 2.0))
        self.center = rng.uniform(0.3, 0.7, 3) if domain == "cube" else rng.uniform(-0.4, 0.4, 3)
        u = self.field(self.X)
        f = u.copy()
        if wave:
            f[: self.ni] = 0.0
        else:
            r2 = np.sum((self.X[: self.ni] - self.center) ** 2, axis=1)
            s = self.sigma
            f[: self.ni] = (4.0 * r2 / s**2 - 6.0 / s + k * k) * u[: self.ni]
        if noise:
            f = f + noise * np.sqrt(np.mean(f * f)) * rng.normal(size=n)
        self.f = f

    def field(self, Q):
        if self.wave:
            return np.sin(self.k * (Q @ self.d))
        return np.exp(-np.sum((Q - self.center) ** 2, axis=1) / self.sigma)


def _dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device=DEV)


def _prec(case):
    return R.RBF_FP64 if case["precision"] == "fp64" else R.RBF_MIXED


def _form(case):
    return R.RBF_FORM_EPS if case.get("form") == "eps" else R.RBF_FORM_C


def _storage(case):
    return R.RBF_ASSEMBLED if case["storage"] == "assembled" else R.RBF_MATRIX_FREE


MANY_C, MANY_K = (0.1, 0.2, 0.5), (2.0, 5.0)
ELLS = tuple(range(10, 151, 10))
T_STRIDE = 4


def _many_params(case):
    return [(c, k) for c in MANY_C for k in MANY_K][: case["count"]]


def _batch_sizes(case):
    r = _rng(5, case["sizes"])
    return [int(v) for v in r.integers(case["n_lo"], case["n_hi"] + 1, case["count"])]


def _batch_problems(case, seed):
    out = []
    for b, n in enumerate(_batch_sizes(case)):
        r = _rng(6, case["sizes"], b)
        domain = "cube" if r.random() < 0.5 else "sphere"
        c, k = float(np.exp(r.uniform(np.log(0.05), np.log(0.5)))), float(r.uniform(1.0, 12.0))
        out.append((_Problem(domain, n, k, seed * 1000 + b, wave=b % 2 == 0), c, k))
    return out


def _train_inputs(case, seed):
    r = _rng(21, seed)
    shapes = ((20, 128), (128, 128), (128, 2))
    parts = []
    for fi, fo in shapes:
        a = math.sqrt(6.0 / (fi + fo))
        parts += [r.uniform(-a, a, fi * fo), 0.05 * r.normal(size=fo)]
    p = np.concatenate(parts).astype(np.float32)
    x = r.normal(size=(case["batch"], 20)).astype(np.float32)
    y = np.stack([np.tanh(x[:, :10].sum(1) / 3.0), 0.5 * x[:, 10] * x[:, 3]], 1) + 0.1 * r.normal(size=(case["batch"], 2))
    m = (1e-2 * r.normal(size=p.size)).astype(np.float32)
    v = (1e-4 * r.uniform(0.5, 2.0, p.size)).astype(np.float32)
    return p, m, v, x, y.astype(np.float32)


TRAIN_T, TRAIN_LR = 1000, 1e-3


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "train":
        p, m, v, x, y = _train_inputs(case, seed)
        st.update(p=_dev(p, torch.float32), m=_dev(m, torch.float32), v=_dev(v, torch.float32),
                  x=_dev(x, torch.float32), y=_dev(y, torch.float32), t=TRAIN_T)
        st["g"] = torch.zeros_like(st["p"])
        return st
    if kind == "projected":
        n, l = case["n"], case["steps"]
        pr, c, k = _projected_problem(case, seed)
        W, Z, a, b = _gkb64(_matrix(pr.X, pr.ni, c, k), _dev(pr.f), l)
        st["state"], *st["keep"] = R.make_state(torch, n, l)
        ctx().rbf_gkb_restore(st["state"], dict(W=W.cpu().numpy(), Z=Z.cpu().numpy(), alpha=a.cpu().numpy(),
                                                beta=b.cpu().numpy(), steps_done=l, breakdown=0,
                                                c_hat=float(a.max())))
        st["coef"] = torch.empty(n, dtype=torch.float64, device=DEV)
        st["curve"] = torch.empty(max(ctx().grid_j, l), dtype=torch.float64, device=DEV)
        return st
    if kind == "matvec":
        pr, x1, x2, c, k = _matvec_inputs(case, seed)
        n = case["n"]
        nodes = _dev(pr.X.T)
        A, lda = None, 0
        if case["storage"] == "assembled":
            lda = R.padded_lda(n, _prec(case))
            A = torch.zeros((n, lda), dtype=torch.float64 if case["precision"] == "fp64" else torch.float32, device=DEV)
        st["op"] = ctx().rbf_operator_init(nodes, n, pr.ni, c, k, _storage(case), _prec(case), _form(case), A, lda)
        if A is not None:
            ctx().rbf_assemble(st["op"])
        st.update(x1=_dev(x1), x2=_dev(x2), y1=torch.empty(n, dtype=torch.float64, device=DEV),
                  y2=torch.empty(n, dtype=torch.float64, device=DEV))
        return st
    if kind == "solve":
        pr = _solve_problem(case, seed)
        st["prob"] = P.to_device(torch, pr.X.T, pr.f, pr.points, pr.ni, case["c"], case["k"])
        st["buf"] = P.allocate(torch, ctx(), st["prob"], case["steps"], _prec(case), _storage(case))
        return st
    if kind == "many":
        n, m = case["n"], case["m"]
        params = _many_params(case)
        prs = [_Problem("cube", n, k, seed, m=m, wave=True) for _, k in params]
        nodes = _dev(prs[0].X.T)
        lda = R.padded_lda(n, R.RBF_FP64)
        st["nodes"], st["points"] = nodes, _dev(prs[0].points.T)
        st["A"] = [torch.empty((n, lda), dtype=torch.float64, device=DEV) for _ in params]
        st["ops"] = [ctx().rbf_operator_init(nodes, n, prs[0].ni, c, k, A=A, lda=lda) for (c, k), A in zip(params, st["A"])]
        st["f"] = [_dev(p.f) for p in prs]
        st["states"], st["keep"] = [], []
        for _ in params:
            s, *kp = R.make_state(torch, n, case["steps"])
            st["states"].append(s)
            st["keep"].append(kp)
        st["coef"] = torch.empty((len(params), n), dtype=torch.float64, device=DEV)
        st["u"] = torch.empty((len(params), m), dtype=torch.float64, device=DEV)
        return st
    if kind == "batch":
        probs = _batch_problems(case, seed)

        class Set:
            def __init__(self, p):
                self.X, self.n_interior = p.X, p.ni

        st["batch"], st["keep"] = R.make_batch(torch, [Set(p) for p, _, _ in probs], [c for _, c, _ in probs],
                                               [k for _, _, k in probs], [p.f for p, _, _ in probs], case["steps"])
        st["coef"] = torch.empty(int(st["keep"]["offsets"][-1]), dtype=torch.float64, device=DEV)
        return st
    if kind == "fullsvd":
        n = case["n"]
        pr = _Problem("cube", n, case["k"], seed, noise=1e-2)
        lda = R.padded_lda(n, R.RBF_FP64)
        st["A"] = torch.zeros((n, lda), dtype=torch.float64, device=DEV)
        st["op"] = ctx().rbf_operator_init(_dev(pr.X.T), n, pr.ni, case["c"], case["k"], A=st["A"], lda=lda)
        ctx().rbf_assemble(st["op"])
        st["f"] = _dev(pr.f)
        st["coef"] = torch.empty(n, dtype=torch.float64, device=DEV)
        return st
    if kind == "evaluate":
        X, ni, pts, coef = _evaluate_inputs(case, seed)
        st["op"] = ctx().rbf_operator_init(_dev(X.T), case["n"], ni, case["c"], 2.0, R.RBF_MATRIX_FREE, R.RBF_MIXED,
                                           _form(case))
        st.update(points=_dev(pts.T), coef=_dev(coef), u=torch.empty(case["m"], dtype=torch.float64, device=DEV))
        return st
    # label
    n, l, m = case["n"], case["steps"], case["m"]
    pr, c, k = _label_problem(case, seed)
    W, Z, a, b = _gkb64(_matrix(pr.X, pr.ni, c, k), _dev(pr.f), l)
    st["state"], *st["keep"] = R.make_state(torch, n, l)
    ctx().rbf_gkb_restore(st["state"], dict(W=W.cpu().numpy(), Z=Z.cpu().numpy(), alpha=a.cpu().numpy(),
                                            beta=b.cpu().numpy(), steps_done=l, breakdown=0, c_hat=float(a.max())))
    st["op"] = ctx().rbf_operator_init(_dev(pr.X.T), n, pr.ni, c, k, R.RBF_MATRIX_FREE, R.RBF_MIXED)
    st["points"], st["uref"] = _dev(pr.points.T), _dev(pr.field(pr.points))
    st["ells"] = [e for e in ELLS if e <= l]
    st["G"] = torch.empty((l, m), dtype=torch.float64, device=DEV)
    st["err"] = torch.empty((len(st["ells"]), (ctx().grid_j - 1) // T_STRIDE + 1), dtype=torch.float64, device=DEV)
    return st


def _projected_problem(case, seed):
    r = _rng(31, seed)
    c, k = float(r.uniform(0.1, 0.3)), float(r.uniform(1.0, 6.0))
    return _Problem("cube", case["n"], k, seed, noise=1e-3), c, k


def _label_problem(case, seed):
    r = _rng(32, seed)
    c, k = float(r.uniform(0.1, 0.3)), float(r.uniform(1.0, 6.0))
    return _Problem("sphere", case["n"], k, seed, m=case["m"]), c, k


def _solve_problem(case, seed):
    return _Problem(case["domain"], case["n"], case["k"], seed, m=case["m"])


def _matvec_inputs(case, seed):
    r = _rng(33, seed)
    c, k = float(r.uniform(0.1, 0.5)), float(r.uniform(1.0, 10.0))
    pr = _Problem("sphere", case["n"], k, seed)
    return pr, r.normal(size=case["n"]), r.normal(size=case["n"]), c, k


def _evaluate_inputs(case, seed):
    r = _rng(34, seed)
    X, ni = _nodes("sphere", case["n"], r)
    return X, ni, _points("sphere", case["m"], r), r.normal(size=case["n"])


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

RULES = {"gcv": (R.RBF_GCV, 0.0), "lcurve": (R.RBF_LCURVE, 0.0), "fixed_t": (R.RBF_FIXED_T, -4.0)}


def run(st):
    case, cx = st["case"], ctx()
    kind = case["kind"]
    if kind == "train":
        cx.rbf_mlp_train_step(st["p"], st["m"], st["v"], st["t"], TRAIN_LR, st["x"], st["y"], case["batch"], st["g"])
        st["t"] += 1
        return {"p": st["p"], "m": st["m"], "v": st["v"], "g": st["g"]}
    if kind == "projected":
        return _run_projected(st, cx)
    if kind == "matvec":
        cx.rbf_matvec(st["op"], 0, st["x1"], st["y1"])
        cx.rbf_matvec(st["op"], 1, st["x2"], st["y2"])
        return {"y1": st["y1"], "y2": st["y2"]}
    if kind == "solve":
        buf = st["buf"]
        _, info = P.solve(cx, st["prob"], buf, case["steps"], _prec(case), _storage(case), method=case["method"],
                          form=_form(case))
        W, Z, a, b = buf.keep
        out = {"W": W, "Z": Z, "alpha": a, "beta": b, "coef": buf.coef, "u": buf.u, "steps": info.steps,
               "sigma1": info.sigma1, "eta": info.eta, "rho": info.rho}
        if case["method"] == "hkt":
            out.update(gcv=buf.curve[: cx.grid_j], index=info.index, lam=info.lambda_)
        else:
            out["rank"] = info.rank
        return out
    if kind == "many":
        m, n = case["m"], case["n"]
        coefs = [st["coef"][i] for i in range(case["count"])]
        cx.rbf_gkb_many(st["ops"], st["f"], case["steps"], st["states"], assemble=True)
        infos = cx.rbf_hkt_many(st["states"], R.RBF_GCV, 0.0, coefs)
        for i in range(0, case["count"], 2):  # two runs of the same c share the basis values
            cnt = min(2, case["count"] - i)
            cx.rbf_evaluate_many(st["ops"][i], st["coef"][i:i + cnt], n, cnt, st["points"], m, st["u"][i:i + cnt])
        out = {"coef": st["coef"], "u": st["u"], "index": [i.index for i in infos], "lam": [i.lambda_ for i in infos]}
        for i, (W, Z, a, b) in enumerate(st["keep"]):
            out.update({f"W{i}": W, f"Z{i}": Z, f"alpha{i}": a, f"beta{i}": b})
        return out
    if kind == "batch":
        bt, keep = st["batch"], st["keep"]
        cx.rbf_batch_gkb(bt, case["steps"])
        lam = cx.rbf_batch_hkt(bt, R.RBF_GCV, st["coef"])
        return {"W": keep["W"], "Z": keep["Z"], "alpha": keep["alpha"], "beta": keep["beta"], "coef": st["coef"],
                "lam": np.asarray(lam), "steps": np.asarray(list(keep["steps_done"]))}
    if kind == "fullsvd":
        if case["method"] == "tikhonov":
            info = cx.rbf_tikhonov(st["op"], st["f"], R.RBF_GCV, 0.0, st["coef"])
            return {"coef": st["coef"], "index": info.index, "lam": info.lambda_, "sigma1": info.sigma1}
        info = cx.rbf_tsvd(st["op"], st["f"], 0, st["coef"])
        return {"coef": st["coef"], "rank": info.rank, "sigma1": info.sigma1}
    if kind == "evaluate":
        cx.rbf_evaluate(st["op"], st["coef"], st["points"], case["m"], st["u"])
        return {"u": st["u"]}
    n, l, m = case["n"], case["steps"], case["m"]
    s = st["state"]
    cx.rbf_evaluate_many(st["op"], s.d_Z, n, l, st["points"], m, st["G"])
    cx.rbf_hkt_error_table(s, st["G"], m, m, st["uref"], st["ells"], T_STRIDE, st["err"])
    return {"G": st["G"], "err": st["err"]}


def _run_projected(st, cx):
    s, coef, curve, meth = st["state"], st["coef"], st["curve"], st["case"]["method"]
    if meth in RULES:
        rule, val = RULES[meth]
        info = cx.rbf_hkt(s, rule, val, coef, curve)
        out = {"coef": coef, "index": info.index, "lam": info.lambda_, "sigma1": info.sigma1, "eta": info.eta,
               "rho": info.rho}
        if meth == "gcv":
            out["gcv"] = curve[: cx.grid_j]
        return out
    if meth == "ine_tsvd":
        info = cx.rbf_ine_tsvd(s, 0, coef)
        return {"coef": coef, "rank": info.rank, "eta": info.eta, "rho": info.rho}
    info = cx.rbf_lsqr(s, R.RBF_GCV, 0, coef, curve)
    return {"coef": coef, "rank": info.rank, "eta": info.eta, "rho": info.rho, "gcv": curve[: st["case"]["steps"]]}


# --------------------------------------------------------------------------
# necessary work of one pass
# --------------------------------------------------------------------------

def _gkb_work(n, l, assembled, bytes_per):
    """One GKB run: 2 l products and the two-pass reorthogonalization of both bases."""
    flops = 2.0 * l * 2.0 * n * n + 2.0 * 8.0 * n * l * (l + 1) / 2.0
    byts = 8.0 * n * (2 * l + 1) + 24.0 * n
    if assembled:
        a = bytes_per * n * n
        byts += a + (a if a <= L2_BYTES else 2.0 * l * a)  # written once, read per product when it leaves the chip
    else:
        flops += 2.0 * l * 10.0 * n * n / 2.0  # every node pair evaluated once per product
    return byts, flops


def work(case):
    kind = case["kind"]
    if kind == "train":
        b, p = case["batch"], R.RBF_MLP_PARAMS
        return {"bytes": 4.0 * (22 * b + 7 * p), "flops": 6.0 * b * p + 12.0 * p}
    if kind == "projected":
        n, l = case["n"], case["steps"]
        return {"bytes": 8.0 * (n * l + n + 2 * l), "flops": 2.0 * n * l + 30.0 * l * l}
    if kind == "matvec":
        n = case["n"]
        a = (8.0 if case["precision"] == "fp64" else 4.0) * n * n if case["storage"] == "assembled" else 24.0 * n
        return {"bytes": 2.0 * a + 32.0 * n, "flops": 4.0 * n * n + (0.0 if case["storage"] == "assembled" else 10.0 * n * n)}
    if kind == "solve":
        n, l, m = case["n"], case["steps"], case["m"]
        b, f = _gkb_work(n, l, case["storage"] == "assembled", 8.0 if case["precision"] == "fp64" else 4.0)
        return {"bytes": b + 8.0 * (n * l + 5 * m), "flops": f + 2.0 * n * l + 12.0 * n * m + 10.0 * n * n}
    if kind == "many":
        n, l, m, q = case["n"], case["steps"], case["m"], case["count"]
        b, f = _gkb_work(n, l, True, 8.0)
        return {"bytes": q * (b + 8.0 * (n * l + 2 * m)), "flops": q * (f + 2.0 * n * l + 12.0 * n * m + 10.0 * n * n)}
    if kind == "batch":
        tot = [_gkb_work(n, case["steps"], False, 4.0) for n in _batch_sizes(case)]
        lift = sum(_batch_sizes(case)) * case["steps"]
        return {"bytes": sum(b for b, _ in tot) + 8.0 * lift, "flops": sum(f for _, f in tot) + 2.0 * lift}
    if kind == "fullsvd":
        n = case["n"]
        return {"bytes": 8.0 * n * n + 16.0 * n, "flops": 8.0 / 3.0 * n**3}
    if kind == "evaluate":
        n, m = case["n"], case["m"]
        return {"bytes": 8.0 * (4 * n + 4 * m), "flops": 12.0 * n * m}
    n, l, m = case["n"], case["steps"], case["m"]
    nt = sum(e for e in ELLS if e <= l) * 81
    return {"bytes": 8.0 * (n * l + 3 * n + m * l), "flops": 10.0 * n * m + 2.0 * n * m * l + 2.0 * nt * m}


# --------------------------------------------------------------------------
# the same results in 64 bits with torch
# --------------------------------------------------------------------------

def _dist2(P1, P2):
    d = P1[:, None, 0] - P2[None, :, 0]
    s = d * d
    for a in (1, 2):
        d = P1[:, None, a] - P2[None, :, a]
        s += d * d
    return s


def _matrix(X, ni, c, k, scale=1.0):
    X = _dev(X)
    n = X.shape[0]
    A = torch.empty((n, n), dtype=torch.float64, device=DEV)
    for i0 in range(0, n, 2048):
        i1 = min(n, i0 + 2048)
        s = _dist2(X[i0:i1], X) + c * c
        q = max(0, min(ni, i1) - i0)
        A[i0 + q:i1] = s[q:].sqrt()
        s = s[:q]
        A[i0:i0 + q] = (c * c + s * (2.0 + k * k * s)) / (s * s.sqrt())
    return A.mul_(scale) if scale != 1.0 else A


def _gkb64(A, f, steps):
    """Golub-Kahan bidiagonalization, classical Gram-Schmidt twice; bases as rows."""
    n = f.numel()
    W = torch.zeros((steps + 1, n), dtype=torch.float64, device=DEV)
    Z = torch.zeros((steps, n), dtype=torch.float64, device=DEV)
    al = torch.zeros(steps, dtype=torch.float64, device=DEV)
    be = torch.zeros(steps + 1, dtype=torch.float64, device=DEV)
    be[0] = f.norm()
    W[0] = f / be[0]
    for j in range(steps):
        r = A.t() @ W[j]
        if j:
            r -= be[j] * Z[j - 1]
            for _ in range(2):
                r = r - Z[:j].t() @ (Z[:j] @ r)
        al[j] = r.norm()
        Z[j] = r / al[j]
        p = A @ Z[j] - al[j] * W[j]
        for _ in range(2):
            p = p - W[:j + 1].t() @ (W[:j + 1] @ p)
        be[j + 1] = p.norm()
        W[j + 1] = p / be[j + 1]
    return W, Z, al, be


def _project64(al, be):
    """SVD of the projected matrix: sigma, f~ = U^T beta_1 e_1 (l + 1 values), V."""
    al, be = al.cpu().numpy(), be.cpu().numpy()
    l = al.size
    C = np.zeros((l + 1, l))
    C[np.arange(l), np.arange(l)] = al
    C[np.arange(1, l + 1), np.arange(l)] = be[1:]
    U, s, Vt = np.linalg.svd(C, full_matrices=True)
    return s, be[0] * U[0], Vt.T


def _grid(s1):
    return s1 * 10.0 ** np.linspace(-16.0, 0.0, 321)


def _hkt64(al, be, Z, rule="gcv"):
    s, ft, V = _project64(al, be)
    l = s.size
    lam = _grid(s[0])[:, None]
    q = lam**2 / (s**2 + lam**2)
    g = s * ft[:l] / (s**2 + lam**2)
    rho2 = np.sum((q * ft[:l]) ** 2, 1) + ft[l] ** 2
    gcv = rho2 / (1.0 + q.sum(1)) ** 2
    if rule == "gcv":
        i = int(np.argmin(gcv))
    elif rule == "lcurve":
        x, y, h = 0.5 * np.log(rho2), 0.5 * np.log(np.sum(g * g, 1)), 0.05
        x1, y1 = (x[2:] - x[:-2]) / (2 * h), (y[2:] - y[:-2]) / (2 * h)
        x2, y2 = (x[2:] - 2 * x[1:-1] + x[:-2]) / h**2, (y[2:] - 2 * y[1:-1] + y[:-2]) / h**2
        sp = x1 * x1 + y1 * y1
        kap = np.where(sp >= 1e-8, (x1 * y2 - x2 * y1) / np.maximum(sp, 1e-8) ** 1.5, -np.inf)
        i = int(np.argmax(kap)) + 1
    else:
        i = -1
        lam1 = s[0] * 10.0 ** RULES[rule][1]
        c = s * ft[:l] / (s**2 + lam1**2)
        rho = math.sqrt(np.sum((lam1**2 / (s**2 + lam1**2) * ft[:l]) ** 2) + ft[l] ** 2)
        return _dev(V @ c) @ Z, i, lam1, s[0], float(np.linalg.norm(c)), rho, gcv
    return (_dev(V @ g[i]) @ Z, i, float(lam[i, 0]), float(s[0]), float(np.linalg.norm(g[i])),
            float(np.sqrt(rho2[i])), gcv)


def _ine_tsvd64(al, be, Z):
    s, ft, V = _project64(al, be)
    l = s.size
    r = int(np.sum(s > (l + 1) * np.finfo(float).eps * s[0]))
    tail = np.cumsum((ft**2)[::-1])[::-1]
    k = int(np.argmin([tail[j] / (l + 1.0 - j) ** 2 for j in range(1, r + 1)])) + 1
    c = np.where(np.arange(l) < k, ft[:l] / s, 0.0)
    return _dev(V @ c) @ Z, k, float(s[0]), float(np.linalg.norm(c)), float(np.sqrt(tail[k]))


def _lsqr64(al, be, Z):
    a, b = al.cpu().numpy(), be.cpu().numpy()
    l = a.size
    C = np.zeros((l + 1, l))
    C[np.arange(l), np.arange(l)] = a
    C[np.arange(1, l + 1), np.arange(l)] = b[1:]
    ys, rho = [], []
    for k in range(1, l + 1):
        rhs = np.zeros(k + 1)
        rhs[0] = b[0]
        q, r = np.linalg.qr(C[:k + 1, :k], mode="complete")
        h = q.T @ rhs
        ys.append(np.linalg.solve(r[:k], h[:k]))
        rho.append(abs(h[k]))
    gcv = np.array([rho[k - 1] ** 2 / (l + 1.0 - k) ** 2 for k in range(1, l + 1)])
    k = int(np.argmin(gcv)) + 1
    return _dev(ys[k - 1]) @ Z[:k], k, float(np.linalg.norm(ys[k - 1])), float(rho[k - 1]), gcv


def _field64(X, pts, c, coefs, scale=1.0):
    """coefs [q][n] -> u [q][m]"""
    X, pts = _dev(X), _dev(pts)
    out = []
    for t in range(0, pts.shape[0], 2048):
        phi = (_dist2(pts[t:t + 2048], X) + c * c).sqrt_()
        out.append(coefs @ phi.t())
    return torch.cat(out, 1) * scale


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "projected":
        pr, c, k = _projected_problem(case, seed)
        _, Z, a, b = _gkb64(_matrix(pr.X, pr.ni, c, k), _dev(pr.f), case["steps"])
        meth = case["method"]
        if meth in RULES:
            coef, i, lam, s1, eta, rho, gcv = _hkt64(a, b, Z, meth)
            out = {"coef": coef, "index": i, "lam": lam, "sigma1": s1, "eta": eta, "rho": rho}
            if meth == "gcv":
                out["gcv"] = gcv
            return out
        if meth == "ine_tsvd":
            coef, r, _, eta, rho = _ine_tsvd64(a, b, Z)
            return {"coef": coef, "rank": r, "eta": eta, "rho": rho}
        coef, r, eta, rho, gcv = _lsqr64(a, b, Z)
        return {"coef": coef, "rank": r, "eta": eta, "rho": rho, "gcv": gcv}
    if kind == "matvec":
        pr, x1, x2, c, k = _matvec_inputs(case, seed)
        A = _matrix(pr.X, pr.ni, c, k, 1.0 / c if case["form"] == "eps" else 1.0)
        return {"y1": A @ _dev(x1), "y2": A.t() @ _dev(x2)}
    if kind == "solve":
        pr = _solve_problem(case, seed)
        c, k = case["c"], case["k"]
        sc = 1.0 / c if case["form"] == "eps" else 1.0
        W, Z, a, b = _gkb64(_matrix(pr.X, pr.ni, c, k, sc), _dev(pr.f), case["steps"])
        out = {"W": W, "Z": Z, "alpha": a, "beta": b, "steps": case["steps"]}
        if case["method"] == "hkt":
            coef, i, lam, s1, eta, rho, gcv = _hkt64(a, b, Z)
            out.update(gcv=gcv, index=i, lam=lam)
        else:
            coef, r, s1, eta, rho = _ine_tsvd64(a, b, Z)
            out["rank"] = r
        out.update(coef=coef, u=_field64(pr.X, pr.points, c, coef[None], sc)[0], sigma1=s1, eta=eta, rho=rho)
        return out
    if kind == "many":
        n = case["n"]
        out, cs, us, ix, ls = {}, [], [], [], []
        for i, (c, k) in enumerate(_many_params(case)):
            pr = _Problem("cube", n, k, seed, m=case["m"], wave=True)
            W, Z, a, b = _gkb64(_matrix(pr.X, pr.ni, c, k), _dev(pr.f), case["steps"])
            coef, idx, lam, *_ = _hkt64(a, b, Z)
            out.update({f"W{i}": W, f"Z{i}": Z, f"alpha{i}": a, f"beta{i}": b})
            cs.append(coef)
            us.append(_field64(pr.X, pr.points, c, coef[None])[0])
            ix.append(idx)
            ls.append(lam)
        out.update(coef=torch.stack(cs), u=torch.stack(us), index=ix, lam=ls)
        return out
    if kind == "batch":
        Ws, Zs, As, Bs, cs, ls = [], [], [], [], [], []
        for pr, c, k in _batch_problems(case, seed):
            W, Z, a, b = _gkb64(_matrix(pr.X, pr.ni, c, k), _dev(pr.f), case["steps"])
            coef, _, lam, *_ = _hkt64(a, b, Z)
            for lst, v in ((Ws, W), (Zs, Z), (As, a), (Bs, b), (cs, coef)):
                lst.append(v.reshape(-1))
            ls.append(lam)
        return {"W": torch.cat(Ws), "Z": torch.cat(Zs), "alpha": torch.cat(As), "beta": torch.cat(Bs),
                "coef": torch.cat(cs), "lam": np.asarray(ls), "steps": np.full(case["count"], case["steps"])}
    if kind == "fullsvd":
        return _exact_fullsvd(case, seed)
    if kind == "evaluate":
        X, _, pts, coef = _evaluate_inputs(case, seed)
        return {"u": _field64(X, pts, case["c"], _dev(coef)[None], 1.0 / case["c"] if case["form"] == "eps" else 1.0)[0]}
    pr, c, k = _label_problem(case, seed)
    l = case["steps"]
    _, Z, a, b = _gkb64(_matrix(pr.X, pr.ni, c, k), _dev(pr.f), l)
    G = _field64(pr.X, pr.points, c, Z)
    uref = _dev(pr.field(pr.points))
    rows = []
    for e in [e for e in ELLS if e <= l]:
        s, ft, V = _project64(a[:e], b[:e + 1])
        lam = _grid(s[0])[::T_STRIDE, None]
        y = _dev((s * ft[:e] / (s**2 + lam**2)) @ V.T)
        rows.append((y @ G[:e] - uref).abs().max(1).values / uref.abs().max())
    return {"G": G, "err": torch.stack(rows)}


def _exact_fullsvd(case, seed):
    n = case["n"]
    if n > 2000:  # a LAPACK SVD of this size takes too long
        return None
    pr = _Problem("cube", n, case["k"], seed, noise=1e-2)
    U, s, Vt = np.linalg.svd(_matrix(pr.X, pr.ni, case["c"], case["k"]).cpu().numpy())
    fh = U.T @ pr.f
    r = int(np.sum(s > n * np.finfo(float).eps * s[0]))
    perp = np.sum(fh[r:] ** 2)
    if case["method"] == "tikhonov":
        lam = _grid(s[0])[:, None]
        q = lam**2 / (s[:r] ** 2 + lam**2)
        i = int(np.argmin((np.sum((q * fh[:r]) ** 2, 1) + perp) / ((n - r) + q.sum(1)) ** 2))
        l1 = lam[i, 0]
        return {"coef": (s[:r] * fh[:r] / (s[:r] ** 2 + l1**2)) @ Vt[:r], "index": i, "lam": float(l1),
                "sigma1": float(s[0])}
    tail = np.concatenate([np.cumsum((fh[:r] ** 2)[::-1])[::-1], [0.0]]) + perp
    k = int(np.argmin([tail[j] / (n - j) ** 2 for j in range(1, min(r, n - 1) + 1)])) + 1
    return {"coef": (fh[:k] / s[:k]) @ Vt[:k], "rank": k, "sigma1": float(s[0])}


def _exact_train(case, seed):
    p, m, v, x, y = (_dev(a) for a in _train_inputs(case, seed))
    p.requires_grad_(True)
    i = 0
    h = x
    for fi, fo, act in ((20, 128, True), (128, 128, True), (128, 2, False)):
        w, b = p[i:i + fi * fo].reshape(fi, fo), p[i + fi * fo:i + fi * fo + fo]
        i += fi * fo + fo
        h = h @ w + b
        h = torch.nn.functional.gelu(h) if act else h
    (((h - y) ** 2).sum() / (2 * case["batch"])).backward()
    g = p.grad
    m = 0.9 * m + 0.1 * g
    v = 0.999 * v + 0.001 * g * g
    t = TRAIN_T
    step = TRAIN_LR * (m / (1 - 0.9**t)) / ((v / (1 - 0.999**t)).sqrt() + 1e-8)
    return {"p": (p - step).detach(), "m": m, "v": v, "g": g}
