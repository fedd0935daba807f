"""Timed cases of the KRR engine: what its users have it do, through the public
binding (``KRR``, ``KRRBatch``).

A case names one *kind* of call and its sizes: ``n`` training patients, ``m``
SNPs, ``p`` phenotypes, ``n_test`` held-out patients, ``tile`` (the context's
tile edge), ``lam`` (the regulariser) and the kind's options.

* ``fit``       Build, Factor, Solve and Predict on new genotypes: the paper's
                whole driver (Alg. 1).  Options: ``kernel`` ("gaussian" or
                "ibs"), ``cohorts`` (structured genotypes, where most factor
                tiles are stored in E4M3) and ``nc`` confounder columns.
* ``refit``     Factor with a regulariser and Solve on a kernel that is kept:
                one step of a scan over lambda.
* ``solve``     a new phenotype set against a kept factor (Sec. IV-C: the
                factors are reused for several phenotypes).
* ``predict``   new patients against a kept model.
* ``gradient``  a fit and the gradient of the held-out loss with respect to
                log gamma and log lambda: one step of a hyperparameter search.
* ``ridge``     ridge regression on genotypes and confounders (Sec. IV-A).
* ``batch``     cross-validation: cohorts of uneven size x lambdas, one run of
                a captured batch.

All of them run in the mixed-precision mode, the default; the plain FP32 mode
is the comparison path of the tests and the benchmark.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2409_01712_gb300 import KRR, KRRBatch, inputs

BATCH_LAMBDAS = (1e-3, 1e-2, 1e-1, 1.0)
#: the cohorts are cross-validation folds of a study: N ~ U[1024, 16384]
BATCH_SPREAD = (1.0, 0.71, 0.48, 0.33, 0.19, 0.0)
EXACT_MAX_N = 20480  # 64-bit factorisations past this take more than a few seconds


def _fit(name, n, m, p, n_test, tile, kernel="gaussian", cohorts=0, nc=0):
    return {"name": name, "kind": "fit", "n": n, "m": m, "p": p, "n_test": n_test, "tile": tile, "lam": 0.1,
            "kernel": kernel, "cohorts": cohorts, "nc": nc}


def _plain(name, kind, n, m, p, n_test, tile, **more):
    return dict({"name": name, "kind": kind, "n": n, "m": m, "p": p, "n_test": n_test, "tile": tile, "lam": 0.1},
                **more)


def listed():
    return [
        # a pilot study, one phenotype: short launches and dependency chains
        _fit("fit_pilot", 2048, 512, 1, 512, 256),
        # a study of a few thousand patients at the default tile edge; every
        # size ragged (the last tile mostly padding)
        _fit("fit_ragged", 5000, 700, 2, 300, 1024),
        # age, sex and principal components beside the genotypes
        _fit("fit_confounders", 10000, 4000, 5, 1000, 1024, nc=10),
        # the precision workload: a mid-size cohort, ten phenotypes
        _fit("fit_mid", 32768, 8192, 10, 4096, 1024),
        # the same sizes from eight subpopulations: the FP8-dominant mosaic
        _fit("fit_cohorts", 32768, 8192, 10, 4096, 1024, cohorts=8),
        # the largest study: the headline workload's SNPs and phenotypes on the
        # patients of which three fits (three resident states) share one GPU
        _fit("fit_biobank", 98304, 16384, 20, 4096, 1024),
        # one lambda of a regularisation path on a kept kernel
        _plain("refit_lambda", "refit", 16384, 8192, 8, 0, 1024),
        # further phenotypes of a study whose factor is kept
        _plain("solve_phenotypes", "solve", 32768, 8192, 10, 0, 1024),
        # risk scores of a clinic's new patients from a kept model
        _plain("predict_patients", "predict", 32768, 8192, 10, 64, 1024),
        # the differentiation workload's sizes, on structured genotypes: one
        # hyperparameter step (with gamma = 1/M on unstructured genotypes the
        # gradient is a small difference of large sums)
        _plain("gradient_step", "gradient", 16384, 8192, 8, 4096, 1024, cohorts=8),
        # the linear model of Sec. IV-A on the same engine
        _plain("ridge", "ridge", 16384, 4096, 4, 1000, 512, lam=10.0, nc=5),
        # cross-validation: six cohorts of uneven size x four lambdas
        _plain("batch_cv", "batch", 16384, 4096, 4, 512, 512, n_lo=1024, cohorts=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit", "fit", "fit", "refit", "solve", "predict", "gradient", "ridge", "batch"])
    p = rng.randint(1, 20)
    opt = rng.choice(["plain", "plain", "ibs", "cohorts", "confounders"]) if kind == "fit" else "plain"
    n = {"fit": _log_int(rng, 1300, 65536), "refit": _log_int(rng, 2048, 49152), "solve": _log_int(rng, 2048, 49152),
         "predict": _log_int(rng, 2048, 65536)}.get(kind) or _log_int(rng, 1024, 20000)
    # patients per SNP as in the listed studies (at most 8, at most 2 for the
    # linear IBS kernel, whose rank is bounded by 2 M)
    m = _log_int(rng, max(300, n // (2 if opt == "ibs" else 8)), max(16384, n // 2))
    tile = 256 if n < 3000 else rng.choice([512, 1024, 1024])
    if kind == "fit":
        c = _fit("", n, m, p, _log_int(rng, 64, 4096), tile, kernel="ibs" if opt == "ibs" else "gaussian",
                 cohorts=8 if opt == "cohorts" else 0, nc=rng.randint(1, 16) if opt == "confounders" else 0)
    elif kind in ("refit", "solve"):
        c = _plain("", kind, n, m, p, 0, tile, lam=rng.choice([0.01, 0.1, 1.0]))
    elif kind == "predict":
        c = _plain("", kind, n, m, p, _log_int(rng, 1, 2048), 1024)
    elif kind == "gradient":
        c = _plain("", kind, n, m, min(p, 16), _log_int(rng, 200, 4096), 256 if n < 3000 else 1024, cohorts=8)
    elif kind == "ridge":  # more patients than columns
        f = _log_int(rng, 700, 8192)
        c = _plain("", kind, _log_int(rng, 2 * f, 40000), f, rng.randint(1, 8), _log_int(rng, 64, 2048),
                   256 if f < 1024 else 512, lam=10.0, nc=rng.randint(0, 16))
    else:
        c = _plain("", kind, _log_int(rng, 4096, 16384), _log_int(rng, 512, 4096), rng.randint(1, 8), 256, 512,
                   n_lo=1024, cohorts=rng.randint(2, 6))
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _structured(case):
    return case["kind"] in ("fit", "gradient") and case.get("cohorts", 0) > 0


def _gamma(case):
    """1/M, and 8/M for the structured cohorts (within-cohort K near 0.02)."""
    return (8.0 if _structured(case) else 1.0) / case["m"]


def _data(case, seed, dev):
    """G, Y, T, Yt and, with confounders, C and Ct, on ``dev``."""
    n, m, p, nc = case["n"], case["m"], case["p"], case.get("nc", 0)
    n_test = max(1, case["n_test"])
    seed = 16 * int(seed) + 2409017120
    if _structured(case):
        d = inputs.structured_problem(n, m, p, n_test, seed=seed, populations=case["cohorts"], fst=0.3, device=dev)
    else:
        d = inputs.problem(n, m, p, n_test, seed=seed, device=dev)
    d = {k: d[k] for k in ("G", "Y", "T", "Yt")}
    if nc:
        # covariates carrying about a tenth of the mean genotype distance
        scale = 2.0 if case["kind"] == "ridge" else math.sqrt(0.1 * 0.74 * m / (2 * nc))
        c = inputs.confounders(n + n_test, nc, seed=seed, scale=scale).to(dev)
        d["C"], d["Ct"] = c[:n].contiguous(), c[n:].contiguous()
    else:
        d["C"] = d["Ct"] = None
    return d


def _cohort_sizes(case):
    """Uneven cohorts between n_lo and n, the largest first."""
    k = case["cohorts"]
    at = [BATCH_SPREAD[round(i * (len(BATCH_SPREAD) - 1) / max(1, k - 1))] for i in range(k)]
    return [case["n_lo"] + int(a * (case["n"] - case["n_lo"])) for a in at]


def _cohorts(case, seed, dev):
    return [inputs.problem(n, case["m"], case["p"], case["n_test"], seed=16 * int(seed) + 2409017120 + 100003 * i,
                           device=dev) for i, n in enumerate(_cohort_sizes(case))]


def prepare(case, seed):
    dev = _device()
    kind = case["kind"]
    state = {"case": case, "gamma": _gamma(case)}
    if kind == "batch":
        problems = [{"G": c["G"], "Y": c["Y"], "T": c["T"], "gamma": state["gamma"], "lam": lam}
                    for c in _cohorts(case, seed, dev) for lam in BATCH_LAMBDAS]
        state["batch"] = KRRBatch(problems, ir_iters=3, autotune=0, tile=case["tile"])
        return state
    state.update(_data(case, seed, dev))
    model = KRR(tile=case["tile"], kernel=case.get("kernel", "gaussian"))
    state["model"] = model
    if kind in ("refit", "solve", "predict"):
        model.build_kernel(state["G"], state["gamma"])
    if kind in ("solve", "predict"):
        model.factor(case["lam"])
    if kind == "predict":
        state["A"], _ = model.solve(state["Y"])
    return state


# ---------------------------------------------------------------------------
# One pass.
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        state["batch"].run()
        return {"A": state["batch"].A, "Yt": state["batch"].Yt}
    model, lam = state["model"], case["lam"]
    if kind == "fit":
        model.build_kernel(state["G"], state["gamma"], conf=state["C"])
        model.factor(lam)
        a, _ = model.solve(state["Y"])
        return {"A": a, "Yt": model.predict(state["T"], a, conf=state["Ct"])}
    if kind == "refit":
        model.factor(lam)
        a, _ = model.solve(state["Y"])
        return {"A": a}
    if kind == "solve":
        a, _ = model.solve(state["Y"])
        return {"A": a}
    if kind == "predict":
        return {"Yt": model.predict(state["T"], state["A"])}
    if kind == "gradient":
        model.build_kernel(state["G"], state["gamma"])
        model.factor(lam)
        a, _ = model.solve(state["Y"])
        loss, dlog_gamma, dlog_lambda = model.grad_hyper(state["T"], state["Yt"], a)
        return {"A": a, "loss": loss, "dlog_gamma": dlog_gamma, "dlog_lambda": dlog_lambda}
    model.rr_build(state["G"], conf=state["C"])
    rhs = model.rr_rhs(state["Y"])
    model.factor(lam)
    beta, _ = model.solve(rhs)
    return {"rhs": rhs, "beta": beta, "Yt": model.rr_predict(state["T"], beta, conf=state["Ct"])}


# ---------------------------------------------------------------------------
# What a pass cannot do without.
# ---------------------------------------------------------------------------
def _build_work(n, m, nc=0):
    """One triangle of the distances."""
    return {"bytes": float(n) * m + 4.0 * n * nc, "flops": float(n) * n * (m + nc)}


def _factor_flops(n):
    return float(n) ** 3 / 3.0


def _solve_work(n, p):
    """One pair of substitutions, Y in and A out."""
    return {"bytes": 8.0 * n * p, "flops": 2.0 * n * n * p}


def _predict_work(n, m, p, n_test, nc=0):
    """T in, Yt out (the model's own operands are counted where they are kept)."""
    return {"bytes": float(n_test) * (m + 4.0 * nc) + 4.0 * n_test * p,
            "flops": 2.0 * n_test * n * (m + nc + p)}


def _sum(*parts):
    return {k: sum(q[k] for q in parts) for k in ("bytes", "flops")}


def work(case):
    n, m, p, nc, kind = case["n"], case["m"], case["p"], case.get("nc", 0), case["kind"]
    enc = 2 * m if case.get("kernel") == "ibs" else m
    factor = {"bytes": 0.0, "flops": _factor_flops(n)}
    if kind == "fit":
        return _sum(_build_work(n, enc, nc), factor, _solve_work(n, p), _predict_work(n, enc, p, case["n_test"], nc))
    if kind == "refit":  # the kept FP32 kernel tiles are an input
        return _sum({"bytes": 2.0 * n * n, "flops": 0.0}, factor, _solve_work(n, p))
    if kind == "solve":  # the kept factor (two bytes an entry) is an input
        return _sum({"bytes": 1.0 * n * n, "flops": 0.0}, _solve_work(n, p))
    if kind == "predict":  # the kept training genotypes and weights are inputs
        return _sum({"bytes": float(n) * m + 4.0 * n * p, "flops": 0.0}, _predict_work(n, m, p, case["n_test"]))
    if kind == "gradient":
        # the held-out kernel once forward and once transposed, one more solve,
        # and the two contractions over it and over one triangle of K
        nt = case["n_test"]
        return _sum(_build_work(n, m), factor, _solve_work(n, p), _predict_work(n, m, p, nt), _solve_work(n, p),
                    {"bytes": 0.0, "flops": 4.0 * nt * n * p + 2.0 * n * n * p})
    if kind == "ridge":
        f = m + nc
        return _sum({"bytes": float(n) * (m + 4.0 * nc), "flops": float(n) * f * f + 2.0 * n * f * p},
                    {"bytes": 0.0, "flops": _factor_flops(f)}, _solve_work(f, p),
                    {"bytes": float(case["n_test"]) * (m + 4.0 * nc + 4.0 * p),
                     "flops": 2.0 * case["n_test"] * f * p})
    parts = []
    for nn in _cohort_sizes(case):
        parts.append(_build_work(nn, m))
        for _ in BATCH_LAMBDAS:
            parts += [{"bytes": 0.0, "flops": _factor_flops(nn)}, _solve_work(nn, p),
                      _predict_work(nn, m, p, case["n_test"])]
    return _sum(*parts)


# ---------------------------------------------------------------------------
# The same values in 64 bits, from the definitions.
# ---------------------------------------------------------------------------
def _distances(a, b, ibs):
    """Squared Euclidean (IBS: L1) distances of genotype rows; exact integers."""
    if ibs:  # |a - b| summed: two indicators per genotype
        a = torch.cat([(a >= 1), (a >= 2)], dim=1).to(torch.float32)
        b = torch.cat([(b >= 1), (b >= 2)], dim=1).to(torch.float32)
    else:
        a, b = a.to(torch.float32), b.to(torch.float32)
    # sums below 2^24: exact in FP32 products with FP32 accumulation
    s = (a @ b.T).to(torch.float64)
    na, nb = a.to(torch.float64).square().sum(1), b.to(torch.float64).square().sum(1)
    return na[:, None] + nb[None, :] - 2.0 * s


def _kernel(case, gamma, a, b, ca=None, cb=None):
    ibs = case.get("kernel") == "ibs"
    d = _distances(a, b, ibs)
    if ibs:
        return (2.0 * case["m"] - d) / case["m"]
    if ca is not None:
        for q in range(ca.shape[1]):
            d += (ca[:, q].double()[:, None] - cb[:, q].double()[None, :]).square()
    return d.mul_(-gamma).exp_()


def _cholesky(k, lam):
    k.diagonal().add_(lam)
    return torch.linalg.cholesky(k)


def _fit64(case, gamma, lam, d):
    chol = _cholesky(_kernel(case, gamma, d["G"], d["G"], d.get("C"), d.get("C")), lam)
    return chol, torch.cholesky_solve(d["Y"].double(), chol)


def _predict64(case, gamma, d, a):
    return _kernel(case, gamma, d["T"], d["G"], d.get("Ct"), d.get("C")) @ a


def _np(x):
    return x.cpu().numpy() if isinstance(x, torch.Tensor) else np.float64(x)


def exact(case, seed):
    """What ``run`` returns, in 64 bits; None past EXACT_MAX_N rows."""
    kind, gamma, dev = case["kind"], _gamma(case), _device()
    tf32 = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = False  # the integer products are exact in FP32 only
    try:
        if kind == "batch":
            out = {"A": [], "Yt": []}
            for c in _cohorts(case, seed, dev):
                for lam in BATCH_LAMBDAS:
                    if c["G"].shape[0] > EXACT_MAX_N // 2:
                        out["A"].append(None)
                        out["Yt"].append(None)
                        continue
                    _, a = _fit64(case, gamma, lam, c)
                    out["A"].append(_np(a))
                    out["Yt"].append(_np(_predict64(case, gamma, c, a)))
            return out
        if case["n"] > EXACT_MAX_N and kind != "ridge":
            return None
        d = _data(case, seed, dev)
        lam = case["lam"]
        if kind == "ridge":
            x, t = d["G"].double(), d["T"].double()
            if d["C"] is not None:
                x, t = torch.cat([x, d["C"].double()], 1), torch.cat([t, d["Ct"].double()], 1)
            rhs = x.T @ d["Y"].double()
            beta = torch.cholesky_solve(rhs, _cholesky(x.T @ x, lam))
            return {"rhs": _np(rhs), "beta": _np(beta), "Yt": _np(t @ beta)}
        chol, a = _fit64(case, gamma, lam, d)
        if kind in ("refit", "solve"):
            return {"A": _np(a)}
        if kind == "fit":
            return {"A": _np(a), "Yt": _np(_predict64(case, gamma, d, a))}
        if kind == "predict":  # Yt of the weights the engine itself keeps is compared, not the weights
            return {"Yt": _np(_predict64(case, gamma, d, a))}
        kt = _kernel(case, gamma, d["T"], d["G"])
        diff = kt @ a - d["Yt"].double()
        gp = 2.0 * diff / diff.numel()
        z = torch.cholesky_solve(kt.T @ gp, chol)
        del chol
        dist = _distances(d["G"], d["G"], False)
        dk = (dist * torch.exp(-gamma * dist) * (z @ a.T)).sum()
        del dist
        dist = _distances(d["T"], d["G"], False)
        dt = (dist * kt * (gp @ a.T)).sum()
        return {"A": _np(a), "loss": _np(diff.square().mean()), "dlog_gamma": _np(gamma * (dk - dt)),
                "dlog_lambda": _np(-lam * (z * a).sum())}
    finally:
        torch.backends.cuda.matmul.allow_tf32 = tf32
