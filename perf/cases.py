"""The calls that a user of the library makes, with inputs to time them on.

Each case is one call (or the few calls that belong together) through
``paper_2204_08183_gb300.binding``: a penalised Cox or Fine-Gray fit, a
cross-validated path, one forward and backward pass of the differentiable
likelihood, one evaluation of l, l' and l'', the arrangement of raw survival
times, or the largest useful L1 strength.  Inputs are drawn on the GPU from a
seed, in the shapes of the synthetic cohorts of ``synth.py``: covariates
N(0, 1) or sparse, exponential event times with rate exp(x beta), censoring,
times on an integer grid so that ties occur.

``exact`` restates each result in 64 bits with plain torch and numpy.
"""
import math

import numpy as np
import torch

from paper_2204_08183_gb300 import binding

DEV = "cuda"
TOL = 1e-8
MAX_SWEEPS = 1000


def listed():
    return [
        # A study of 10,000 subjects with ten covariates, everything in
        # double precision: the smallest fit that is run in earnest.
        {"name": "cox_dense_f64_10k", "kind": "fit", "model": "cox", "layout": "dense", "dtype": "f64",
         "precision": "f64", "n": 10_000, "p": 10, "grid": 365, "censored": 0.30, "penalty": "l2", "lam": 1.0},
        # The large-sample regression the library is for: 10^7 subjects, 100
        # indicator covariates at 5 %, an L1 penalty, times in days.
        {"name": "cox_csc_10m", "kind": "fit", "model": "cox", "layout": "csc", "dtype": "f32", "values": "ones",
         "density": 0.05, "precision": "f32c", "n": 10_000_000, "p": 100, "grid": 3650, "censored": 0.50,
         "penalty": "l1", "lam": 1000.0},
        # Sparse measurements rather than indicators, times recorded finely
        # (hardly any ties), a size that divides by nothing.
        {"name": "cox_csc_real_333k", "kind": "fit", "model": "cox", "layout": "csc", "dtype": "f32",
         "values": "real", "density": 0.02, "precision": "f32c", "n": 333_331, "p": 80, "grid": 5_000_000,
         "censored": 0.30, "penalty": "l2", "lam": 1.0},
        # Dense covariates kept in bfloat16 (embeddings, scores), L1.
        {"name": "cox_dense_bf16_500k", "kind": "fit", "model": "cox", "layout": "dense", "dtype": "bf16",
         "precision": "f32c", "n": 500_009, "p": 24, "grid": 3650, "censored": 0.50, "penalty": "l1", "lam": 50.0},
        # Competing risks at scale: 5 x 10^6 subjects, 50 dense covariates.
        {"name": "fg_dense_5m", "kind": "fit", "model": "fg", "layout": "dense", "dtype": "f32",
         "precision": "f32c", "n": 5_000_000, "p": 50, "grid": 1000, "censored": 0.40, "penalty": "l2", "lam": 10.0},
        # Competing risks with sparse indicators, given without values.
        {"name": "fg_csc_200k", "kind": "fit", "model": "fg", "layout": "csc", "dtype": "f32", "values": "none",
         "density": 0.05, "precision": "f32c", "n": 200_003, "p": 40, "grid": 1000, "censored": 0.40,
         "penalty": "l2", "lam": 10.0},
        # Choosing the L1 strength by 10-fold cross-validation over 20
        # strengths: 200 fits in one call.
        {"name": "cv_csc_1m", "kind": "cv", "model": "cox", "layout": "csc", "dtype": "f32", "values": "ones",
         "density": 0.01, "precision": "f32c", "n": 1_000_000, "p": 500, "grid": 3650, "censored": 0.40,
         "folds": 10, "lambdas": 20},
        # A training step of 64 linear predictors on a large cohort.
        {"name": "nll_4m_p256_c64", "kind": "nll", "n": 1 << 22, "p": 256, "cols": 64, "grid": 5000,
         "censored": 0.30},
        # The same step in a small study: sizes that fit no tile.
        {"name": "nll_20k_p50_c5", "kind": "nll", "n": 20_011, "p": 50, "cols": 5, "grid": 365, "censored": 0.30},
        # l, l' and l'' of one coordinate: what a caller's own optimiser asks for.
        {"name": "score_csc_100k", "kind": "score", "model": "cox", "layout": "csc", "dtype": "f32",
         "values": "ones", "density": 0.05, "precision": "f32c", "n": 100_003, "p": 100, "grid": 3650,
         "censored": 0.50, "noalloc": False},
        # Raw records into the library's order, and their tie groups with the
        # censoring survival.
        {"name": "arrange_10m", "kind": "arrange", "n": 10_000_000, "grid": 3650, "censored": 0.50},
        # Where an L1 path starts.
        {"name": "lambda_max_1m", "kind": "lambda_max", "model": "cox", "layout": "csc", "dtype": "f32",
         "values": "ones", "density": 0.01, "n": 1_000_000, "p": 500, "grid": 3650, "censored": 0.40},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _matrix(rng, n_lo, n_hi, cells, p_lo, p_hi, allow_bf16=True):
    """n, p, layout, type and (sparse) density of X; `cells` bounds the stored entries."""
    n = _log_uniform(rng, n_lo, n_hi)
    layout = rng.choice(["csc", "dense"])
    density = 1.0 if layout == "dense" else round(math.exp(rng.uniform(math.log(0.005), math.log(0.08))), 4)
    p = _log_uniform(rng, p_lo, max(p_lo, min(p_hi, int(cells / (n * density)))))
    c = {"layout": layout, "n": n, "p": p}
    if layout == "csc":
        c["density"] = density
        c["values"] = rng.choice(["ones", "none", "real"])
        c["dtype"] = "f32"
    else:
        c["dtype"] = rng.choice(["f32", "bf16"] if allow_bf16 else ["f32"])
    return c


def draw(rng):
    kind = rng.choice(["fit", "fit", "fit", "cv", "nll", "nll", "score", "arrange", "lambda_max"])
    grid = rng.choice([365, 1000, 3650, 100_000])
    censored = round(rng.uniform(0.25, 0.55), 3)
    if kind == "nll":
        n = _log_uniform(rng, 2_000, 1 << 22)
        return {"kind": kind, "n": n, "p": _log_uniform(rng, 8, 256), "cols": _log_uniform(rng, 1, 64),
                "grid": rng.choice([365, 5000]), "censored": censored}
    if kind == "arrange":
        return {"kind": kind, "n": _log_uniform(rng, 10_000, 10_000_000), "grid": grid, "censored": censored}
    if kind == "fit":
        c = _matrix(rng, 5_000, 5_000_000, 5e7, 5, 100)
        c["model"] = rng.choice(["cox", "cox", "fg"])
        c["precision"] = "f32c"
        if c["n"] * c["p"] * c.get("density", 1.0) < 2e6 and rng.random() < 0.5:
            c["precision"] = "f64"
            c["dtype"] = "f64"
        c["penalty"] = rng.choice(["l1", "l2"])
        c["lam"] = round(1e-4 * c["n"], 3) if c["penalty"] == "l1" else rng.choice([1.0, 10.0])
    elif kind == "cv":
        c = _matrix(rng, 10_000, 500_000, 2e6, 10, 200, allow_bf16=False)
        c.update(model="cox", precision="f32c", folds=rng.choice([5, 10]), lambdas=rng.randint(5, 20))
    elif kind == "score":
        c = _matrix(rng, 10_000, 2_000_000, 2e7, 5, 100)
        c["model"] = rng.choice(["cox", "fg"])
        c["precision"] = "f32c"
        c["noalloc"] = c["layout"] == "csc" and c["n"] <= 200_000 and rng.random() < 0.5
    else:
        c = _matrix(rng, 10_000, 2_000_000, 2e7, 10, 500)
        c["model"] = "cox"
    c.update(kind=kind, grid=grid, censored=censored)
    return c


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _times(eta1, eta2, case, g):
    """Integer times (not yet arranged) and status codes for the linear
    predictors of the event and, with competing risks, of the competing one."""
    n = eta1.shape[0]

    def expo():
        return torch.empty(n, device=DEV, dtype=torch.float32).exponential_(generator=g)

    if eta2 is None:
        t, u = expo() / torch.exp(eta1), torch.rand(n, device=DEV, generator=g)
        lo, hi = 0.0, 64.0 * float(t.mean())
        for _ in range(30):  # uniform censoring at the wanted share
            mid = 0.5 * (lo + hi)
            if float((mid * u < t).float().mean()) > case["censored"]:
                lo = mid
            else:
                hi = mid
        c = 0.5 * (lo + hi) * u
        y, status = torch.minimum(t, c), (t <= c).to(torch.int8)
    else:  # event : competing : censored as 0.35 : 0.25 : the censored share's odds
        t1, t2 = expo() / (0.35 * torch.exp(eta1)), expo() / (0.25 * torch.exp(eta2))
        c = expo() / (0.60 * case["censored"] / (1.0 - case["censored"]))
        y = torch.minimum(torch.minimum(t1, t2), c)
        status = torch.where(c <= torch.minimum(t1, t2), 0, torch.where(t1 <= t2, 1, 2)).to(torch.int8)
    q = torch.kthvalue(y, max(1, int(0.99 * n))).values
    time = torch.clamp(torch.ceil(case["grid"] * y.double() / q.double()), 1, case["grid"]).to(torch.int32)
    return time, status


_DTYPE = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16}


def _cohort(case, seed):
    """time and status in decreasing time order, X (dense, stored by column:
    shape (p, n)) or CSC arrays, and the coefficients that drew the times."""
    g = _generator(seed)
    n, p = case["n"], case["p"]
    fg = case["model"] == "fg"
    k = min(10, p)
    b1 = torch.zeros(p, device=DEV)
    b2 = torch.zeros(p, device=DEV)
    true = torch.randperm(p, device=DEV, generator=g)[:k]
    b1[true] = 0.3 * torch.randn(k, device=DEV, generator=g)
    b2[true.flip(0)] = 0.3 * torch.randn(k, device=DEV, generator=g)
    out = {}
    if case["layout"] == "dense":
        X = torch.randn((p, n), device=DEV, generator=g)
        if case["dtype"] == "bf16":
            X = X.bfloat16().float()
        time, status = _times(b1 @ X, b2 @ X if fg else None, case, g)
        perm = torch.sort(time, descending=True, stable=True).indices
        out["X"] = torch.stack([X[j][perm].to(_DTYPE[case["dtype"]]) for j in range(p)])
    else:
        real = case["values"] == "real"
        eta1, eta2 = torch.zeros(n, device=DEV), torch.zeros(n, device=DEV)
        cols = []
        for j in range(p):
            rows = (torch.rand(n, device=DEV, generator=g) < case["density"]).nonzero().flatten()
            if rows.numel() == 0:
                rows = torch.zeros(1, device=DEV, dtype=torch.int64)
            vals = torch.randn(rows.numel(), device=DEV, generator=g) if real else None
            cols.append((rows, vals))
            if j in set(true.tolist()):
                x = vals if real else torch.ones(rows.numel(), device=DEV)
                eta1[rows] += b1[j] * x
                eta2[rows] += b2[j] * x
        time, status = _times(eta1, eta2 if fg else None, case, g)
        perm = torch.sort(time, descending=True, stable=True).indices
        inv = torch.empty_like(perm)
        inv[perm] = torch.arange(n, device=DEV)
        ptr, ri, va = [0], [], []
        for rows, vals in cols:
            r, o = torch.sort(inv[rows])
            ri.append(r.to(torch.int32))
            if real:
                va.append(vals[o])
            ptr.append(ptr[-1] + rows.numel())
        out["col_ptr"] = torch.tensor(ptr, dtype=torch.int64, device=DEV)
        out["row_idx"] = torch.cat(ri)
        out["values"] = None
        if real:
            out["values"] = torch.cat(va).to(_DTYPE[case["dtype"]])
        elif case["values"] == "ones":
            out["values"] = torch.ones(ptr[-1], device=DEV, dtype=_DTYPE[case["dtype"]])
    out["time"], out["status"] = time[perm].contiguous(), status[perm].contiguous()
    out["beta"] = b1.double()
    return out


def _survdata(case, d):
    if case["layout"] == "dense":
        return binding.SurvData(d["time"], d["status"], X=d["X"])
    return binding.SurvData(d["time"], d["status"], col_ptr=d["col_ptr"], row_idx=d["row_idx"], values=d["values"],
                            n=case["n"], p=case["p"])


def _folds(case, seed):
    """Uneven folds: sizes evenly spaced from 0.8 to 1.2 of n / folds, at random."""
    n, k = case["n"], case["folds"]
    w = np.linspace(0.8, 1.2, k)
    edge = torch.tensor(np.floor(np.cumsum(w / w.sum()) * n).astype(np.int64)[:-1], device=DEV)
    g = _generator(seed + 7919)
    rank = torch.randperm(n, device=DEV, generator=g)
    return torch.searchsorted(edge, rank, right=True).to(torch.int8)


def _lambdas(case):
    """Strengths of a path, from about the largest useful one down by 10^3."""
    if case["layout"] == "csc":
        scale = 0.1 * case["n"] * case["density"]
    else:
        scale = 0.1 * case["n"]
    return scale * np.logspace(0.0, -3.0, case["lambdas"])


def _nll_inputs(case, seed):
    g = _generator(seed)
    n, p, c = case["n"], case["p"], case["cols"]
    X = torch.empty((n, p), device=DEV, dtype=torch.bfloat16)
    for i in range(0, n, 1 << 20):  # by parts: the float32 draw is twice X
        m = min(1 << 20, n - i)
        X[i:i + m] = torch.randn((m, p), device=DEV, generator=g)
    B = 0.05 * torch.randn((p, c), device=DEV, generator=g)
    time = torch.randint(1, case["grid"] + 1, (n,), device=DEV, generator=g, dtype=torch.int32)
    time = torch.sort(time, descending=True).values.contiguous()
    status = (torch.rand(n, device=DEV, generator=g) >= case["censored"]).to(torch.int8)
    return X, B, time, status


def _raw_times(case, seed):
    g = _generator(seed)
    return _times(torch.zeros(case["n"], device=DEV), None, case, g)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "nll":
        X, B, time, status = _nll_inputs(case, seed)
        return {"case": case, "X": X, "B": B.requires_grad_(True), "time": time, "status": status}
    if kind == "arrange":
        time, status = _raw_times(case, seed)
        return {"case": case, "time": time, "status": status}
    d = _cohort(case, seed)
    s = {"case": case, "data": _survdata(case, d)}
    if kind != "lambda_max":
        s["workspace"] = binding.Workspace()
    if kind == "cv":
        s["folds"], s["lambdas"] = _folds(case, seed), _lambdas(case)
    if kind == "score":
        s["beta"], s["j"] = d["beta"].cpu().numpy(), case["p"] // 2
    return s


# --------------------------------------------------------------------- run
def _coefficients(case, beta):
    # the coefficients in the precision that the fit's sums were asked for
    return beta if case["precision"] == "f64" else beta.astype(np.float32)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "fit":
        fit = binding.cox_fit if case["model"] == "cox" else binding.fg_fit
        beta, info, _ = fit(state["data"], penalty=case["penalty"], lam=case["lam"], tol=TOL, max_sweeps=MAX_SWEEPS,
                            precision=case["precision"], workspace=state["workspace"])
        return {"beta": _coefficients(case, beta), "loglik": info["loglik"], "objective": info["objective"]}
    if kind == "cv":
        r = binding.cox_cv_path(state["data"], state["folds"], case["folds"], state["lambdas"], penalty="l1",
                                tol=TOL, max_sweeps=MAX_SWEEPS, precision=case["precision"],
                                workspace=state["workspace"])
        return {"beta": _coefficients(case, r["beta"]), "heldout": r["heldout"], "cv_mean": r["cv_mean"],
                "best": r["info"]["best_lambda"]}
    if kind == "nll":
        nll = binding.cox_nll(state["B"], state["X"], state["time"], state["status"])
        (grad,) = torch.autograd.grad(nll.sum(), state["B"])
        return {"nll": nll.detach(), "grad": grad}
    if kind == "score":
        if case["noalloc"]:
            l, g, h = binding.loglik_grad_hess_noalloc(state["data"], case["model"], state["beta"], state["j"],
                                                       precision=case["precision"])
        else:
            l, g, h = binding.loglik_grad_hess(state["data"], case["model"], state["beta"], state["j"],
                                               precision=case["precision"], workspace=state["workspace"])
        return {"loglik": l, "grad": g, "hess": h}
    if kind == "arrange":
        perm = binding.surv_sort_desc(state["time"])
        at = perm.long()
        time, status = state["time"][at], state["status"][at]
        gend, dk, gk = binding.surv_groups(time, status)
        return {"perm": perm, "gend": gend, "dk": dk, "Gk": gk}
    return {"lambda_max": binding.cox_lambda_max(state["data"])}


# -------------------------------------------------------------------- work
def work(case):
    """Each input read once, each result written once; the operations of one
    evaluation of every coordinate."""
    n = case["n"]
    if case["kind"] == "nll":
        p, c = case["p"], case["cols"]
        return {"bytes": 2 * n * p + 5 * n + 8 * p * c + 8 * c, "flops": 4 * n * p * c}
    if case["kind"] == "arrange":
        return {"bytes": 4 * n + n + 4 * n + 16 * min(n, case["grid"]), "flops": n}
    p = case["p"]
    if case["layout"] == "dense":
        entries = n * p
        x = entries * {"f32": 4, "f64": 8, "bf16": 2}[case["dtype"]]
    else:
        entries = int(n * p * case["density"])
        x = entries * (4 + (0 if case["values"] == "none" else 8 if case["dtype"] == "f64" else 4)) + 8 * (p + 1)
    fits = case["folds"] * case["lambdas"] if case["kind"] == "cv" else 1
    if case["kind"] == "score":  # beta X needs the columns of ten coefficients, the sums one more
        entries, x = entries * 11 // max(11, p), x * 11 // max(11, p)
    return {"bytes": x + 5 * n + (n if case["kind"] == "cv" else 0) + 8 * p * fits, "flops": 4 * entries * fits}


# ------------------------------------------------------------------- exact
def _group_ends(time):
    n = time.shape[0]
    last = torch.ones(n, dtype=torch.bool, device=time.device)
    last[:-1] = time[1:] != time[:-1]
    return last.nonzero().flatten()


def _per_group(flag, gend):
    c = torch.cumsum(flag.double(), 0)[gend]
    return torch.diff(c, prepend=c.new_zeros(1))


def _survival_of_censoring(status, gend):
    """Kaplan-Meier G(t_k): factors 1 - c / n multiplied from the smallest time upward."""
    ck = _per_group(status == 0, gend).cpu().numpy()
    f = 1.0 - ck / (gend.cpu().numpy().astype(np.float64) + 1.0)
    return np.cumprod(f[::-1])[::-1].copy()


def _newton(beta, grad, hess, penalty, lam):
    """Newton step on l plus the penalty, one entry a fit (torch, float64)."""
    h = -hess
    ok = h > 0
    hs = torch.where(ok, h, torch.ones_like(h))
    if penalty == "l2":
        step = (grad - lam * beta) / (hs + lam)
    else:
        at0 = torch.where(grad > lam, (grad - lam) / hs, torch.where(grad < -lam, (grad + lam) / hs, grad * 0))
        s = torch.sign(beta)
        moved = (grad - lam * s) / hs
        moved = torch.where((beta + moved) * s > 0, moved, -beta)
        step = torch.where(beta == 0, at0, moved)
    return torch.where(ok, step, torch.zeros_like(step))


class _Column:
    """Column j of X in 64 bits: its rows (None: all of them) and values."""

    def __init__(self, case, d):
        self.case, self.d = case, d
        if case["layout"] == "csc":
            self.ptr = d["col_ptr"].tolist()

    def __call__(self, j):
        d = self.d
        if self.case["layout"] == "dense":
            return None, d["X"][j].double()
        a, b = self.ptr[j], self.ptr[j + 1]
        rows = d["row_idx"][a:b].long()
        return rows, (torch.ones(b - a, dtype=torch.float64, device=DEV) if d["values"] is None
                      else d["values"][a:b].double())


class _Model:
    """Sums over risk sets of `fits` Cox fits at once (keep[f] is 0 for the
    subjects that fit f leaves out), or of one Fine-Gray fit."""

    def __init__(self, case, d, keep=None):
        self.case, self.col = case, _Column(case, d)
        self.fg = case["model"] == "fg"
        n = case["n"]
        self.gend = _group_ends(d["time"])
        self.keep = torch.ones((1, 1), dtype=torch.float64, device=DEV) if keep is None else keep
        event = (d["status"] == 1).double()[None, :] * self.keep
        fits = event.shape[0]
        c = torch.cumsum(event, 1)[:, self.gend]
        self.dk = torch.diff(c, prepend=c.new_zeros((fits, 1)), dim=1)
        self.dtx = torch.stack([(event if r is None else event[:, r]) @ x for r, x in map(self.col, range(case["p"]))], 1)
        del event
        if self.fg:
            self.gk = torch.tensor(_survival_of_censoring(d["status"], self.gend), device=DEV)
            size = torch.diff(self.gend, prepend=self.gend.new_full((1,), -1))
            self.w = torch.repeat_interleave(1.0 / self.gk, size) * (d["status"] == 2)
        self.eta = torch.zeros((fits, n), dtype=torch.float64, device=DEV)
        self.e = torch.exp(self.eta) * self.keep
        self.den = self._at_ends(None, self.e)

    def _at_ends(self, rows, v):
        """Risk-set sums at every group's end of v, given on `rows` (None: all)."""
        at = self.gend + 1 if rows is None else torch.searchsorted(rows, self.gend, right=True)

        def prefix(u):
            c = torch.cumsum(u, 1)
            return torch.cat([c.new_zeros((c.shape[0], 1)), c], 1)

        c = prefix(v)
        s = c[:, at]
        if self.fg:  # competing events stay, weighted, after their time
            c = prefix(v * (self.w if rows is None else self.w[rows]))
            s = s + self.gk * (c[:, -1:] - c[:, at])
        return s

    def derivatives(self, j):
        rows, x = self.col(j)
        a = (self.e if rows is None else self.e[:, rows]) * x
        some = self.dk > 0
        den = torch.where(some, self.den, torch.ones_like(self.den))
        g = self._at_ends(rows, a) / den
        h = self._at_ends(rows, a * x) / den
        zero = torch.zeros_like(g)
        grad = self.dtx[:, j] - torch.where(some, self.dk * g, zero).sum(1)
        hess = -torch.where(some, self.dk * (h - g * g), zero).sum(1)
        return grad, hess

    def log_den(self):
        some = self.dk > 0
        return torch.where(some, self.dk * torch.log(torch.where(some, self.den, torch.ones_like(self.den))),
                           torch.zeros_like(self.dk)).sum(1)

    def move(self, j, step):
        if not bool((step != 0).any()):
            return
        rows, x = self.col(j)
        if rows is None:
            self.eta += step[:, None] * x
            self.e = torch.exp(self.eta) * self.keep
            self.den = self._at_ends(None, self.e)
        else:
            eta = self.eta[:, rows] + step[:, None] * x
            keep = self.keep if self.keep.shape[1] == 1 else self.keep[:, rows]
            e = torch.exp(eta) * keep
            self.den += self._at_ends(rows, e - self.e[:, rows])
            self.eta[:, rows], self.e[:, rows] = eta, e


def _fit_exact(m, penalty, lam):
    """Cyclic coordinate descent with trust regions, every fit of `m` by its
    own stopping rule; lam: one strength a fit."""
    fits, p = m.dtx.shape
    beta = torch.zeros((fits, p), dtype=torch.float64, device=DEV)
    width = torch.ones_like(beta)
    running = torch.ones(fits, dtype=torch.bool, device=DEV)
    f_prev = loglik = objective = None
    for sweep in range(MAX_SWEEPS + 1):
        ll = (m.dtx * beta).sum(1) - m.log_den()
        pen = (beta.abs().sum(1) if penalty == "l1" else 0.5 * (beta * beta).sum(1)) * lam
        f = ll - pen
        loglik = ll if loglik is None else torch.where(running, ll, loglik)
        objective = f if objective is None else torch.where(running, f, objective)
        if sweep:
            running &= ~((f - f_prev).abs() / f.abs() < TOL)
        if sweep >= MAX_SWEEPS or not bool(running.any()):
            break
        f_prev = f
        for j in range(p):
            grad, hess = m.derivatives(j)
            step = _newton(beta[:, j], grad, hess, penalty, lam)
            step = torch.sign(step) * torch.minimum(step.abs(), width[:, j])
            step = torch.where(running, step, torch.zeros_like(step))
            beta[:, j] += step
            width[:, j] = torch.where(running, torch.maximum(2 * step.abs(), width[:, j] / 2), width[:, j])
            m.move(j, step)
    return beta, loglik, objective


def _heldout_exact(m, d, inside):
    """Each fit's log partial likelihood of its own fold, on the fold's risk sets."""
    event = (d["status"] == 1).double()[None, :] * inside
    lin = (event * m.eta).sum(1)
    c = torch.cumsum(event, 1)[:, m.gend]
    dk = torch.diff(c, prepend=c.new_zeros((c.shape[0], 1)), dim=1)
    del event
    den = torch.cumsum(torch.exp(m.eta) * inside, 1)[:, m.gend]
    return lin - torch.where(dk > 0, dk * torch.log(torch.where(dk > 0, den, torch.ones_like(den))),
                             torch.zeros_like(dk)).sum(1)


def _nll_exact(case, seed):
    X, B, time, status = _nll_inputs(case, seed)
    gend = _group_ends(time)
    dk = _per_group(status == 1, gend)
    delta = (status == 1).double()
    parts = 1 << 19
    eta = torch.cat([X[i:i + parts].double() @ B.double() for i in range(0, case["n"], parts)])
    e = torch.exp(eta)
    den = torch.cumsum(e, 0)[gend]
    nll = -(delta @ eta) + dk @ torch.log(den)
    lam = torch.flip(torch.cumsum(torch.flip(dk[:, None] / den, [0]), 0), [0])
    size = torch.diff(gend, prepend=gend.new_full((1,), -1))
    e *= torch.repeat_interleave(lam, size, dim=0)
    e -= delta[:, None]
    grad = sum(X[i:i + parts].double().T @ e[i:i + parts] for i in range(0, case["n"], parts))
    return {"nll": nll, "grad": grad}


def exact(case, seed):
    kind = case["kind"]
    if kind == "nll":
        return _nll_exact(case, seed)
    if kind == "arrange":
        time, status = _raw_times(case, seed)
        time, perm = torch.sort(time, descending=True, stable=True)
        status = status[perm]
        gend = _group_ends(time)
        return {"perm": perm.to(torch.int32), "gend": gend.to(torch.int32),
                "dk": _per_group(status == 1, gend).to(torch.int32), "Gk": _survival_of_censoring(status, gend)}
    d = _cohort(case, seed)
    if kind == "lambda_max":
        m = _Model(case, d)
        return {"lambda_max": max(abs(float(m.derivatives(j)[0])) for j in range(case["p"]))}
    if kind == "score":
        m = _Model(case, d)
        for j in range(case["p"]):
            m.move(j, d["beta"][j:j + 1])
        grad, hess = m.derivatives(case["p"] // 2)
        return {"loglik": float((m.dtx @ d["beta"]) - m.log_den()), "grad": float(grad), "hess": float(hess)}
    if kind == "fit":
        m = _Model(case, d)
        beta, ll, f = _fit_exact(m, case["penalty"], torch.tensor([case["lam"]], dtype=torch.float64, device=DEV))
        return {"beta": beta[0], "loglik": float(ll), "objective": float(f)}
    # the cross-validated path: every (strength, fold) fit beside the others
    fold = _folds(case, seed)
    lam = torch.tensor(_lambdas(case), device=DEV)
    inside = torch.stack([(fold == k) for k in range(case["folds"])]).double().repeat(case["lambdas"], 1)
    m = _Model(case, d, keep=1.0 - inside)
    beta, _, _ = _fit_exact(m, "l1", lam.repeat_interleave(case["folds"]))
    held = _heldout_exact(m, d, inside).reshape(case["lambdas"], case["folds"])
    mean = held.mean(1)
    return {"beta": beta.reshape(case["lambdas"], case["folds"], case["p"]), "heldout": held, "cv_mean": mean,
            "best": int(torch.argmax(mean))}
