"""Every schedule of a fit, at sizes where the default takes it and with the
schedule that ran asserted: batches of four coordinates (fewer row passes than
coordinates), the kernel pair replayed as a graph, and one cluster (a handful of
launches).  More than 1024 covariates, more than 300,000 subjects (FP32) or
40,000 (FP64) never run on a cluster.  Tolerances of the parity tests."""
import numpy as np
import pytest

import oracle
from paper_2204_08183_gb300 import binding, synth

from gpu_util import oracle_X, small_csc, survdata

pytestmark = pytest.mark.gpu
ONE = binding.SURV_FLAG_ONE_COORDINATE


def _ran(info, p):
    if info["row_passes"] < info["coordinate_passes"]:
        return "batches"
    return "pair" if info["kernel_launches"] >= 2 * p * max(1, info["sweeps"]) else "cluster"


def _cohort(model, layout, n, p, n_times, precision="f32c", **kw):
    if layout == "csc":
        d = small_csc(n, p, seed=n + p, n_times=n_times, competing=0.25 if model == "fg" else 0.0, **kw)
        if d["values"] is not None and precision == "f64":
            d["values"] = d["values"].astype(np.float64)
    else:
        d = synth.cohort_small(n, p, n + p, n_times=n_times, competing_frac=0.25 if model == "fg" else 0.0)
        d["n"], d["p"] = n, p
    return d


def _check(model, d, precision, penalty, lam, sweeps, schedule, flags=0, **kw):
    fit = binding.cox_fit if model == "cox" else binding.fg_fit
    b, i, _ = fit(survdata(d), penalty=penalty, lam=lam, precision=precision, tol=0.0, max_sweeps=sweeps, flags=flags,
                  **kw)
    st = d["status"] if model == "fg" else np.where(d["status"] == 2, 0, d["status"]).astype(np.int8)
    ref = oracle.ccd_fit(model, d["time"], st, oracle_X(d), penalty, lam, tol=0.0, max_sweeps=sweeps)
    f64 = precision == "f64"
    np.testing.assert_allclose(b, ref["beta"], rtol=0, atol=1e-9 if f64 else 1e-5)
    assert i["loglik"] == pytest.approx(ref["loglik"], rel=1e-10 if f64 else 1e-6)
    if penalty == "l1":
        assert np.array_equal(b == 0.0, ref["beta"] == 0.0)
    assert i["sweeps"] == sweeps and _ran(i, d["p"]) == schedule
    return b, i


@pytest.mark.parametrize("binary", [True, False])
@pytest.mark.parametrize("n,p,n_times,density", [(3001, 1031, 40, 0.05), (37, 1030, 6, 0.2), (300_001, 10, 300, 0.05),
                                                  (300_033, 13, 3000, 0.1)])
def test_batches_of_four(lib, n, p, n_times, density, binary):
    d = _cohort("cox", "csc", n, p, n_times, density=density, binary=binary)
    lam = 0.3 * oracle.lambda_max("cox", d["time"], d["status"], oracle_X(d))
    b, i = _check("cox", d, "f32c", "l1", lam, 4, "batches")
    b0, i0 = _check("cox", d, "f32c", "l1", lam, 4, "pair", flags=ONE)
    np.testing.assert_allclose(b, b0, rtol=0, atol=1e-6)
    assert i["coordinate_passes"] == i0["coordinate_passes"] and i["row_passes"] < i0["row_passes"]


@pytest.mark.parametrize("sweeps", [0, 1, 2])
def test_batches_stop_after_few_sweeps(lib, sweeps):
    d = _cohort("cox", "csc", 300_001, 6, 100, density=0.1)
    sd = survdata(d)
    kw = dict(penalty="l1", lam=500.0, tol=0.0, max_sweeps=sweeps)
    b, i, rc = binding.cox_fit(sd, **kw)
    b0, i0, rc0 = binding.cox_fit(sd, flags=ONE, **kw)
    assert i["sweeps"] == i0["sweeps"] == sweeps and rc == rc0
    np.testing.assert_allclose(b, b0, rtol=0, atol=1e-7)
    assert i["loglik"] == pytest.approx(i0["loglik"], rel=1e-9)
    assert sweeps == 0 or _ran(i, 6) == "batches"


@pytest.mark.parametrize("flags", [0, ONE])
def test_graph_kept_in_a_workspace(lib, flags):
    """The second fit replays the kept graph, other strengths and group counts on
    either side of 4096 (the transform's cluster) capture a new one."""
    ws = binding.Workspace()
    few, many = (_cohort("cox", "csc", 300_001, 5, k, density=0.05, binary=True) for k in (900, 6000))
    lam = 0.3 * oracle.lambda_max("cox", few["time"], few["status"], oracle_X(few))
    runs = [(few, lam), (few, lam), (few, 0.3 * lam), (many, lam), (many, lam), (few, lam)]
    data = {id(d): survdata(d) for d in (few, many)}
    for d, strength in runs:
        kw = dict(penalty="l1", lam=strength, tol=0.0, max_sweeps=3, flags=flags)
        b, i, _ = binding.cox_fit(data[id(d)], workspace=ws, **kw)
        b0, i0, _ = binding.cox_fit(data[id(d)], workspace=binding.Workspace(), **kw)
        assert np.array_equal(b, b0) and i["loglik"] == i0["loglik"] and i["n_groups"] == i0["n_groups"]
        if strength == lam and d is few:   # (with every coordinate moving a batch serves one)
            assert _ran(i, 5) == ("pair" if flags else "batches")
        assert _ran(i, 5) != "cluster"
    assert i["n_groups"] <= 4096 < binding.cox_fit(data[id(many)], penalty="l2", lam=1.0, max_sweeps=0, tol=0.0)[1]["n_groups"]


@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("model,layout,precision,n", [
    ("fg", "dense", "f32c", 300_001), ("fg", "csc", "f32c", 300_001), ("cox", "dense", "f32c", 300_001),
    ("fg", "dense", "f64", 40_001), ("cox", "csc", "f64", 40_001), ("cox", "dense", "f64", 40_001)])
def test_kernel_pair(lib, model, layout, precision, n, p):
    kw = dict(density=0.1) if layout == "csc" else {}
    _check(model, _cohort(model, layout, n, p, 700, precision, **kw), precision, "l2", 10.0, 3, "pair")


# words a warp and a CTA's rows fill at 8192; the ends of a cluster (32,768), and
# the rows up to which one is taken
@pytest.mark.parametrize("model,layout,precision,n,K,schedule", [
    ("cox", "csc", "f32c", 8192, 2000, "cluster"), ("cox", "csc", "f32c", 8193, 2000, "cluster"),
    ("fg", "dense", "f64", 16_384, 16_000, "cluster"), ("fg", "dense", "f64", 16_385, 16_000, "cluster"),
    ("cox", "csc", "f64", 40_000, 300, "cluster"), ("cox", "csc", "f64", 40_001, 300, "pair"),
    ("cox", "csc", "f32c", 40_000, 32_767, "cluster"), ("cox", "csc", "f32c", 40_000, 32_768, "cluster"),
    ("cox", "csc", "f32c", 40_000, 32_769, "pair"), ("fg", "csc", "f32c", 40_000, 32_769, "pair"),
    ("cox", "dense", "f32c", 300_000, 20, "cluster"), ("cox", "dense", "f32c", 300_001, 20, "pair")])
def test_edges_of_the_cluster(lib, model, layout, precision, n, K, schedule):
    p = 4
    kw = dict(density=0.02) if layout == "csc" else {}
    d = _cohort(model, layout, n, p, 5, precision, **kw)
    d["time"] = (K - np.arange(n) * K // n).astype(np.int32)
    b, i = _check(model, d, precision, "l2", 2.0, 3, schedule)
    assert i["n_groups"] == K
