"""The one-cluster schedule of small cohorts against the kernel pair it
stands in for (SURV_FLAG_ONE_COORDINATE) and the oracle: every model, layout
and precision, at sizes around a word, a warp's rows, a CTA's rows and one
subject per group."""
import numpy as np
import pytest

import oracle
from paper_2204_08183_gb300 import binding, synth

from gpu_util import oracle_X, small_csc, survdata

pytestmark = pytest.mark.gpu
PAIR = binding.SURV_FLAG_ONE_COORDINATE


def _cohort(model, layout, n, p, n_times):
    if layout == "csc":
        return small_csc(n, p, seed=n + p, density=0.2, n_times=n_times, competing=0.25 if model == "fg" else 0.0)
    d = synth.cohort_small(n, p, n + p, n_times=n_times, competing_frac=0.25 if model == "fg" else 0.0)
    d["n"], d["p"] = n, p
    return d


# 16 CTAs of up to 16 row warps: 513 words is the first size with two words a
# warp; 16,385 the first past one word for every warp
@pytest.mark.parametrize("precision", ["f32c", "f64"])
@pytest.mark.parametrize("layout", ["csc", "dense"])
@pytest.mark.parametrize("model", ["cox", "fg"])
@pytest.mark.parametrize("n,p,n_times", [(33, 1, 5), (515, 3, 600), (8193, 4, 40), (16_417, 5, 20_000)])
def test_cluster_fit(lib, model, layout, precision, n, p, n_times):
    d = _cohort(model, layout, n, p, n_times)
    fit = binding.cox_fit if model == "cox" else binding.fg_fit
    sd = survdata(d)
    kw = dict(penalty="l2", lam=1.0, precision=precision, tol=0.0, max_sweeps=4)
    b, i, _ = fit(sd, **kw)
    b0, i0, _ = fit(sd, flags=PAIR, **kw)
    ref = oracle.ccd_fit(model, d["time"], d["status"], oracle_X(d), "l2", 1.0, tol=0.0, max_sweeps=4)
    tol = 1e-9 if precision == "f64" else 1e-5     # the bars of the parity tests
    np.testing.assert_allclose(b, ref["beta"], rtol=0, atol=tol)
    np.testing.assert_allclose(b, b0, rtol=0, atol=tol)
    assert i["sweeps"] == i0["sweeps"] == 4 and i["coordinate_passes"] == i0["coordinate_passes"]
    assert i["loglik"] == pytest.approx(ref["loglik"], rel=1e-10 if precision == "f64" else 1e-6)


def test_cluster_launches_in_turn(lib):
    """More sweeps than one launch runs (8192 coordinates): the state passes
    from launch to launch."""
    d = _cohort("cox", "dense", 2000, 900, 300)
    sd = survdata(d)
    kw = dict(penalty="l2", lam=5.0, precision="f64", tol=0.0, max_sweeps=20)
    b, i, _ = binding.cox_fit(sd, **kw)
    b0, i0, _ = binding.cox_fit(sd, flags=PAIR, **kw)
    np.testing.assert_allclose(b, b0, rtol=0, atol=1e-9)
    assert i["sweeps"] == i0["sweeps"] == 20 and i["eta_updates"] == i0["eta_updates"]


def test_cluster_warm_start_and_l1(lib):
    d = small_csc(5000, 7, seed=9, density=0.2, n_times=200, binary=True)
    sd = survdata(d)
    lam = 0.2 * oracle.lambda_max("cox", d["time"], d["status"], oracle_X(d))
    start = np.linspace(-0.3, 0.3, 7)
    b, i, _ = binding.cox_fit(sd, beta=start.copy(), penalty="l1", lam=lam, tol=0.0, max_sweeps=6)
    ref = oracle.ccd_fit("cox", d["time"], d["status"], oracle_X(d), "l1", lam, beta0=start, tol=0.0, max_sweeps=6)
    np.testing.assert_allclose(b, ref["beta"], rtol=0, atol=1e-5)
    assert np.array_equal(b == 0.0, ref["beta"] == 0.0)
