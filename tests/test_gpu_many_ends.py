"""The row pass of warps that hold many group ends (kernel pair, more groups
than twice its warps): windows of 32 ends, tiles and rounds with none, one
and many ends, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2204_08183_gb300 import binding, synth

from gpu_util import oracle_X, small_csc, survdata

pytestmark = pytest.mark.gpu
PAIR = binding.SURV_FLAG_ONE_COORDINATE


def _times(kind, n, rng):
    if kind == "unique":
        return np.arange(n, 0, -1)
    # half of the subjects alone in their group, half in a few large groups
    t = np.where(rng.random(n) < 0.5, rng.choice(10 * n, n, replace=False) + 100, rng.integers(1, 6, n) * (2 * n))
    return np.sort(t)[::-1]


# 4864 warps on 152 SMs: two or more groups a warp from 9728 groups on
@pytest.mark.parametrize("precision", ["f32c", "f64"])
@pytest.mark.parametrize("layout,density", [("csc", 0.01), ("csc", 0.4), ("dense", 1.0)])
@pytest.mark.parametrize("n,kind", [(20_011, "unique"), (160_003, "mixed")])
def test_many_ends(lib, n, kind, layout, density, precision):
    rng = np.random.default_rng(n)
    if layout == "csc":
        d = small_csc(n, 3, seed=n, density=density, n_times=5)
    else:
        d = synth.cohort_small(n, 3, n, n_times=5)
    d["time"] = np.ascontiguousarray(_times(kind, n, rng).astype(np.int32))
    assert len(oracle.tie_groups(d["time"])) >= 9728
    kw = dict(penalty="l2", lam=1.0, precision=precision, tol=0.0, max_sweeps=2, flags=PAIR)
    b, i, _ = binding.cox_fit(survdata(d), **kw)
    ref = oracle.ccd_fit("cox", d["time"], d["status"], oracle_X(d), "l2", 1.0, tol=0.0, max_sweeps=2)
    f64 = precision == "f64"
    np.testing.assert_allclose(b, ref["beta"], rtol=0, atol=1e-9 if f64 else 1e-5)
    assert i["loglik"] == pytest.approx(ref["loglik"], rel=1e-10 if f64 else 1e-6)


# few rows a warp: the same form although the groups are fewer than the warps
@pytest.mark.parametrize("precision", ["f32c", "f64"])
@pytest.mark.parametrize("layout", ["csc", "dense"])
@pytest.mark.parametrize("model", ["cox", "fg"])
@pytest.mark.parametrize("n", [2, 31, 4099, 160_003])
def test_few_rows_a_warp(lib, n, model, layout, precision):
    competing = 0.25 if model == "fg" else 0.0
    if layout == "csc":
        d = small_csc(n, 2, seed=n + 1, density=0.3, n_times=200, competing=competing)
    else:
        d = synth.cohort_small(n, 2, n + 1, n_times=200, competing_frac=competing)
    d["status"][-1] = 1
    fit = binding.cox_fit if model == "cox" else binding.fg_fit
    kw = dict(penalty="l2", lam=1.0, precision=precision, tol=0.0, max_sweeps=2, flags=PAIR)
    b, i, _ = fit(survdata(d), **kw)
    ref = oracle.ccd_fit(model, d["time"], d["status"], oracle_X(d), "l2", 1.0, tol=0.0, max_sweeps=2)
    f64 = precision == "f64"
    np.testing.assert_allclose(b, ref["beta"], rtol=0, atol=1e-9 if f64 else 1e-5)
    assert i["loglik"] == pytest.approx(ref["loglik"], rel=1e-10 if f64 else 1e-6, abs=1e-12 if f64 else 1e-6)
