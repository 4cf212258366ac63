"""The transforms at the group counts where their form changes: one cluster of
at most 16 CTAs (up to 4096 ends of one coordinate, or 16,384 items of a
batch), the ticket beyond; against the oracle, with the tolerances of the
many-ends tests."""
import numpy as np
import pytest

import oracle
from paper_2204_08183_gb300 import binding, synth

from gpu_util import oracle_X, small_csc, survdata

pytestmark = pytest.mark.gpu
FLAGS = {"one": binding.SURV_FLAG_ONE_COORDINATE, "b4": binding.SURV_FLAG_NO_PDL, "b8": binding.SURV_FLAG_SPEC_B8}


@pytest.mark.parametrize("schedule,model,precision", [("one", "cox", "f32c"), ("one", "fg", "f64"),
                                                      ("b4", "cox", "f32c"), ("b8", "cox", "f32c")])
@pytest.mark.parametrize("K", [1, 128, 129, 2048, 2049, 4096, 4097])
def test_group_counts(lib, K, schedule, model, precision):
    n, p = 30_011, 3
    if model == "cox":
        d = small_csc(n, p, seed=K, density=0.2, n_times=5, binary=True)
    else:
        d = synth.cohort_small(n, p, K, n_times=5, competing_frac=0.25)
    d["time"] = np.sort(np.arange(n) % K + 1)[::-1].astype(np.int32).copy()
    assert len(oracle.tie_groups(d["time"])) == K
    fit = binding.cox_fit if model == "cox" else binding.fg_fit
    kw = dict(penalty="l2", lam=1.0, precision=precision, tol=0.0, max_sweeps=2, flags=FLAGS[schedule])
    b, i, _ = fit(survdata(d), **kw)
    ref = oracle.ccd_fit(model, d["time"], d["status"], oracle_X(d), "l2", 1.0, tol=0.0, max_sweeps=2)
    f64 = precision == "f64"
    np.testing.assert_allclose(b, ref["beta"], rtol=0, atol=1e-9 if f64 else 1e-5)
    assert i["loglik"] == pytest.approx(ref["loglik"], rel=1e-10 if f64 else 1e-6)
