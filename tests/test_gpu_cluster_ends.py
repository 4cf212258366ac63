"""One-cluster fits at the group counts where the row pass changes its form
(96 ends in the FP32 mode with 8 words a warp, twice the warps with fewer; one
form in FP64), with the ends spread evenly or
crowded into the latest times; against the oracle and the kernel pair, with
the tolerances of the parity tests."""
import numpy as np
import pytest

import oracle
from paper_2204_08183_gb300 import binding, synth

from gpu_util import oracle_X, small_csc, survdata

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("crowded", [False, True])
@pytest.mark.parametrize("K", [1, 2, 95, 96, 400])
@pytest.mark.parametrize("precision", ["f32c", "f64"])
@pytest.mark.parametrize("model,layout", [("cox", "csc"), ("cox", "dense"), ("fg", "csc"), ("fg", "dense")])
def test_forms_of_the_row_pass(lib, model, layout, precision, K, crowded):
    n, p = 12_007 if precision == "f64" or K == 400 else 58_001, 3
    if layout == "csc":
        d = small_csc(n, p, seed=K, density=0.2, n_times=5, competing=0.25 if model == "fg" else 0.0)
        d["values"] = d["values"].astype(np.float64 if precision == "f64" else np.float32)
    else:
        d = synth.cohort_small(n, p, K, n_times=5, competing_frac=0.25 if model == "fg" else 0.0)
    # crowded: K - 1 groups of one subject at the latest times, the others tied
    t = np.minimum(np.arange(n), K - 1) if crowded else np.arange(n) * K // n
    d["time"] = (K - t).astype(np.int32)
    d["status"][:K] = np.where(np.arange(K) % 3 == 0, 1, d["status"][:K])
    assert len(oracle.tie_groups(d["time"])) == K
    fit = binding.cox_fit if model == "cox" else binding.fg_fit
    kw = dict(penalty="l2", lam=1.0, precision=precision, tol=0.0, max_sweeps=3)
    sd = survdata(d)
    b, i, _ = fit(sd, **kw)
    b0, i0, _ = fit(sd, flags=binding.SURV_FLAG_ONE_COORDINATE, **kw)
    ref = oracle.ccd_fit(model, d["time"], d["status"], oracle_X(d), "l2", 1.0, tol=0.0, max_sweeps=3)
    f64 = precision == "f64"
    for beta, loglik in ((b0, i0["loglik"]), (ref["beta"], ref["loglik"])):
        np.testing.assert_allclose(b, beta, rtol=0, atol=1e-9 if f64 else 1e-5)
        assert i["loglik"] == pytest.approx(loglik, rel=1e-10 if f64 else 1e-6)
