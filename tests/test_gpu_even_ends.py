"""Kernel-pair Fine-Gray fits with two or more group ends a warp on average,
spread evenly (the plain row pass) or crowded into the latest times (the
many-ends form); against the oracle, with the tolerances of the parity tests."""
import numpy as np
import pytest

import oracle
from paper_2204_08183_gb300 import binding, synth

from gpu_util import oracle_X, small_csc, survdata

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("crowded", [False, True])
@pytest.mark.parametrize("layout,n", [("csc", 100_003), ("dense", 60_001), ("dense", 330_007)])
def test_even_and_crowded_ends(lib, layout, n, crowded):
    p, K = 2, 10_000
    if layout == "csc":
        d = small_csc(n, p, seed=n, density=0.1, n_times=5, competing=0.25)
    else:
        d = synth.cohort_small(n, p, n, n_times=5, competing_frac=0.25)
    t = np.minimum(np.arange(n), K - 1) if crowded else np.arange(n) * K // n
    d["time"] = (K - t).astype(np.int32)
    assert len(oracle.tie_groups(d["time"])) == K
    kw = dict(penalty="l2", lam=1.0, tol=0.0, max_sweeps=2)
    b, i, _ = binding.fg_fit(survdata(d), flags=binding.SURV_FLAG_ONE_COORDINATE, **kw)
    ref = oracle.ccd_fit("fg", d["time"], d["status"], oracle_X(d), "l2", 1.0, tol=0.0, max_sweeps=2)
    np.testing.assert_allclose(b, ref["beta"], rtol=0, atol=1e-5)
    assert i["loglik"] == pytest.approx(ref["loglik"], rel=1e-6)
