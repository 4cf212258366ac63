"""The transform of sparse Cox fits (FP32, one coordinate a pass) around the
group count where its blocks grow; against the oracle with the tolerances of
the parity tests."""
import numpy as np
import pytest

import oracle
from paper_2204_08183_gb300 import binding

from gpu_util import oracle_X, small_csc, survdata

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [8191, 8192, 8193, 9729, 20_000])
def test_block_sizes(lib, K):
    n = 30_011
    d = small_csc(n, 3, seed=K, density=0.2, n_times=5, binary=True)
    d["time"] = np.sort(np.arange(n) % K + 1)[::-1].astype(np.int32).copy()
    assert len(oracle.tie_groups(d["time"])) == K
    kw = dict(penalty="l2", lam=1.0, tol=0.0, max_sweeps=2)
    b, i, _ = binding.cox_fit(survdata(d), flags=binding.SURV_FLAG_ONE_COORDINATE, **kw)
    ref = oracle.ccd_fit("cox", d["time"], d["status"], oracle_X(d), "l2", 1.0, tol=0.0, max_sweeps=2)
    np.testing.assert_allclose(b, ref["beta"], rtol=0, atol=1e-5)
    assert i["loglik"] == pytest.approx(ref["loglik"], rel=1e-6)
