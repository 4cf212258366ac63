"""L1 fits of sparse Cox data: where few coordinates move, batches of four a row
pass; where most do, one cluster.  The start decides: gradients at beta = 0
beyond their strengths, or the nonzeros of a warm beta.  Either way the result
is the one-coordinate schedule's."""
import numpy as np
import pytest

from paper_2204_08183_gb300 import binding

from gpu_util import dev

pytestmark = pytest.mark.gpu
P = 40


@pytest.fixture(scope="module")
def cohort():
    rng = np.random.default_rng(11)
    n = 100_003
    y = rng.exponential(size=n)
    time = np.sort(np.clip(np.ceil(3650 * y / np.quantile(y, 0.99)), 1, 3650).astype(np.int32))[::-1].copy()
    status = rng.integers(0, 2, n).astype(np.int8)
    cols = [np.flatnonzero(rng.random(n) < 0.05).astype(np.int32) for _ in range(P)]
    ptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
    return binding.SurvData(dev(time), dev(status), col_ptr=dev(ptr), row_idx=dev(np.concatenate(cols)), n=n, p=P)


@pytest.mark.parametrize("strength,start,factors,one_cluster", [
    (1.1, None, None, False), (0.7, None, None, False), (0.001, None, None, True), (1.1, None, "none", True),
    (0.7, "few", None, False), (0.001, "all", None, True)])
def test_schedule_follows_the_moving_share(lib, cohort, strength, start, factors, one_cluster):
    lam = strength * binding.cox_lambda_max(cohort)
    beta = np.zeros(P)
    if start:
        beta[:3 if start == "few" else P] = 0.01
    pf = np.zeros(P) if factors == "none" else None
    kw = dict(penalty="l1", lam=lam, penalty_factor=pf, tol=0.0, max_sweeps=3)
    for ws in (None, binding.Workspace()):
        b, i, _ = binding.cox_fit(cohort, beta=beta.copy(), workspace=ws, **kw)
        b0, i0, _ = binding.cox_fit(cohort, beta=beta.copy(), workspace=ws, flags=binding.SURV_FLAG_ONE_COORDINATE, **kw)
        np.testing.assert_allclose(b, b0, rtol=0, atol=1e-5)
        assert np.array_equal(b == 0.0, b0 == 0.0) and i["sweeps"] == i0["sweeps"] == 3
        assert i["loglik"] == pytest.approx(i0["loglik"], rel=1e-6)
        assert (i["row_passes"] == i["coordinate_passes"]) == one_cluster
        assert (i["kernel_launches"] < 2 * P) == one_cluster
