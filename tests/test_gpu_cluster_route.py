"""Which default fits run on one cluster: the choice follows rows, group ends
and stored entries together.  A fit on the cluster takes a handful of launches,
one on the kernel pair or in batches at least two a row pass; both give the
result of the one-coordinate schedule."""
import numpy as np
import pytest

from paper_2204_08183_gb300 import binding

from gpu_util import dev

pytestmark = pytest.mark.gpu


def _cohort(model, layout, n, p, K, density, seed=5):
    rng = np.random.default_rng(seed)
    y = rng.exponential(size=n)
    t = np.clip(np.ceil(K * y / np.quantile(y, 0.99)), 1, K).astype(np.int32)
    time = np.sort(t)[::-1].copy()
    status = rng.choice([0, 1, 2] if model == "fg" else [0, 1], n).astype(np.int8)
    if layout == "dense":
        return binding.SurvData(dev(time), dev(status), X=dev(rng.standard_normal((p, n)).astype(np.float32)))
    cols = [np.flatnonzero(rng.random(n) < density).astype(np.int32) for _ in range(p)]
    ptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
    return binding.SurvData(dev(time), dev(status), col_ptr=dev(ptr), row_idx=dev(np.concatenate(cols)), n=n, p=p)


@pytest.mark.parametrize("model,layout,n,K,density,one_cluster", [
    ("cox", "csc", 50_000, 3650, 0.05, True), ("cox", "csc", 300_000, 1000, 0.5, False),
    ("cox", "csc", 150_000, 40_000, 0.05, False), ("cox", "csc", 20_000, 40_000, 0.01, True),
    ("fg", "csc", 100_000, 1000, 0.02, True), ("fg", "csc", 200_000, 1000, 0.5, False),
    ("cox", "dense", 30_000, 365, 1.0, False), ("cox", "dense", 8_000, 3650, 1.0, True),
    ("fg", "dense", 100_000, 10_000, 1.0, False), ("fg", "dense", 10_000, 1000, 1.0, True)])
def test_route_of_a_fit(lib, model, layout, n, K, density, one_cluster):
    p = 12
    sd = _cohort(model, layout, n, p, K, density)
    fit = binding.cox_fit if model == "cox" else binding.fg_fit
    kw = dict(penalty="l2", lam=2.0, tol=0.0, max_sweeps=2)
    b, i, _ = fit(sd, **kw)
    b0, i0, _ = fit(sd, flags=binding.SURV_FLAG_ONE_COORDINATE, **kw)
    np.testing.assert_allclose(b, b0, rtol=0, atol=1e-5)
    assert i["loglik"] == pytest.approx(i0["loglik"], rel=1e-6)
    assert (i["kernel_launches"] < 2 * p) == one_cluster
