"""The choice of the schedule sees how group ends crowd: the same rows, columns
and number of groups, spread evenly or crowded into the latest times as those of
exponential times are, which costs whoever walks them one after another (the
cluster below 96 ends or a tile of rows a warp; batches).  Every choice agrees
with the one-coordinate schedule."""
import numpy as np
import pytest

from paper_2204_08183_gb300 import binding

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,layout,n,K,density,even_cluster,crowded_cluster", [
    ("fg", "dense", 30_000, 365, 1.0, True, False), ("cox", "dense", 30_000, 365, 1.0, True, False),
    ("cox", "csc", 200_000, 3000, 0.5, False, True), ("cox", "csc", 100_000, 2000, 0.2, True, True)])
def test_evenly_spread_and_crowded_ends(lib, model, layout, n, K, density, even_cluster, crowded_cluster):
    p = 12
    rng = np.random.default_rng(n + K)
    even = np.arange(n) * K // n
    crowded = np.minimum(np.arange(n), (K * (1.0 - np.exp(-np.arange(n) / (K / 4.6)))).astype(np.int64))
    crowded = np.minimum(crowded, K - 1)
    if layout == "dense":
        X = dict(X=dev(rng.standard_normal((p, n)).astype(np.float32)))
    else:
        cols = [np.flatnonzero(rng.random(n) < density).astype(np.int32) for _ in range(p)]
        ptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
        X = dict(col_ptr=dev(ptr), row_idx=dev(np.concatenate(cols)), n=n, p=p)
    status = dev(rng.choice([0, 1, 2] if model == "fg" else [0, 1], n).astype(np.int8))
    fit = binding.cox_fit if model == "cox" else binding.fg_fit
    kw = dict(penalty="l2", lam=2.0, tol=0.0, max_sweeps=2)
    for group, one_cluster in ((even, even_cluster), (crowded, crowded_cluster)):
        sd = binding.SurvData(dev((K - group).astype(np.int32)), status, **X)
        b, i, _ = fit(sd, **kw)
        b0, i0, _ = fit(sd, flags=binding.SURV_FLAG_ONE_COORDINATE, **kw)
        np.testing.assert_allclose(b, b0, rtol=0, atol=1e-5)
        assert i["loglik"] == pytest.approx(i0["loglik"], rel=1e-6)
        assert (i["kernel_launches"] < 2 * p) == one_cluster, i["n_groups"]
