"""One-cluster fits that need more than one launch (8192 coordinates each),
with a zero step as the last of a launch: the next launch starts from what the
earlier one left in global memory alone.  Long one-block kernels on other
streams move the cluster to other SMs from launch to launch; 8 sweeps of 1000
coordinates put the objective on the first pass of the second launch."""
import functools

import numpy as np
import pytest

import oracle
from paper_2204_08183_gb300 import binding

from gpu_util import oracle_X, small_csc, survdata

pytestmark = pytest.mark.gpu
P = 1000
CASES = {"l1": 20.0, "l2": 5.0}     # L1: the last coefficient stays 0; L2: an empty last column


@functools.lru_cache(None)
def _cohort(model, penalty):
    d = small_csc(3000, P, seed=3, density=0.05, n_times=100, competing=0.25 if model == "fg" else 0.0)
    if penalty == "l2":
        d["col_ptr"][-1] = d["col_ptr"][-2]
        d["row_idx"], d["values"] = (d[k][:d["col_ptr"][-1]].copy() for k in ("row_idx", "values"))
    return d


@functools.lru_cache(None)
def _oracle(model, penalty, sweeps):
    d = _cohort(model, penalty)
    return oracle.ccd_fit(model, d["time"], d["status"], oracle_X(d), penalty, CASES[penalty], tol=0.0,
                          max_sweeps=sweeps)


@pytest.mark.parametrize("precision", ["f32c", "f64"])
@pytest.mark.parametrize("penalty", list(CASES))
@pytest.mark.parametrize("model", ["cox", "fg"])
def test_relaunch_after_a_zero_step(lib, model, penalty, precision):
    import torch
    d = dict(_cohort(model, penalty))
    d["values"] = d["values"].astype(np.float64 if precision == "f64" else np.float32)
    sd = survdata(d)
    fit = binding.cox_fit if model == "cox" else binding.fg_fit
    kw = dict(penalty=penalty, lam=CASES[penalty], precision=precision, tol=0.0, max_sweeps=8)
    b0, i0, _ = fit(sd, flags=binding.SURV_FLAG_ONE_COORDINATE, **kw)
    ref = _oracle(model, penalty, 8)
    assert ref["beta"][-1] == 0.0
    streams = [torch.cuda.Stream() for _ in range(8)]
    rng = np.random.default_rng(0)
    f64 = precision == "f64"
    for _ in range(20):
        for other in streams:
            with torch.cuda.stream(other):
                for _ in range(60):
                    torch.cuda._sleep(int(rng.integers(200_000, 3_000_000)))
        b, i, _ = fit(sd, **kw)
        torch.cuda.synchronize()
        for beta, loglik in ((b0, i0["loglik"]), (ref["beta"], ref["loglik"])):
            np.testing.assert_allclose(b, beta, rtol=0, atol=1e-9 if f64 else 1e-5)
            assert i["loglik"] == pytest.approx(loglik, rel=1e-10 if f64 else 1e-6)
        assert b[-1] == 0.0 and i["sweeps"] == 8
