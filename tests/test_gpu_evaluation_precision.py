"""l' and l'' of one coordinate in the FP32 mode, where every sum over subjects
is exact (beta = 0, integer covariates), against rational arithmetic: what is
left is the arithmetic at the group ends, which is FP64.

Tolerance of l'': H and G^2 are near x^2 <= 1025^2 and carry at most 4
roundings of 2^-53 each, 4.7e-10 in all per event, against a variance of at
least 0.2 per event: 2.4e-9, and the sums (float-float, 1e-14) add nothing."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2204_08183_gb300 import binding

from gpu_util import dev

pytestmark = pytest.mark.gpu


def _exact(model, time, status, x):
    """(l', l'') at beta = 0; with competing events but no censoring every weight is 1."""
    n = len(time)
    ends = [i for i in range(n) if i == n - 1 or time[i] != time[i + 1]]
    g, h, a = Fraction(int(x[status == 1].sum())), Fraction(0), 0
    for e in ends:
        d = int((status[a:e + 1] == 1).sum())
        risk = x[:e + 1]
        later = x[e + 1:][status[e + 1:] == 2] if model == "fg" else x[:0]
        s = [Fraction(int((risk ** m).sum() + (later ** m).sum())) for m in range(3)]
        g -= d * s[1] / s[0]
        h -= d * (s[2] / s[0] - (s[1] / s[0]) ** 2)
        a = e + 1
    return float(g), float(h)


@pytest.mark.parametrize("layout", ["csc", "dense"])
@pytest.mark.parametrize("model", ["cox", "fg"])
@pytest.mark.parametrize("n,K", [(40, 1), (1000, 3), (5003, 7), (20_011, 40)])
def test_cancelling_second_derivative(lib, model, layout, n, K):
    rng = np.random.default_rng(n + K)
    p = 6
    time = np.sort(rng.integers(1, K + 1, n))[::-1].astype(np.int32).copy()
    status = rng.integers(1, 3, n).astype(np.int8) if model == "fg" else rng.integers(0, 2, n).astype(np.int8)
    X = 1024 + (rng.random((n, p)) < 0.4).astype(np.int64)
    if layout == "csc":
        sd = binding.SurvData(dev(time), dev(status), col_ptr=dev(np.arange(p + 1, dtype=np.int64) * n),
                              row_idx=dev(np.tile(np.arange(n, dtype=np.int32), p)),
                              values=dev(X.T.astype(np.float32).reshape(-1)), n=n, p=p)
    else:
        sd = binding.SurvData(dev(time), dev(status), X=dev(X.T.astype(np.float32)))
    for j in range(p):
        _, g, h = binding.loglik_grad_hess(sd, model, np.zeros(p), j)
        g0, h0 = _exact(model, time, status, X[:, j])
        assert h == pytest.approx(h0, rel=4e-9)
        assert g == pytest.approx(g0, abs=1e-12 * 1025 * n)
