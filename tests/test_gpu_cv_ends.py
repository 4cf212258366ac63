"""Cross-validated paths whose transform has more, and fewer, CTAs than the
pass: one subject per group, and a handful of groups."""
import numpy as np
import pytest

from paper_2204_08183_gb300 import binding, synth

from gpu_util import small_csc, survdata
from test_gpu_cv import _compare

pytestmark = pytest.mark.gpu


# 512 ends a CTA of the batched transform, at most 152 of them
@pytest.mark.parametrize("n,n_times", [(2000, 3), (4001, 512), (4001, 513), (100_003, 10**8)])
def test_cv_path_by_groups(lib, n, n_times):
    d = small_csc(n, 3, seed=n, density=0.1, n_times=n_times)
    fold = synth.cv_folds(n, 2, seed=3)
    lam = synth.lambda_grid(binding.cox_lambda_max(survdata(d)), 2, ratio=1e-1)
    _compare(d, fold, 2, lam, "l1", "f32c", 2)
