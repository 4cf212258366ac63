"""The differentiable form with eta kept on the chip (p <= 256) at the edges
of its tiles: 64 subjects a tile, 64 covariates a box and 128 an MMA tile, 16
columns a warp quadrant; groups of one and of many subjects.  Bounds as derived
in test_gpu_nll."""
import numpy as np
import pytest

import oracle
from paper_2204_08183_gb300 import binding

from test_gpu_nll import _accumulation_bound, _case, _grad_tol, _split

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ties", [True, False])
@pytest.mark.parametrize("n,p,C", [(2, 8, 1), (63, 8, 2), (64, 50, 5), (65, 64, 16), (129, 65, 17), (4097, 128, 33),
                                   (9731, 129, 64), (20_011, 192, 48), (40_001, 256, 64), (39_000, 200, 32),
                                   (80_000, 7, 64), (38_913, 256, 1)])
def test_shapes(lib, n, p, C, ties):
    import torch
    c, X, B, t, s, Xo = _case(n, p, C, seed=n + p + C, n_times=max(1, n // 40) if ties else 50 * n)
    Bt = B.clone().requires_grad_(True)
    nll = binding.cox_nll(Bt, X, t, s)
    w = torch.linspace(0.5, 1.5, C, dtype=torch.float64, device="cuda")
    (g,) = torch.autograd.grad((nll * w).sum(), Bt)
    eta = Xo @ _split(c["B"])
    ref = oracle.cox_nll(c["time"], c["status"], eta)
    np.testing.assert_allclose(nll.detach().cpu().numpy(), ref, rtol=1e-7, atol=1e-6)
    ge = oracle.cox_nll_grad_eta(c["time"], c["status"], eta) * w.cpu().numpy()[None, :]
    gref = Xo.T @ ge
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    # FP32 storage of Lambda and of G: 2^-23 of every term's parts
    parts = np.abs(Xo).T @ (np.abs(ge) + (c["status"] == 1)[:, None] * w.cpu().numpy()[None, :])
    tol = _grad_tol(Xo, ge, gref) + _accumulation_bound(Xo, ge, n_sm) + 2.0 ** -22 * parts
    assert np.all(np.abs(g.cpu().numpy() - gref) <= tol)


def test_wide_x_takes_the_separate_kernels(lib):
    """p > 256: eta and G in memory, as before."""
    import torch
    c, X, B, t, s, Xo = _case(3000, 264, 8, seed=7)
    Bt = B.clone().requires_grad_(True)
    nll = binding.cox_nll(Bt, X, t, s)
    (g,) = torch.autograd.grad(nll.sum(), Bt)
    eta = Xo @ _split(c["B"])
    np.testing.assert_allclose(nll.detach().cpu().numpy(), oracle.cox_nll(c["time"], c["status"], eta), rtol=1e-7)
    ge = oracle.cox_nll_grad_eta(c["time"], c["status"], eta)
    assert np.all(np.abs(g.cpu().numpy() - Xo.T @ ge) <= _grad_tol(Xo, ge, Xo.T @ ge))
