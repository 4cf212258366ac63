"""Host arrays are read in the order of the call's stream: what earlier work on
that stream writes into them (here a host function behind a long kernel) is
what the call sees."""
import ctypes as C

import numpy as np
import pytest

from paper_2204_08183_gb300 import binding

from gpu_util import small_csc, survdata

pytestmark = pytest.mark.gpu


def _after_a_while(stream, write):
    """Enqueue a kernel of some tens of ms and write() behind it on `stream`."""
    import torch
    fn = C.CFUNCTYPE(None, C.c_void_p)
    call = fn(lambda _: write())
    cu = C.CDLL("libcuda.so.1")
    cu.cuLaunchHostFunc.argtypes = [C.c_void_p, fn, C.c_void_p]
    torch.cuda._sleep(100_000_000)
    assert cu.cuLaunchHostFunc(stream.cuda_stream, call, None) == 0
    return call


@pytest.mark.parametrize("what", ["beta", "warm_start", "penalty_factor", "col_ptr"])
def test_host_array_written_by_earlier_work(lib, what):
    import torch
    d = small_csc(2000, 6, seed=4, density=0.2, n_times=50)
    sd = survdata(d)
    beta = np.linspace(-0.2, 0.3, 6)
    pf = np.array([0.0, 1.0, 2.0, 0.5, 1.0, 3.0])

    def call(beta_in, pf_in, data):
        if what in ("beta", "col_ptr"):
            return binding.loglik_grad_hess(data, "cox", beta_in, 2)
        b, info, _ = binding.cox_fit(data, beta=beta_in, penalty="l2", lam=3.0, penalty_factor=pf_in, tol=0.0,
                                     max_sweeps=2)
        return tuple(b) + (info["loglik"],)

    want = call(beta.copy(), pf, sd)
    beta_in, pf_in, ptr = beta.copy(), pf.copy(), d["col_ptr"].copy()
    late = binding.SurvData(sd._keep[0], sd._keep[1], col_ptr=ptr, row_idx=sd._keep[4], values=sd._keep[5],
                            n=d["n"], p=d["p"])
    target, value = {"beta": (beta_in, beta), "warm_start": (beta_in, beta), "penalty_factor": (pf_in, pf),
                     "col_ptr": (ptr, d["col_ptr"])}[what]
    target[:] = 0.0 if what != "col_ptr" else np.minimum(value, value[1])
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        keep = _after_a_while(s, lambda: target.__setitem__(slice(None), value))
        got = call(beta_in, pf_in, late)
    torch.cuda.synchronize()
    assert got == want
    del keep
