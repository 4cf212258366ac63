"""The once-per-call preparation at the sizes where its tiles end: tie groups
and the stable order, exact against the oracle (integers, and the ordered
Kaplan-Meier product up to 4096 groups)."""
import numpy as np
import pytest

import oracle
from paper_2204_08183_gb300 import binding

pytestmark = pytest.mark.gpu

# blocks of the group kernels hold 4096 subjects, warps 512, rounds 128
EDGES = [1, 2, 31, 127, 128, 129, 511, 513, 4095, 4096, 4097, 12289]


@pytest.mark.parametrize("offset", [0, 1])   # 1: arrays that start off a 16-byte boundary
@pytest.mark.parametrize("n_times", [1, 3, 4000, 10**6])
@pytest.mark.parametrize("n", EDGES)
def test_groups_at_block_edges(lib, n, n_times, offset):
    import torch
    rng = np.random.default_rng(n + n_times)
    time = np.sort(rng.integers(1, n_times + 1, n).astype(np.int32))[::-1].copy()
    status = rng.integers(0, 3, n).astype(np.int8)
    t = torch.zeros(n + offset, dtype=torch.int32, device="cuda")
    s = torch.zeros(n + offset, dtype=torch.int8, device="cuda")
    t[offset:] = torch.from_numpy(time)
    s[offset:] = torch.from_numpy(status)
    gend, dk, Gk = binding.surv_groups(t[offset:], s[offset:])
    ref = np.asarray(oracle.tie_groups(time))
    np.testing.assert_array_equal(gend, ref)
    np.testing.assert_array_equal(dk, oracle.group_counts(ref, status, 1))
    G = oracle.km_censoring_groups(time, status, ref)
    if len(ref) <= 4096:
        np.testing.assert_array_equal(Gk, G)
    else:   # the chunked product: below (2 L + 12 + K) u relative of the sequential one
        K = len(ref)
        np.testing.assert_allclose(Gk, G, rtol=(2 * -(-K // 1024) + 12 + K) * 2.0 ** -53)


# tiles of the sort hold 4096 elements; the spans need 0, 1, 8, 9, 17 and 32
# key bits: 0 to 4 passes of equal digits
@pytest.mark.parametrize("span", [1, 2, 256, 257, 100_000, 2**32])
@pytest.mark.parametrize("n", [1, 33, 4095, 4096, 4097, 70_001])
def test_sort_at_tile_edges_and_key_spans(lib, n, span):
    import torch
    rng = np.random.default_rng(n + span)
    lo = -(span // 2)
    time = rng.integers(lo, lo + span, n).astype(np.int32)
    time[0], time[-1] = lo, lo + span - 1
    ref = oracle.sort_desc(time).astype(np.int32)
    t = torch.from_numpy(time).cuda()
    np.testing.assert_array_equal(binding.surv_sort_desc(t).cpu().numpy(), ref)
    binding.surv_sort_desc(t, perm=t)   # the order written over the times
    np.testing.assert_array_equal(t.cpu().numpy(), ref)
