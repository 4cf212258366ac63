"""A call without a workspace keeps at most 256 MiB of device memory after it
returns, before anybody synchronises."""
import pytest

from paper_2204_08183_gb300 import binding

pytestmark = pytest.mark.gpu
KEEP = 256 << 20
SLACK = 48 << 20     # the device allocates in blocks of 32 MiB or less


def test_large_call_gives_its_memory_back(lib):
    import torch
    n = 60_000_000    # 720 MB of keys, values and counts
    t = torch.randint(0, 3650, (n,), device="cuda", dtype=torch.int32)
    perm = torch.empty(n, device="cuda", dtype=torch.int32)
    binding.surv_sort_desc(t[:1000].clone())
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    binding.surv_sort_desc(t, perm)
    assert free - torch.cuda.mem_get_info()[0] <= KEEP + SLACK
    order = torch.sort(t, descending=True, stable=True).indices.to(torch.int32)
    assert torch.equal(perm, order)
