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


def _against_oracle(model, d, X, values, where, j_list):
    """l, l', l'' in the FP64 mode: 1e-10 of the sums of magnitudes, as the
    parity tests hold it."""
    import torch
    put = (lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda())
    if where == "csc":
        import scipy.sparse
        S = scipy.sparse.csc_matrix(X)
        S.sort_indices()
        sd = binding.SurvData(put(d["time"]), put(d["status"]), col_ptr=put(S.indptr.astype(np.int64)),
                              row_idx=put(S.indices.astype(np.int32)), values=put(S.data) if values else None,
                              n=X.shape[0], p=X.shape[1])
    else:
        sd = binding.SurvData(put(d["time"]), put(d["status"]), X=put(np.ascontiguousarray(X.T)))
    beta = np.linspace(-0.2, 0.2, X.shape[1])
    ev = d["status"] == 1
    for j in j_list:
        l, g, h = binding.loglik_grad_hess(sd, model, beta, j, precision="f64")
        lo, go, ho = oracle.model_terms(model, d["time"], d["status"], X, beta, j)
        m = np.max(np.abs(X[:, j]), initial=0.0)
        scale = max(1.0, float(np.count_nonzero(ev)))
        assert abs(l - lo) <= 1e-10 * max(1.0, abs(lo))
        assert abs(g - go) <= 1e-10 * scale * max(m, 1e-300)
        assert abs(h - ho) <= 1e-10 * scale * max(m * m, 1e-300)


# the column pass takes 1024 entries a round and 4096 a block
@pytest.mark.parametrize("values", [False, True])
def test_columns_of_every_length(lib, values):
    from paper_2204_08183_gb300 import synth
    n = 9001
    d = synth.cohort_small(n, 1, seed=5, n_times=700)
    rng = np.random.default_rng(6)
    lengths = [0, 1, 2, 31, 33, 1023, 1024, 1025, 4095, 4097, n]
    X = np.zeros((n, len(lengths)))
    for j, k in enumerate(lengths):
        rows = np.sort(rng.choice(n, k, replace=False))
        if k in (1, 2):
            rows = np.array([0, n - 1])[:k] if k == 2 else np.array([n - 1])
        X[rows, j] = rng.normal(size=k) if values else 1.0
    _against_oracle("cox", d, X, values, "csc", range(len(lengths)))


# four entries a load, and columns that start and end inside one: a fault is
# found at every place
@pytest.mark.parametrize("values", [None, "ones", "real"])
@pytest.mark.parametrize("first", [0, 1, 3, 4])
def test_faults_at_every_entry(lib, first, values):
    rng = np.random.default_rng(first)
    n, k = 300, 22
    time = np.arange(n, 0, -1).astype(np.int32)
    status = (rng.random(n) < 0.6).astype(np.int8)
    rows = np.concatenate([np.sort(rng.choice(n, m, replace=False)) for m in (first, k, 5)]).astype(np.int32)
    col_ptr = np.array([0, first, first + k, first + k + 5], dtype=np.int64)
    vals = None if values is None else (np.ones(len(rows)) if values == "ones" else rng.normal(size=len(rows)))

    def code(rows, vals):
        d = binding.SurvData(time, status, col_ptr=col_ptr, row_idx=rows, values=vals, n=n, p=3)
        try:
            binding.cox_lambda_max(d)
        except binding.SurvError as e:
            return e.code
        return 0

    assert code(rows, vals) == 0
    for i in range(first, first + k):
        for bad in ([-1, n] if i == first else [-1, n, rows[i - 1]]):
            r = rows.copy()
            r[i] = bad
            assert code(r, vals) == binding.SURV_E_INDEX, (i, bad)
        if vals is not None:
            for bad in (np.nan, np.inf):
                v = vals.copy()
                v[i] = bad
                assert code(rows, v) == binding.SURV_E_NONFINITE, (i, bad)


@pytest.mark.parametrize("n", [1, 5, 127, 4095, 4097, 8193, 20003])
def test_dense_and_weights_at_block_edges(lib, n):
    from paper_2204_08183_gb300 import synth
    d = synth.cohort_small(n, 3, seed=n, n_times=max(1, n // 7), competing_frac=0.3)
    d["status"][0] = 1
    _against_oracle("fg", d, np.asarray(d["X"]), True, "dense", range(3))


def test_one_call_scratch_from_threads_and_streams(lib):
    """Calls without a workspace share the device's scratch pool: several
    threads on streams of their own, sizes that grow and shrink."""
    import threading

    import torch
    sizes = [1000, 300_000, 5000, 1_200_000]
    times = [torch.randint(1, 3650, (n,), dtype=torch.int32, device="cuda") for n in sizes]
    refs = [oracle.sort_desc(t.cpu().numpy()).astype(np.int32) for t in times]
    torch.cuda.synchronize()
    bad = []

    def work(k):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for r in range(12):
                i = (k + r) % len(sizes)
                perm = binding.surv_sort_desc(times[i])
                st.synchronize()
                if not np.array_equal(perm.cpu().numpy(), refs[i]):
                    bad.append((k, r))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
