"""GPU parity of stages 1 and 2 where their launch shapes change: average rows that take groups of
4, 8, 16 and 32 lanes, hub rows a whole block takes, row counts around a block, a scan tile and
the number of tiles whose sums the blocks add up themselves.  All results are integers, compared
exactly with the oracle's Algorithms 2 and 3."""
import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("avg", [1, 5, 12, 40, 100])
@pytest.mark.parametrize("m", [1, 31, 257, 2049, 5000, 40000])
@pytest.mark.parametrize("bits", [32, 64])
def test_bounds_and_bins(oracle_mod, avg, m, bits):
    import paper_1504_05022_gb300 as spg
    rng = np.random.default_rng(avg * 100003 + m)
    k = 3000
    n = rng.integers(0, 2 * avg, m)
    n[rng.integers(0, m, 3)] = 0
    n[rng.integers(0, m, 2)] = (2500, 513)   # hub rows: more than 16 entries per lane of any group
    n = np.minimum(n, k)
    rows = np.repeat(np.arange(m), n)
    cols = np.concatenate([rng.choice(k, size=x, replace=False) for x in n]) if rows.size else rows
    A = gen.from_coo(m, k, rows, cols, None)
    B = gen.erdos_renyi(k, 3, seed=avg, ncols=2000)
    rdt = torch.int32 if bits == 32 else torch.int64
    plan = spg.Plan(spg.CSR.from_host(A, rowptr_dtype=rdt), spg.CSR.from_host(B, rowptr_dtype=rdt), dense_min_u=-1)
    arr = plan.arrays()
    u = oracle_mod.upper_bound(A, B)
    b, sz, cnt, order, total = oracle_mod.binning(u)
    assert np.array_equal(arr["u"], u)
    assert np.array_equal(arr["bin"].astype(np.int32), b)
    assert np.array_equal(arr["bin_rows"], order)
    assert np.array_equal(np.diff(arr["bin_start"]), cnt)
    assert np.array_equal(np.diff(arr["ctilde_row_ptr"]), sz) and int(arr["ctilde_row_ptr"][-1]) == total
    assert plan.upper_bound_nnz == int(u.sum())


@pytest.mark.parametrize("policy", ["hybrid", "precise"])
@pytest.mark.parametrize("extra", [0, 1])
def test_many_scan_tiles(policy, extra):
    """A diagonal matrix of 2,048 x 2,048 rows (the most whose tiles the scan adds up itself), and
    of one row more."""
    import paper_1504_05022_gb300 as spg
    n = 2048 * 2048 + extra
    idx = torch.arange(n, device="cuda", dtype=torch.int32)
    val = (idx % 7 - 3).double()
    A = spg.CSR(torch.arange(n + 1, device="cuda"), idx, val, (n, n))
    C = spg.spgemm(A, A, alloc_policy=policy)
    assert torch.equal(C.row_ptr, A.row_ptr) and torch.equal(C.col, idx) and torch.equal(C.val, val * val)
