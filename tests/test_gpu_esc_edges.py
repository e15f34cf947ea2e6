"""GPU parity of the bitonic ESC kernels at the edges of their networks (u_i around 8, 16, 32, 64,
128, 256 and 512), with 32-bit packed keys and with the 64-bit ones of a wide B, rows of A longer
than a group of lanes, empty B rows between the others, and many or no equal columns.
Small-integer values, so every sum is exact in either precision and in any order."""
import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = [u + d for u in (8, 16, 32, 64, 128, 256, 512) for d in (-1, 0, 1) if u + d <= 512]


def _matrices(ncols, longest, seed):
    """Row i of A*B has EDGES[i % n] products, from B rows of 0..longest entries whose columns
    come from a small set (many equal) or from all of B's."""
    rng = np.random.default_rng(seed)
    ar, ac, br, bc = [], [], [], []
    nb = 0
    for i, u in enumerate(EDGES * 3):
        left = u
        pool = np.unique(np.concatenate([rng.integers(0, ncols, 8 if i % 3 == 0 else 3 * longest + u),
                                         np.arange(longest), [ncols - 1]]))
        while left > 0:
            n = min(left, int(rng.integers(0, longest + 1)))
            bc.append(np.sort(rng.choice(pool, size=n, replace=False)))
            br.append(np.full(n, nb))
            ar.append(i)
            ac.append(nb)
            nb += 1
            left -= n
    b_r, b_c = np.concatenate(br), np.concatenate(bc)
    B = gen.from_coo(nb, ncols, b_r, b_c, rng.integers(-4, 5, b_r.size).astype(np.float64))
    A = gen.from_coo(len(EDGES) * 3, nb, np.array(ar), np.array(ac), rng.integers(-4, 5, len(ar)).astype(np.float64))
    return A, B


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ncols", [700, (1 << 23) - 1, 1 << 23, 1 << 27, (1 << 31) - 1])
@pytest.mark.parametrize("longest", [1, 5, 40])
def test_esc_exact(dtype, ncols, longest):
    import paper_1504_05022_gb300 as spg
    A, B = _matrices(ncols, longest, seed=ncols % 1000 + longest)
    used = np.unique(B.col)  # the oracle's accumulator takes the used columns, renumbered
    Bc = gen.HostCSR(B.nrows, used.size, B.row_ptr, np.searchsorted(used, B.col).astype(np.int32), B.val)
    import oracle
    ref = oracle.spgemm(A, Bc)
    Ad, Bd = (spg.CSR.from_host(M, dtype=dtype) for M in (A, B))
    policies = ["hybrid", "upper_bound"] + (["precise"] if ncols <= 1 << 23 else [])
    for policy in policies:
        plan = spg.Plan(Ad, Bd, alloc_policy=policy)
        C = plan.numeric()
        for _ in range(2):  # the product, then a values-only replay
            rp, col, val = C.to_host()
            assert np.array_equal(rp, ref.row_ptr), policy
            assert np.array_equal(col, used[ref.col]), policy
            assert np.array_equal(val.astype(np.float64), ref.val), policy
            C.val.zero_()
            plan.replay()
            plan.check()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ncols", [900, (1 << 27) - 1, 1 << 29])
@pytest.mark.parametrize("longest", [1, 3, 12])
def test_many_short_rows_exact(dtype, ncols, longest):
    """Enough rows of u_i = 2..32 for the kernels with a thread per row (every network width), with
    empty B rows, many and no equal columns, and 32- and 64-bit keys."""
    import oracle
    import paper_1504_05022_gb300 as spg
    rng = np.random.default_rng(longest + ncols % 97)
    m, nb = 60000, 5000
    n = rng.integers(0, longest + 1, nb)
    n[0] = 0
    b_r = np.repeat(np.arange(nb), n)
    pool = np.unique(rng.integers(0, ncols, 40 if ncols == 900 else 20000))
    b_c = np.concatenate([np.sort(rng.choice(pool, size=x, replace=False)) for x in n])
    B = gen.from_coo(nb, ncols, b_r, b_c, rng.integers(-4, 5, b_r.size).astype(np.float64))
    k = rng.integers(1, max(2, 64 // (longest + 1)), m)
    a_r = np.repeat(np.arange(m), k)
    A = gen.from_coo(m, nb, a_r, rng.integers(0, nb, a_r.size), None)
    A.val = rng.integers(-4, 5, A.nnz).astype(np.float64)
    used = np.unique(B.col)
    ref = oracle.spgemm(A, gen.HostCSR(nb, used.size, B.row_ptr, np.searchsorted(used, B.col).astype(np.int32), B.val))
    Ad, Bd = (spg.CSR.from_host(M, dtype=dtype) for M in (A, B))
    plans = [spg.Plan(Ad, Bd, alloc_policy=p) for p in ["hybrid"] + (["precise"] if ncols == 900 else [])]
    bins = plans[0].stats()["bin_count"]
    assert max(sum(bins[2:9]), sum(bins[9:17]), sum(bins[17:33])) >= 16384
    for plan in plans:
        C = plan.numeric()
        for _ in range(2):  # the product, then a values-only replay
            rp, col, val = C.to_host()
            assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, used[ref.col])
            assert np.array_equal(val.astype(np.float64), ref.val)
            C.val.zero_()
            plan.replay()
            plan.check()
