"""The table of slice boundaries is optional: a few long rows in a B of many rows do not build it, a
plan without the memory for it is computed without it, and both forms give the oracle's C."""
import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _hubs(n, hubs, entries, seed):
    """n x n, three entries a row and `hubs` rows of `entries`; small integers."""
    rng = np.random.default_rng(seed)
    r = [np.repeat(np.arange(n), 3)] + [np.full(entries, (n // hubs) * h + 1) for h in range(hubs)]
    c = [rng.integers(0, n, 3 * n)] + [rng.integers(0, n, entries) for _ in range(hubs)]
    key = np.unique(np.concatenate(r).astype(np.int64) * n + np.concatenate(c))
    return gen.from_coo(n, n, key // n, key % n, rng.integers(-4, 5, key.size).astype(np.float64))


def test_few_long_rows_fit_where_no_slice_row_would_need_more(oracle_mod):
    import paper_1504_05022_gb300 as spg
    A = _hubs(600000, 3, 4000, 1)
    ref = oracle_mod.spgemm(A, A)
    Ad = spg.CSR.from_host(A)
    off = spg.Plan(Ad, Ad, dense_min_u=1 << 30)  # the merge kernels take the hubs
    off.numeric()
    st = off.stats()
    assert st["rows_dense"] == 0 and st["bin_count"][37] >= 3
    plan = spg.Plan(Ad, Ad, max_bytes=st["peak_bytes"])  # the default line sends them to the slices
    C = plan.numeric()
    new = plan.stats()
    assert new["rows_dense"] >= 3 and new["dense_slices"] > 1
    assert new["held_bytes"] <= st["held_bytes"] + (1 << 20)  # no table of B's rows
    for again in (False, True):
        if again:
            Ad.val.mul_(2.0)
            plan.replay()
            plan.check()
        rp, col, val = C.to_host()
        assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
        assert np.array_equal(val, (4.0 if again else 1.0) * ref.val)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("policy", ["hybrid", "precise"])
@pytest.mark.parametrize("span", [1024, 2080])
def test_without_room_for_the_table(oracle_mod, dtype, policy, span):
    """Rows that build the table, and a limit that leaves no room for it: B rows of 0 to hundreds of entries
    in up to 30 slices, first and last columns of slices among them."""
    import paper_1504_05022_gb300 as spg
    rng = np.random.default_rng(span)
    n, nb = 30001, 900
    edges = np.concatenate([np.arange(span, n, span) - 1, np.arange(span, n, span), [0, n - 1]])
    br, bc = [], []
    for k in range(nb):
        m = (0, 1, 7, 300)[k % 4]
        c = np.unique(np.concatenate([rng.integers(0, n, m), rng.choice(edges, size=min(m, 20), replace=False)]))
        br.append(np.full(c.size, k)); bc.append(c)
    bc = np.concatenate(bc)
    B = gen.from_coo(nb, n, np.concatenate(br), bc, rng.integers(-4, 5, bc.size).astype(np.float64))
    ar = np.repeat(np.arange(120), 200)
    ac = np.concatenate([np.sort(rng.choice(nb, 200, replace=False)) for _ in range(120)])
    A = gen.from_coo(120, nb, ar, ac, rng.integers(-4, 5, ac.size).astype(np.float64))
    ref = oracle_mod.spgemm(A, B)
    Ad, Bd = (spg.CSR.from_host(M, dtype=dtype) for M in (A, B))
    opts = {"alloc_policy": policy, "dense_span": span, "dense_min_u": 600}
    full = spg.Plan(Ad, Bd, **opts)
    full.numeric()
    st = full.stats()
    table = 4 * (st["dense_slices"] + 1) * nb
    assert st["rows_dense"] == 120 and st["dense_slices"] > 10
    plan = spg.Plan(Ad, Bd, max_bytes=st["peak_bytes"] - table, **opts)
    plan.numeric()
    assert plan.stats()["held_bytes"] <= st["held_bytes"] - table
    for p in (full, plan):
        for scale in (1.0, 3.0):
            if scale > 1.0:
                Ad.val.mul_(3.0)
                p.replay()
                p.check()
            rp, col, val = p.numeric().to_host()
            assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
            assert np.array_equal(val.astype(np.float64), scale * ref.val)
        Ad.val.div_(3.0)
