"""GPU parity of the column-slice kernels' product walk where it can go wrong: B-row parts of
0, 1, 31..33, 127..129 and thousands of entries, A rows that fill a 256-entry window exactly or
by one more or less, and results from a few entries to a whole slice of 131,072 columns (every
size class of the single-precision fill, and its pieces).  Small-integer values, so every sum
is exact in either precision and in any order."""
import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PARTS = (0, 1, 31, 32, 33, 0, 127, 128, 129, 2, 700, 64)


def _matrices(ncols, seed):
    rng = np.random.default_rng(seed)
    nb = 700
    rows, cols = [], []
    for k in range(nb):
        n = ncols if k == nb - 1 else min(ncols, 30000 if k == nb - 2 else PARTS[k % len(PARTS)])
        rows.append(np.full(n, k))
        cols.append(np.sort(rng.choice(ncols, size=n, replace=False)))
    r, c = np.concatenate(rows), np.concatenate(cols)
    B = gen.from_coo(nb, ncols, r, c, rng.integers(-4, 5, r.size).astype(np.float64))
    sizes = (1, 3, 40, 255, 256, 257, 511, 513, 650)
    ar, ac = [], []
    for i, n in enumerate(sizes * 2):
        # the second half of the rows also selects the two long B rows
        pick = np.sort(rng.choice(nb - 2, size=n, replace=False))
        if i >= len(sizes):
            pick = np.concatenate([pick[:-2], [nb - 2, nb - 1]]) if n > 2 else np.array([nb - 1])
        ar.append(np.full(pick.size, i))
        ac.append(pick)
    r, c = np.concatenate(ar), np.concatenate(ac)
    A = gen.from_coo(2 * len(sizes), nb, r, c, rng.integers(-4, 5, r.size).astype(np.float64))
    return A, B


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ncols,span", [(4000, 0), (131072, 0), (131073, 0), (150001, 65536)])
@pytest.mark.parametrize("policy,keep", [("hybrid", 0), ("hybrid", -1), ("precise", 0)])
def test_slices_exact(oracle_mod, dtype, ncols, span, policy, keep):
    import paper_1504_05022_gb300 as spg
    A, B = _matrices(ncols, seed=ncols)
    Ad, Bd = (spg.CSR.from_host(M, dtype=dtype) for M in (A, B))
    plan = spg.Plan(Ad, Bd, alloc_policy=policy, dense_min_u=513, dense_span=span, dense_keep=keep)
    C = plan.numeric()
    ref = oracle_mod.spgemm(A, B)
    assert plan.stats()["rows_dense"] > 8
    for scale in (1.0, 3.0):  # the product, then a values-only replay with A scaled
        if scale != 1.0:
            Ad.val.mul_(scale)
            plan.replay()
        plan.check()
        rp, col, val = C.to_host()
        assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
        assert np.array_equal(val.astype(np.float64), scale * ref.val)
