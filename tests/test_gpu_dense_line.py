"""Which bin-37 rows the column slices take by default, on both sides of the line."""
import numpy as np
import pytest

import gen
from tests.helpers import assert_csr_equal

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _line(A, B):
    """u_i and the width of the column range of every row of A*B."""
    n = np.diff(B.row_ptr)
    full = n > 0
    rows = np.repeat(np.arange(A.nrows), np.diff(A.row_ptr))
    u = np.zeros(A.nrows, dtype=np.int64)
    np.add.at(u, rows, n[A.col])
    lo, hi = np.full(A.nrows, B.ncols), np.zeros(A.nrows, dtype=np.int64)
    keep = full[A.col]
    np.minimum.at(lo, rows[keep], B.col[B.row_ptr[:-1][A.col[keep]]])
    np.maximum.at(hi, rows[keep], B.col[B.row_ptr[1:][A.col[keep]] - 1] + 1)
    return u, hi - lo


def _graded(ncols, per, us, seed):
    """Rows of A that select u / per rows of B, each of `per` uniformly random columns."""
    B = gen.erdos_renyi(600, per, seed=seed, ncols=ncols)
    rng = np.random.default_rng(seed)
    c = [np.sort(rng.choice(600, size=u // per, replace=False)) for u in us]
    r = np.repeat(np.arange(len(us)), [x.size for x in c])
    return gen.from_coo(len(us), 600, r, np.concatenate(c), rng.uniform(-1, 1, r.size)), B


CASES = {"ranges up to 16,384": lambda: _graded(16384, 8, range(1520, 2400, 24), 1),
         "ranges above 16,384": lambda: _graded(65536, 8, range(1800, 2300, 24), 2),
         "rows below 1,024 products": lambda: _graded(20000, 8, range(520, 1500, 24), 5),
         "rows above 8,192 products": lambda: _graded(8192 * 512, 40, range(7800, 8600, 40), 3),
         "R-MAT": lambda: (gen.rmat(15, 8, seed=4),) * 2}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("policy", ["hybrid", "upper_bound"])
@pytest.mark.parametrize("case", list(CASES))
def test_default_line(oracle_mod, case, policy, dtype):
    import paper_1504_05022_gb300 as spg
    A, B = CASES[case]()
    for M in (A, B):
        M.val[:] = np.rint(4 * M.val)  # small integers: every sum is exact
    u, span = _line(A, B)
    div = np.where(u > 8192, 512, np.where(span > 16384, 32, 8))
    ref = oracle_mod.spgemm(A, B)
    Ad, Bd = (spg.CSR.from_host(M, dtype=dtype) for M in (A, B))
    for opts, d in (({}, div), ({"dense_span_div": 8}, 8)):
        plan = spg.Plan(Ad, Bd, alloc_policy=policy, **opts)
        rp, col, val = plan.numeric().to_host()
        plan.check()
        assert plan.stats()["rows_dense"] == ((u > 512) & (d * u >= span) & ((u >= 1024) | (span <= 16384) | (d is not div))).sum()
        assert_csr_equal(rp, col, val.astype(np.float64), ref.row_ptr, ref.col, ref.val, ref.den, label=case)
