"""GPU parity of the dense-slice rows that reach few columns (a warp per row): column ranges around
256 and 1,024, B rows of consecutive columns and of scattered ones, parts of 1, 31..33 and hundreds
of entries, A rows longer than a warp, ranges that cross slice boundaries, and rows of every width
in one product.  Small-integer values, so every sum is exact in either precision."""
import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WIDTHS = (33, 79, 255, 256, 257, 1000, 1023, 1024, 1025, 5000)


def _matrices(ncols, seed):
    """Row i of A selects B rows inside one window of WIDTHS[i] columns, some of them the
    window's first and last column."""
    rng = np.random.default_rng(seed)
    ar, ac, br, bc, nb = [], [], [], [], 0
    for i, w in enumerate(WIDTHS * 4):
        lo = int(rng.integers(0, ncols - w + 1))
        if i >= 2 * len(WIDTHS):
            lo = max(0, min(ncols - w, 2048 * (1 + i % 3) - w // 2))  # across a multiple of 2,048
        total = 0
        for q in range(200):
            kind, n = (q + i) % 3, min(w, (1, 31, 32, 33, 64, 300, w)[q % 7])
            if q < 2:
                c = np.array([lo if q == 0 else lo + w - 1])
            elif kind == 0:
                c = np.sort(rng.choice(w, size=n, replace=False)) + lo
            elif kind == 1:
                c = np.arange(n) + lo + int(rng.integers(0, w - n + 1))
            else:
                c = np.zeros(0, dtype=np.int64)
            br.append(np.full(c.size, nb)); bc.append(c); ar.append(i); ac.append(nb)
            nb += 1
            total += c.size
            if total > 700 and q > 40 + 50 * (i % 3):
                break
    b_r, b_c = np.concatenate(br), np.concatenate(bc)
    B = gen.from_coo(nb, ncols, b_r, b_c, rng.integers(-4, 5, b_r.size).astype(np.float64))
    A = gen.from_coo(4 * len(WIDTHS), nb, np.array(ar), np.array(ac), rng.integers(-4, 5, len(ar)).astype(np.float64))
    return A, B


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ncols,span", [(9000, 0), (9000, 2048), (9000, 1024), (1500, 1024)])
@pytest.mark.parametrize("policy", ["hybrid", "precise", "device"])
def test_narrow_rows_exact(oracle_mod, dtype, ncols, span, policy):
    import paper_1504_05022_gb300 as spg
    A, B = _matrices(max(ncols, 5000), seed=ncols + span) if ncols > 5000 else _clip(ncols, span)
    ref = oracle_mod.spgemm(A, B)
    Ad, Bd = (spg.CSR.from_host(M, dtype=dtype) for M in (A, B))
    if policy == "device":
        plan = spg.DevicePlan(Ad, Bd, ref.col.size, dense_span=span)
        runs = [plan.run, plan.run]
    else:
        plan = spg.Plan(Ad, Bd, alloc_policy=policy, dense_min_u=513, dense_span=span)
        plan.numeric()
        first = np.concatenate([[0], np.cumsum(np.diff(B.row_ptr)[A.col])])
        u = first[A.row_ptr[1:]] - first[A.row_ptr[:-1]]
        assert plan.stats()["rows_dense"] == (u >= 513).sum() > 0
        runs = [lambda: None, plan.replay]
    scale = 1.0
    for k, again in enumerate(runs):  # the product, then with A scaled (a values-only replay)
        if k:
            Ad.val.mul_(3.0)
            scale = 3.0
        again()
        C = plan.result() if policy == "device" else plan.numeric()
        if policy != "device":
            plan.check()
        rp, col, val = C.to_host()
        assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
        assert np.array_equal(val.astype(np.float64), scale * ref.val)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("long", [True, False])
@pytest.mark.parametrize("scattered", [0, 1, 33])
def test_consecutive_parts_exact(oracle_mod, dtype, long, scattered):
    """Rows whose B rows are runs of consecutive columns, long or short beside the range, with
    `scattered` others (whole windows of 32 runs, mixed windows); small integers are exact."""
    import paper_1504_05022_gb300 as spg
    rng = np.random.default_rng(40 + scattered + long)
    ar, ac, br, bc, nb = [], [], [], [], 0
    for i, w in enumerate((31, 32, 33, 63, 64, 65, 200, 255, 256, 257)):
        lo = int(rng.integers(0, 3000))
        for q in range(700 if not long else 96):
            n = max(1, w - q % 3) if long else 1 + q % 2
            f = lo + (0 if q == 0 else w - n if q == 1 else int(rng.integers(0, w - n + 1)))
            c = np.arange(f, f + n)
            if q % 16 == 5 and q // 16 < scattered:
                c = np.unique(np.array([lo, lo + w // 2, lo + w - 1]))
            br.append(np.full(c.size, nb)); bc.append(c); ar.append(i); ac.append(nb)
            nb += 1
    b_r, b_c = np.concatenate(br), np.concatenate(bc)
    B = gen.from_coo(nb, 5000, b_r, b_c, rng.integers(-4, 5, b_r.size).astype(np.float64))
    A = gen.from_coo(10, nb, np.array(ar), np.array(ac), rng.integers(-4, 5, len(ar)).astype(np.float64))
    ref = oracle_mod.spgemm(A, B)
    Ad, Bd = (spg.CSR.from_host(M, dtype=dtype) for M in (A, B))
    plan = spg.Plan(Ad, Bd, dense_min_u=513)
    plan.numeric()
    assert plan.stats()["rows_dense"] == 10
    for scale in (1.0, 3.0):
        if scale > 1.0:
            Ad.val.mul_(scale)
            plan.replay()
        C = plan.numeric()
        plan.check()
        rp, col, val = C.to_host()
        assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
        assert np.array_equal(val.astype(np.float64), scale * ref.val)


def _clip(ncols, span):
    """The same rows folded into a B of ncols columns (slices narrower than 1,024)."""
    A, B = _matrices(5000, seed=ncols + span)
    rows = np.repeat(np.arange(B.nrows), np.diff(B.row_ptr))
    keep = B.col < ncols
    return A, gen.from_coo(B.nrows, ncols, rows[keep], B.col[keep].astype(np.int64), B.val[keep])


def test_replay_sees_a_changed_structure():
    """A product whose column C does not hold is reported, and nothing else is written."""
    import paper_1504_05022_gb300 as spg
    M = spg.CSR.from_host(gen.banded(3000, 40, seed=5))
    plan = spg.Plan(M, M)
    plan.numeric()
    assert plan.stats()["rows_dense"] > 0
    plan.replay()
    plan.check()
    M.col[-1] -= 1200  # the last row's last entry selects a B row far from the others
    M.col[M.row_ptr[-2]:] = torch.sort(M.col[M.row_ptr[-2]:])[0]
    plan.replay()
    with pytest.raises(spg.SpgemmError):
        plan.check()
