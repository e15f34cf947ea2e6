"""GPU parity and speed of the dense-slice rows that reach few columns with many products or in
short parts, which take CTAs although a warp per row serves their neighbours: parts of 0 to 40
columns on both sides of the lines, ranges from one column to 1,024, A rows of one window and of
several, ranges that cross slice boundaries, long rows among few and among many.  Small-integer
values: every sum is exact."""
import time

import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (entries of A, columns of a part, columns of the range)
ROWS = ((520, 1, 1), (511, 2, 33), (512, 3, 200), (513, 2, 255), (1025, 1, 256), (300, 7, 257), (1500, 2, 1000),
        (140, 11, 1023), (2100, 40, 1024), (150, 40, 700), (600, 8, 64), (240, 18, 90), (230, 17, 90), (110, 14, 300))


def _matrices(ncols, seed, times):
    rng = np.random.default_rng(seed)
    ar, ac, br, bc, nb = [], [], [], [], 0
    for i, (na, part, w) in enumerate(ROWS * times):
        lo = int(rng.integers(0, ncols - w + 1))
        if i % 2:
            lo = max(0, min(ncols - w, 1024 * (1 + i % 5) - w // 2))  # across a multiple of 1,024
        for q in range(na):
            n = min(w, part + (0 if part < 3 else int(rng.integers(-1, 2))))
            if q < 2:
                c = np.array([lo if q == 0 else lo + w - 1])
            elif part > 1 and q % 11 == 7:
                c = np.zeros(0, dtype=np.int64)
            else:
                c = np.sort(rng.choice(w, size=n, replace=False)) + lo
            br.append(np.full(c.size, nb)); bc.append(c); ar.append(i); ac.append(nb)
            nb += 1
    b_r, b_c = np.concatenate(br), np.concatenate(bc)
    B = gen.from_coo(nb, ncols, b_r, b_c, rng.integers(-4, 5, b_r.size).astype(np.float64))
    A = gen.from_coo(len(ROWS) * times, nb, np.array(ar), np.array(ac), rng.integers(-4, 5, len(ar)).astype(np.float64))
    return A, B


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ncols,span", [(1024, 0), (9000, 0), (9000, 1024)])
@pytest.mark.parametrize("policy", ["hybrid", "precise", "device"])
def test_heavy_rows_exact(oracle_mod, dtype, ncols, span, policy):
    import paper_1504_05022_gb300 as spg
    A, B = _matrices(ncols, seed=ncols + span, times=2)
    ref = oracle_mod.spgemm(A, B)
    Ad, Bd = (spg.CSR.from_host(M, dtype=dtype) for M in (A, B))
    if policy == "device":
        plan = spg.DevicePlan(Ad, Bd, ref.col.size, dense_span=span)
        runs = [plan.run, plan.run]
    else:
        plan = spg.Plan(Ad, Bd, alloc_policy=policy, dense_span=span)
        plan.numeric()
        st = plan.stats()
        assert st["rows_dense"] > 0 and (policy == "hybrid" or st["rows_dense"] == st["bin_count"][37])
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


def test_long_rows_among_many(oracle_mod):
    """A few rows of 10,000 products beside 3,000 of 600: the long ones change kernels, the others stay."""
    import paper_1504_05022_gb300 as spg
    rng = np.random.default_rng(11)
    ar, ac, nb = [], [], 400
    for i in range(3000):
        k = 250 if i % 500 == 7 else 15
        ar.append(np.full(k, i)); ac.append(np.sort(rng.choice(nb, size=k, replace=False)))
    f = rng.integers(0, 60, nb)
    bc = (f[:, None] + np.arange(40)[None, :]).reshape(-1)
    A = gen.from_coo(3000, nb, np.concatenate(ar), np.concatenate(ac), rng.integers(-4, 5, sum(a.size for a in ar)).astype(np.float64))
    B = gen.from_coo(nb, 100, np.repeat(np.arange(nb), 40), bc, rng.integers(-4, 5, bc.size).astype(np.float64))
    ref = oracle_mod.spgemm(A, B)
    Ad, Bd = spg.CSR.from_host(A), spg.CSR.from_host(B)
    for policy in ("hybrid", "precise"):
        plan = spg.Plan(Ad, Bd, alloc_policy=policy)
        C = plan.numeric()
        plan.replay()
        plan.check()
        assert plan.stats()["rows_dense"] == 3000
        rp, col, val = C.to_host()
        assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col) and np.array_equal(val, ref.val)


def _gram(n, m, per_row, spread):
    """A^T A of an m x n matrix with per_row entries a row; B's columns `spread` apart."""
    rng = np.random.default_rng(n)
    c = rng.integers(0, n, size=(m, per_row), dtype=np.int64)
    key = np.unique(np.arange(m)[:, None] * n + c)
    r, c = key // n, key % n
    v = rng.integers(-4, 5, key.size).astype(np.float64)
    return gen.from_coo(n, m, c, r, v), gen.from_coo(m, n * spread, r, c * spread, v)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n", [64, 200])
def test_gram_product_is_no_slower_in_a_narrow_range(dtype, n):
    """The same products over a range of more than 1,024 columns take a CTA per slice: a narrower
    range must not take longer (by a warp per row, 4 to 15 times as long)."""
    import paper_1504_05022_gb300 as spg

    def ms(spread):
        A, B = (spg.CSR.from_host(M, dtype=dtype) for M in _gram(n, 300000, 8, spread))
        best = 1e9
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            spg.spgemm(A, B)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        return 1e3 * best

    assert ms(1) < 1.5 * ms(2048 // n)
