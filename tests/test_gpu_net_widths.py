"""GPU parity of the thread-per-row kernels with enough rows at every width of their network, so that
each of the three sorts (8, 16 and 32 keys) runs for B rows of one, of few and of many entries."""
import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ncols", [900, (1 << 27) - 1, 1 << 29])  # 32- and 64-bit keys
@pytest.mark.parametrize("longest", [1, 3, 12])
def test_every_width_has_its_rows(dtype, ncols, longest):
    import oracle
    import paper_1504_05022_gb300 as spg
    rng = np.random.default_rng(longest + ncols % 97)
    m, nb = 120000, 5000
    n = rng.integers(0, longest + 1, nb)
    b_r = np.repeat(np.arange(nb), n)
    pool = np.unique(rng.integers(0, ncols, 40 if ncols == 900 else 20000))
    b_c = np.concatenate([np.sort(rng.choice(pool, size=x, replace=False)) for x in n])
    B = gen.from_coo(nb, ncols, b_r, b_c, rng.integers(-4, 5, b_r.size).astype(np.float64))
    # up to 40 entries of A while the row's products stay within a target that is spread over 2..32
    target = np.repeat([8, 16, 32], m // 3)[:, None]
    k = np.sort(rng.integers(0, nb, (m, 40)), axis=1)
    take = np.cumsum(n[k], axis=1) <= target
    r, c = np.nonzero(take)
    key = np.unique(r * nb + k[r, c])
    A = gen.from_coo(m, nb, key // nb, key % nb, rng.integers(-4, 5, key.size).astype(np.float64))
    assert A.nnz <= 32 * m
    used = np.unique(B.col)
    ref = oracle.spgemm(A, gen.HostCSR(nb, used.size, B.row_ptr, np.searchsorted(used, B.col).astype(np.int32), B.val))
    Ad, Bd = (spg.CSR.from_host(M, dtype=dtype) for M in (A, B))
    for policy in ["hybrid"] + (["precise"] if ncols == 900 else []):
        plan = spg.Plan(Ad, Bd, alloc_policy=policy)
        C = plan.numeric()
        bins = plan.stats()["bin_count"]
        assert min(sum(bins[2:9]), sum(bins[9:17]), sum(bins[17:33])) >= 16384, bins[:33]
        for _ in range(2):  # the product, then a values-only replay
            rp, col, val = C.to_host()
            assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, used[ref.col])
            assert np.array_equal(val.astype(np.float64), ref.val)
            C.val.zero_()
            plan.replay()
            plan.check()
