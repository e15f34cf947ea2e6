"""Rows of A with many entries of which few select a row of B that is not empty: one product (bin 1) or
at most 32.  Every place of the selected entries, and the time of the search in long rows."""
import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _selecting(rows, nb, filled, width, seed):
    """A from (entries, selected places) per row: the places select filled rows of B, of `width` columns."""
    rng = np.random.default_rng(seed)
    full = np.sort(rng.choice(nb, size=filled, replace=False))
    is_full = np.zeros(nb, dtype=bool)
    is_full[full] = True
    ar, ac = [], []
    for i, (n, places) in enumerate(rows):
        # a window of B's rows in which just the places are full
        c, want, k = [], set(places), int(rng.integers(0, nb // 4))
        while len(c) < n:
            if is_full[k] == (len(c) in want):
                c.append(k)
            k += 1
        ar.append(np.full(n, i)); ac.append(np.array(c))
    ac = np.concatenate(ac)
    bc = np.concatenate([np.sort(rng.choice(5000, size=width, replace=False)) for _ in range(filled)])
    B = gen.from_coo(nb, 5000, np.repeat(full, width), bc, rng.integers(-4, 5, bc.size).astype(np.float64))
    A = gen.from_coo(len(rows), nb, np.concatenate(ar), ac, rng.integers(-4, 5, ac.size).astype(np.float64))
    return A, B


@pytest.mark.parametrize("policy", ["hybrid", "precise", "device"])
@pytest.mark.parametrize("entries", [1, 6, 40, 300])
def test_one_product(oracle_mod, policy, entries):
    import paper_1504_05022_gb300 as spg
    rng = np.random.default_rng(entries)
    rows = []
    for n in sorted({entries, max(1, entries - 1), entries + 3}):
        for p in {0, n - 1, n // 2, min(n - 1, 15), min(n - 1, 16), min(n - 1, 63), min(n - 1, 64), min(n - 1, 255)}:
            rows += [(n, [p])] * 3
    # one row in a launch of short ones that is long
    rows += [(2000, [int(rng.integers(0, 2000))]), (1999, [1998]), (1025, [512])]
    A, B = _selecting(rows, 60000, 30000, 1, entries)
    ref = oracle_mod.spgemm(A, B)
    assert np.all(np.diff(ref.row_ptr) == 1)
    Ad, Bd = spg.CSR.from_host(A), spg.CSR.from_host(B)
    if policy == "device":
        plan = spg.DevicePlan(Ad, Bd, ref.col.size)
        plan.run()
        C = plan.result()
    else:
        plan = spg.Plan(Ad, Bd, alloc_policy=policy)
        C = plan.numeric()
        plan.replay()
        plan.check()
    rp, col, val = C.to_host()
    assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col) and np.array_equal(val, ref.val)


@pytest.mark.parametrize("policy", ["hybrid", "precise"])
@pytest.mark.parametrize("entries", [20, 60])
def test_few_products_in_launches_of_many(oracle_mod, policy, entries):
    """20,000 rows whose bins reach the line of the thread-per-row kernels, on both sides of their line of
    A's average row."""
    import paper_1504_05022_gb300 as spg
    rng = np.random.default_rng(entries)
    nb, m = 40000, 20000
    full = rng.random(nb) < 10 / entries / 1.5
    w = np.where(full, rng.integers(1, 3, nb), 0)
    br = np.repeat(np.arange(nb), w)
    bc = rng.integers(0, 3000, br.size)
    key = np.unique(br * 3000 + bc)
    B = gen.from_coo(nb, 3000, key // 3000, key % 3000, rng.integers(-4, 5, key.size).astype(np.float64))
    key = np.unique(np.repeat(np.arange(m), entries) * nb + rng.integers(0, nb, m * entries))
    A = gen.from_coo(m, nb, key // nb, key % nb, rng.integers(-4, 5, key.size).astype(np.float64))
    ref = oracle_mod.spgemm(A, B)
    plan = spg.Plan(spg.CSR.from_host(A), spg.CSR.from_host(B), alloc_policy=policy)
    C = plan.numeric()
    plan.replay()
    plan.check()
    rp, col, val = C.to_host()
    assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col) and np.array_equal(val, ref.val)


def test_search_of_long_rows_is_wide():
    """100 rows of 200,000 entries with one product in some: the search takes 0.7 ms (13 ms by four lanes a row)."""
    import paper_1504_05022_gb300 as spg
    rng = np.random.default_rng(2)
    m, n, nb = 100, 200000, 500000
    full = np.sort(rng.choice(nb, 3, replace=False))
    ac = np.concatenate([np.sort(rng.choice(nb, n, replace=False)) for _ in range(m)])
    A = gen.from_coo(m, nb, np.repeat(np.arange(m), n), ac, np.ones(m * n))
    B = gen.from_coo(nb, nb, full, rng.integers(0, nb, 3), np.ones(3))
    Ad, Bd = spg.CSR.from_host(A), spg.CSR.from_host(B)
    best = 1e9
    for _ in range(3):
        plan = spg.Plan(Ad, Bd, alloc_policy="precise", record_timing=True)
        plan.numeric()
        torch.cuda.synchronize()
        st = plan.stats()
        best = min(best, st["kernel_ms"]["arrange"])
    assert st["bin_count"][1] > 0
    assert best < 4.0


def test_thread_per_row_only_where_rows_of_a_are_short():
    """100,000 rows of 512 entries with about 16 products: counted and filled by groups of lanes, in 3.4 times what
    stage 1 takes for the same entries (8.3 times by a thread per row)."""
    import paper_1504_05022_gb300 as spg
    g = torch.Generator(device="cuda")
    g.manual_seed(5)

    def uniform(r, n, m):
        key = torch.unique(r * n + torch.randint(0, n, (r.numel(),), device="cuda", generator=g))
        rp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
        rp[1:] = torch.cumsum(torch.bincount(key // n, minlength=m), 0)
        return spg.CSR(rp, (key % n).to(torch.int32), torch.ones(key.numel(), dtype=torch.float64, device="cuda"), (m, n))

    nb = 200000
    rows = torch.arange(nb, device="cuda")
    B = uniform(rows[torch.rand(nb, device="cuda", generator=g) < 1 / 64].repeat_interleave(2), nb, nb)

    m = 100000
    A = uniform(torch.arange(m, device="cuda").repeat_interleave(512), nb, m)
    best, bound = 1e9, 1e9
    for _ in range(4):
        plan = spg.Plan(A, B, alloc_policy="precise", record_timing=True)
        plan.numeric()
        ms = plan.stats()["kernel_ms"]
        best, bound = min(best, ms["esc"]), min(bound, ms["bound"])
    assert best < 5 * bound
