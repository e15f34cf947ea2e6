"""GPU parity of the bin-37 rows whose products fit a CTA's registers: u_i around 513, 2,048, 4,096 and
8,192, rows of A around 256, 512 and 1,024 entries (more go to the batched kernel), results around
the first capacity and beyond it, flat and two-level widths of B, and small largest capacities
under which the row is left to the batched kernel.  Small-integer values: exact in any order."""
import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

US = (513, 600, 2047, 2048, 2049, 4095, 4096, 4097, 8191, 8192, 8193, 9000)
NAS = (20, 255, 256, 257, 511, 513, 1023, 1025)


def _matrices(ncols, distinct, seed):
    """One row of A per (u, entries of A); B rows of any length that add up to u, whose columns come
    from `distinct` columns spread over B (many equal ones) or from all of B (0)."""
    rng = np.random.default_rng(seed)
    pool = np.sort(rng.choice(ncols, size=min(distinct or ncols, ncols), replace=False)) if distinct or ncols < 1 << 20 else None
    ar, ac, br, bc, nb, i = [], [], [], [], 0, 0
    for u in US:
        for na in NAS:
            if na > u:
                continue
            # na lengths (some zero) that add up to u
            cuts = np.sort(rng.integers(0, u + 1, na - 1))
            lens = np.diff(np.concatenate([[0], cuts, [u]]))
            while (big := lens > (pool.size if pool is not None else u)).any():
                lens = np.concatenate([np.where(big, lens // 2, lens), (lens - lens // 2)[big]])
            for n in lens:
                if pool is not None:
                    c = np.sort(rng.choice(pool, size=n, replace=False))
                else:
                    c = np.unique(rng.integers(0, ncols, 2 * n + 8))
                    c = np.sort(rng.choice(c, size=n, replace=False))
                br.append(np.full(n, nb)); bc.append(c); ar.append(i); ac.append(nb)
                nb += 1
            i += 1
    b_r, b_c = np.concatenate(br), np.concatenate(bc)
    B = gen.from_coo(nb, ncols, b_r, b_c, rng.integers(-4, 5, b_r.size).astype(np.float64))
    A = gen.from_coo(i, nb, np.array(ar), np.array(ac), rng.integers(-4, 5, len(ar)).astype(np.float64))
    return A, B


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ncols,distinct", [(20000, 0), (20000, 300), (131072, 0), (131073, 3000), (4194304, 0)])
def test_small_rows_exact(oracle_mod, dtype, ncols, distinct):
    import paper_1504_05022_gb300 as spg
    from paper_1504_05022_gb300.predictor import Predictor
    A, B = _matrices(ncols, distinct, seed=ncols % 1009 + distinct)
    ref = oracle_mod.spgemm(A, B)
    Ad, Bd = (spg.CSR.from_host(M, dtype=dtype) for M in (A, B))
    learned = Predictor.load(dtype="f64" if dtype == torch.float64 else "f32").opts()
    for opts in ({}, {"initial_cap": 32}, {"smem_cap_max": 1024}, {"alloc_policy": "upper_bound"}, learned,
                 dict(learned, predictor_margin=0.01)):
        plan = spg.Plan(Ad, Bd, dense_min_u=-1, **opts)
        C = plan.numeric()
        for scale in (1.0, 3.0):  # the product, then a values-only replay with A scaled
            if scale != 1.0:
                Ad.val.mul_(scale)
                plan.replay()
            plan.check()
            rp, col, val = C.to_host()
            assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col), opts
            assert np.array_equal(val.astype(np.float64), scale * ref.val), opts
        Ad.val.div_(3.0)
        plan.free()
