"""Products of the bounds-checked build that tests/checked_cases.py is too small for: launches of 16,384
short rows (the thread-per-row kernels of every width), ranges of up to 1,024 columns by warps and by
CTAs, slices without a table of boundaries, rows of one product, the register merge at every width, and
each of them sized on the device where that form differs.  Test infrastructure, run by
tests/test_gpu_check_rows.py in a process of its own; exits non-zero at the first failure."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import ctypes  # noqa: E402

import numpy as np  # noqa: E402
import torch  # noqa: E402

import gen  # noqa: E402
import oracle  # noqa: E402
from tests import test_gpu_heavy_rows, test_gpu_long_rows_few_products, test_gpu_narrow_rows, test_gpu_slice_table  # noqa: E402


def _short(m, entries, nb, width, seed):
    """m rows of `entries` entries that select rows of B of 1..width columns: up to entries * width products."""
    rng = np.random.default_rng(seed)
    n = rng.integers(1, width + 1, nb)
    bc = np.concatenate([np.sort(rng.choice(4000, size=x, replace=False)) for x in n])
    B = gen.from_coo(nb, 4000, np.repeat(np.arange(nb), n), bc, rng.integers(-4, 5, bc.size).astype(np.float64))
    ac = (np.arange(m)[:, None] * 7 + np.arange(entries)[None, :] * 3 + rng.integers(0, 3, (m, entries))) % nb
    key = np.unique(np.repeat(np.arange(m), entries) * nb + ac.reshape(-1))
    return gen.from_coo(m, nb, key // nb, key % nb, rng.integers(-4, 5, key.size).astype(np.float64)), B


def main():
    assert os.environ.get("SPGEMM_CHECKED") == "1"
    from paper_1504_05022_gb300 import _build, _lib
    _build.build_check()
    oracle.build()
    import paper_1504_05022_gb300 as spg
    L = spg.load_library()
    assert L._name.endswith("libspgemm_check.so"), L._name
    code = ctypes.c_int64(0)

    def status():
        torch.cuda.synchronize()
        _lib.check(L.spgemm_check_status(ctypes.byref(code), 1), "spgemm_check_status")
        return code.value

    assert status() == 0
    few = test_gpu_long_rows_few_products._selecting([(n, [n // 2]) for n in (1, 9, 70, 300, 3000)] * 40, 60000, 30000, 1, 3)
    hubs = test_gpu_slice_table._hubs(300000, 3, 4000, 4)
    regs = (gen.rmat(12, 24, seed=109), gen.erdos_renyi(4096, 20, seed=110, ncols=30001))
    # (label, A, B, options of the plans, lowest bin and highest bin that must hold 16,384 rows, or None)
    cases = [
        ("net of 8", *_short(30000, 4, 3000, 2, 1), {}, (2, 8)),
        ("net of 16", *_short(30000, 5, 3000, 4, 2), {}, (9, 16)),
        ("net of 32", *_short(30000, 8, 3000, 5, 3), {}, (17, 32)),
        ("narrow rows", *test_gpu_narrow_rows._matrices(9000, 5), {"dense_min_u": 513, "dense_span": 2048}, None),
        ("heavy narrow rows", *test_gpu_heavy_rows._matrices(9000, 6, 2), {"dense_span": 1024}, None),
        ("slices without a table", hubs, hubs, {}, None),
        ("rows of one product", *few, {}, None),
        ("register merge", *regs, {"dense_min_u": -1}, None),
    ]
    for label, A, B, opts, bins in cases:
        ref = oracle.spgemm(A, B)
        Ad, Bd = spg.CSR.from_host(A), spg.CSR.from_host(B)

        def check(C, what):
            rp, col, val = C.to_host()
            assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col), f"{label} {what}"
            assert np.all(np.abs(val - ref.val) <= 1e-12 * ref.den), f"{label} {what}"
            s = status()
            print(f"{label} {what}: nnz(C) {C.nnz}, status {s}", flush=True)
            assert s == 0, f"{label} {what}: a bounds check failed at site {s}"

        for policy in ("hybrid", "precise"):
            if policy == "precise" and "dense_min_u" in opts and opts["dense_min_u"] < 0:
                continue
            plan = spg.Plan(Ad, Bd, alloc_policy=policy, **opts)
            C = plan.numeric()
            count = plan.stats()["bin_count"]
            assert bins is None or sum(count[bins[0]:bins[1] + 1]) >= 16384, (label, count)
            check(C, policy)
            plan.replay()
            plan.check()
            check(C, policy + " replay")
        dp = spg.DevicePlan(Ad, Bd, ref.col.size, dense_span=opts.get("dense_span", 0))
        dp.run()
        check(dp.result(), "device")
    print("all clean")


if __name__ == "__main__":
    main()
