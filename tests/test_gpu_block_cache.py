"""Freed device blocks are kept for later calls: products of different sizes on several streams and
host threads at once get memory of their own, results outlive the plans and calls around them, and
trimming gives the kept blocks back."""
import threading

import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_threads_and_streams(oracle_mod):
    import paper_1504_05022_gb300 as spg
    cases = []
    for A, opts in ((gen.lap2d(40), {}), (gen.banded(5000, 24, 3), {}), (gen.rmat(12, 16, 7), {}),
                    (gen.erdos_renyi(9000, 9, 5), {}), (gen.rmat(12, 12, 9), {"alloc_policy": "precise"})):
        A.val[:] = (A.val * 8).round()  # small integers: exact in any order
        ref = oracle_mod.spgemm(A, A)
        cases.append((spg.CSR.from_host(A), opts, torch.from_numpy(ref.col).cuda(), torch.from_numpy(ref.val).cuda()))
    torch.cuda.synchronize()
    bad = []

    def work(k):
        try:
            st = torch.cuda.Stream()
            kept = []
            for i in range(12):
                j = (k + i) % len(cases)
                A, opts, col, val = cases[j]
                kept.append((j, spg.spgemm(A, A, stream=st, **opts)))
                if len(kept) > 3:
                    kept.pop(0)
                st.synchronize()
                for j, C in kept:  # this product and the ones before it
                    if not (torch.equal(C.col, cases[j][2]) and torch.equal(C.val, cases[j][3])):
                        bad.append((k, i, j))
        except Exception as e:  # noqa: BLE001
            bad.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad[:5]


def test_trim_returns_kept_blocks():
    import paper_1504_05022_gb300 as spg
    A = spg.CSR.from_host(gen.rmat(14, 16, seed=3))
    spg.pool_trim()
    free0 = torch.cuda.mem_get_info()[0]
    C = spg.spgemm(A, A)
    size = C.col.numel() * 12
    del C
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] < free0 - size  # kept
    spg.pool_trim()
    assert torch.cuda.mem_get_info()[0] >= free0 - (8 << 20)
