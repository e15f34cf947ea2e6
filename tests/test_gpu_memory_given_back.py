"""Memory of freed plans belongs to the whole process: an allocation elsewhere that needs it gets it
without a call to pool_trim, and trimming to a size keeps that much and waits for nothing."""
import gc

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _uniform(m, n, k, seed):
    """m rows of at most k sorted columns out of n, on the device."""
    import paper_1504_05022_gb300 as spg
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    r = torch.arange(m, device="cuda").repeat_interleave(k)
    key = torch.unique(r * n + torch.randint(0, n, (m * k,), device="cuda", generator=g))
    rp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(key // n, minlength=m), 0)
    return spg.CSR(rp, (key % n).to(torch.int32), torch.ones(key.numel(), dtype=torch.float64, device="cuda"), (m, n))


def test_freed_result_is_free_to_others():
    import paper_1504_05022_gb300 as spg
    A, B = _uniform(24000, 200000, 300, 1), _uniform(200000, 200000, 300, 2)
    gc.collect()
    torch.cuda.empty_cache()
    C = spg.spgemm(A, B)
    size = C.nnz * 12
    assert size > 16e9
    del C
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    x = torch.empty(free + size // 2, dtype=torch.uint8, device="cuda")  # raised OutOfMemoryError
    del x
    torch.cuda.empty_cache()
    assert spg.spgemm(A, B).nnz * 12 == size
    torch.cuda.synchronize()
    spg.pool_trim()


def test_trim_to_a_size():
    import paper_1504_05022_gb300 as spg
    A, B = _uniform(2000, 100000, 200, 3), _uniform(100000, 100000, 200, 4)
    torch.cuda.synchronize()
    spg.pool_trim()
    free0 = torch.cuda.mem_get_info()[0]
    C = spg.spgemm(A, B)
    size = C.nnz * 12
    del C
    torch.cuda.synchronize()
    held = free0 - torch.cuda.mem_get_info()[0]
    assert held >= size
    spg.pool_trim(keep_bytes=2 * held)
    assert free0 - torch.cuda.mem_get_info()[0] == held  # nothing to give back
    keep = held // 2
    spg.pool_trim(keep_bytes=keep)
    assert free0 - torch.cuda.mem_get_info()[0] <= keep + (64 << 20)  # pools hold memory in pieces of 32 MB
    spg.pool_trim()
    assert torch.cuda.mem_get_info()[0] >= free0 - (8 << 20)


def test_plans_freed_inside_a_capture_leave_it_valid():
    """A finaliser may run while a graph is captured: plans of other streams go, the graph stays good."""
    import paper_1504_05022_gb300 as spg
    A = _uniform(3000, 3000, 9, 6)
    side = torch.cuda.Stream()
    Cs = [spg.spgemm(A, A) for _ in range(3)]
    with torch.cuda.stream(side):
        Cs += [spg.spgemm(A, A) for _ in range(3)]
    want = Cs[0].val.clone()
    x = torch.ones(1000, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        y = x * 2
        del Cs
        y = y + 1
    graph.replay()
    torch.cuda.synchronize()
    assert y[0].item() == 3.0
    assert torch.equal(spg.spgemm(A, A).val, want)
