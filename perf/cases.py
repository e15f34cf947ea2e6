"""Performance cases: what a user of this library has it compute, through its public entry points.

A case is a dict of plain values.  prepare() makes its inputs on the GPU from a seed (the
structure of the random families and all values depend on it), run() is one pass and returns
the whole result, exact() is the same result in 64 bits from plain torch.

The matrices are those of the repository's generators and benchmark: 5-point and 27-point
Laplacians and their aggregation hierarchies (values perturbed, as for a variable
coefficient), R-MAT graphs, Erdos-Renyi, banded and block-diagonal matrices."""
import math

import torch

import paper_1504_05022_gb300 as spg
from paper_1504_05022_gb300.predictor import Predictor, Trainer

DEV = "cuda:0"
DTYPES = {"f64": torch.float64, "f32": torch.float32}
# R-MAT quadrant probabilities of the benchmark
RMAT_A, RMAT_B, RMAT_C = 0.57, 0.19, 0.19


def listed():
    return [
        # the smallest call: A*A of a 64 x 64 grid's 5-point Laplacian, where launches and
        # read-backs are all the time (coarse levels, unit-sized problems, interactive use)
        {"name": "lap2d_64", "kind": "product", "family": "lap2d", "n": 64, "param": 5, "dtype": "f64", "bits": 32,
         "policy": "hybrid"},
        # the set-up step of an aggregation multigrid: R*(A*P) of the 27-point operator on 64^3
        {"name": "galerkin27_64", "kind": "galerkin", "family": "lap3d27", "n": 64, "dtype": "f64", "bits": 32,
         "policy": "learned"},
        # the same step for an operator whose structure may change, both products in one CUDA
        # graph with every size on the device; 7-point operator, a grid that is no power of two
        {"name": "galerkin7_graph_80", "kind": "galerkin_graph", "family": "lap3d7", "n": 80, "dtype": "f64",
         "bits": 64},
        # time stepping: the 27-point chain's values again, structure unchanged
        {"name": "galerkin27_replay_64", "kind": "galerkin_replay", "family": "lap3d27", "n": 64, "dtype": "f64",
         "bits": 32, "policy": "hybrid"},
        # evenly sparse rows of an odd size (graph and network matrices without hubs): ~256
        # products a row, the bitonic bins
        {"name": "er_100003x16", "kind": "product", "family": "er", "n": 100003, "param": 16, "dtype": "f64",
         "bits": 32, "policy": "hybrid"},
        # a band matrix in single precision (finite elements, 1D couplings): all rows in bin 37,
        # each in a narrow column range
        {"name": "banded_50021w40_f32", "kind": "product", "family": "banded", "n": 50021, "param": 40, "dtype": "f32",
         "bits": 32, "policy": "hybrid"},
        # a mid-sized power-law graph in single precision, an odd number of rows
        {"name": "rmat_30011x8_f32", "kind": "product", "family": "rmat", "n": 30011, "param": 8, "dtype": "f32",
         "bits": 64, "policy": "hybrid"},
        # the benchmark's power-law matrix: every bin, hub rows, the learned preallocation
        {"name": "rmat_2p16x16", "kind": "product", "family": "rmat", "n": 65536, "param": 16, "dtype": "f64",
         "bits": 64, "policy": "learned"},
        # a larger graph where memory counts: counted first, then computed into an exact C
        {"name": "rmat_2p18x8_precise", "kind": "product", "family": "rmat", "n": 262144, "param": 8, "dtype": "f64",
         "bits": 64, "policy": "precise"},
        # many independent products of uneven sizes and of all families in one call
        {"name": "batch_20", "kind": "batch", "npairs": 20, "lo": 256, "hi": 65536, "dtype": "f64", "bits": 32,
         "policy": "learned"},
        # the largest: the headline benchmark (3.6 G entries of C), with the parameters that the
        # autotuner keeps for matrices of this kind
        {"name": "rmat_2p20x8", "kind": "product", "family": "rmat", "n": 1048576, "param": 8, "dtype": "f64",
         "bits": 64, "policy": "learned", "dense_min_u": 8192, "merge_miss": 2048},
        # training the row-size predictor on logged rows: loss, gradients and one Adam step
        {"name": "train_8192", "kind": "train", "batch": 8192},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product"] * 6 + ["galerkin", "galerkin_graph", "galerkin_replay", "replay", "batch", "train"])
    dtype = "f64" if rng.random() < 0.7 else "f32"
    c = {"kind": kind, "dtype": dtype, "bits": rng.choice([32, 64])}
    if kind == "train":
        return {"kind": kind, "batch": _log_int(rng, 512, 16384)}
    if kind == "batch":
        c.update(npairs=rng.randint(4, 20), lo=256, hi=_log_int(rng, 4096, 65536), policy=rng.choice(["hybrid", "learned"]))
        return c
    if kind.startswith("galerkin"):
        fam = rng.choice(["lap2d9", "lap3d7", "lap3d27"])
        g = _log_int(rng, 32, 512) if fam == "lap2d9" else _log_int(rng, 16, 80 if fam == "lap3d7" else 64)
        c.update(family=fam, n=g + (g & 1))
        if kind != "galerkin_graph":
            c["policy"] = rng.choice(["hybrid", "learned"])
        return c
    fam = rng.choice(["lap2d", "lap3d27", "er", "banded", "blockdiag", "rmat", "rmat"])
    policy = rng.choice(["hybrid", "hybrid", "learned", "learned", "upper_bound", "precise"])
    if fam == "lap2d":
        n, param = _log_int(rng, 32, 512), 5
    elif fam == "lap3d27":
        n, param = _log_int(rng, 12, 64), 27
    elif fam == "er":
        n, param = _log_int(rng, 1000, 200000), _log_int(rng, 4, 32)
    elif fam == "banded":
        n, param = _log_int(rng, 1000, 200000), _log_int(rng, 3, 64)
    elif fam == "blockdiag":
        n, param = _log_int(rng, 1000, 200000), _log_int(rng, 8, 64)
    else:
        n, param = _log_int(rng, 1000, 131072), _log_int(rng, 4, 16)
    c.update(family=fam, n=n, param=param, policy=policy)
    return c


# ---------------- inputs ----------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(n, g):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * 2.0 - 1.0


def _csr(rows, cols, vals, shape, dtype, bits):
    """CSR of sorted, unique coordinates."""
    rp = torch.zeros(shape[0] + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(rows, minlength=shape[0]), 0, out=rp[1:])
    return spg.CSR(rp.to(torch.int32 if bits == 32 else torch.int64), cols.to(torch.int32), vals.to(DTYPES[dtype]),
                   tuple(shape))


def _from_keys(r, c, n, g, shift, dtype, bits):
    """The n x n matrix with the given coordinates (duplicates merged), its rows and columns
    renumbered by cyclic shifts, with random values."""
    key = torch.unique((r + shift[0]) % n * n + (c + shift[1]) % n)
    rows = torch.div(key, n, rounding_mode="floor")
    return _csr(rows, key - rows * n, _uniform(key.numel(), g), (n, n), dtype, bits)


# The random families draw their coordinates from a generator of the case's own, and every
# seed renumbers them by shifts of its own (up to a sixteenth of the matrix): each seed has
# another structure, of the same sizes.
def _shift(n, seed, k):
    return (seed * 7919 + k * 104729) % max(1, n // 16)


def _rmat(n, avg, g, own, shift, dtype, bits):
    """avg samples a row of the 2^scale R-MAT that covers n, cut to its leading n x n block."""
    scale = max(1, math.ceil(math.log2(n)))
    m = avg << scale
    r = torch.zeros(m, dtype=torch.int64, device=DEV)
    c = torch.zeros(m, dtype=torch.int64, device=DEV)
    for lvl in range(scale):
        u = torch.rand(m, generator=own, device=DEV)
        bit = 1 << (scale - 1 - lvl)
        down = u >= RMAT_A + RMAT_B
        r += bit * down
        c += bit * (((u >= RMAT_A) & ~down) | (u >= RMAT_A + RMAT_B + RMAT_C))
    if n < 1 << scale:
        keep = (r < n) & (c < n)
        r, c = r[keep], c[keep]
    return _from_keys(r, c, n, g, shift, dtype, bits)


def _grid(family, size, g, dtype, bits):
    """A stencil operator on a size^dim grid, Dirichlet truncation, its coefficients perturbed."""
    dim = 2 if family.startswith("lap2d") else 3
    n = size ** dim
    idx = torch.arange(n, device=DEV)
    xyz = [torch.div(idx, size ** d, rounding_mode="floor") % size for d in range(dim)]
    full = family in ("lap2d9", "lap3d27")
    axis = (-1, 0, 1)
    offs = [(x, y, z) for z in (axis if dim == 3 else (0,)) for y in axis for x in axis
            if full or abs(x) + abs(y) + abs(z) <= 1]
    diag = float(len(offs) - 1)
    cols, oks, base = [], [], []
    for o in offs:  # ascending columns: z, then y, then x
        ok = torch.ones(n, dtype=torch.bool, device=DEV)
        for d in range(dim):
            ok &= (xyz[d] + o[d] >= 0) & (xyz[d] + o[d] < size)
        cols.append(idx + sum(o[d] * size ** d for d in range(dim)))
        oks.append(ok)
        base.append(diag if o == (0, 0, 0) else -1.0)
    ok = torch.stack(oks, 1).reshape(-1)
    col = torch.stack(cols, 1).reshape(-1)[ok]
    row = idx.repeat_interleave(len(offs))[ok]
    val = torch.tensor(base, dtype=torch.float64, device=DEV).repeat(n)[ok]
    return _csr(row, col, val * (1.0 + 0.1 * _uniform(val.numel(), g)), (n, n), dtype, bits)


def _aggregates(family, size, g, dtype, bits):
    """P (piecewise constant over 2^dim cells, one scaled entry a row) and R = its transpose."""
    dim = 2 if family.startswith("lap2d") else 3
    n, h = size ** dim, size // 2
    idx = torch.arange(n, device=DEV)
    agg = torch.zeros(n, dtype=torch.int64, device=DEV)
    for d in range(dim):
        agg += torch.div(torch.div(idx, size ** d, rounding_mode="floor") % size, 2, rounding_mode="floor") * h ** d
    val = 1.0 + 0.1 * _uniform(n, g)
    P = _csr(idx, agg, val, (n, h ** dim), dtype, bits)
    order = torch.argsort(agg, stable=True)
    return P, _csr(agg[order], order, val[order], (h ** dim, n), dtype, bits)


def _matrix(family, n, param, g, dtype, bits, own=1, shift=(0, 0)):
    if family in ("lap2d", "lap2d9", "lap3d7", "lap3d27"):
        return _grid(family, n, g, dtype, bits)
    if family == "rmat":
        return _rmat(n, param, g, _gen(own), shift, dtype, bits)
    if family == "er":
        rows = torch.arange(n, device=DEV).repeat_interleave(param)
        cols = torch.randint(0, n, (n * param,), generator=_gen(own), device=DEV)
        return _from_keys(rows, cols, n, g, shift, dtype, bits)
    rows = torch.arange(n, device=DEV)[:, None]
    if family == "banded":
        cols = rows + torch.arange(-(param // 2), param - param // 2, device=DEV)[None, :]
        ok = (cols >= 0) & (cols < n)
    else:  # blockdiag: dense param x param blocks, the last one cut
        cols = rows - rows % param + torch.arange(param, device=DEV)[None, :]
        ok = cols < n
    rows = rows.expand_as(cols)[ok]
    return _csr(rows, cols[ok], _uniform(rows.numel(), g), (n, n), dtype, bits)


FAMILIES = ("banded", "blockdiag", "er", "rmat")


def _pairs(case, g, seed):
    """Sizes spread over the logarithm of [lo, hi], the families in turn, 4 to 32 entries a row."""
    As, Bs = [], []
    for i in range(case["npairs"]):
        n = int(case["lo"] * (case["hi"] / case["lo"]) ** ((i + 0.5) / case["npairs"]))
        avg = 4 + (11 * i) % 29
        inner = _shift(n, seed, i + 1)
        As.append(_matrix(FAMILIES[i % 4], n, avg, g, case["dtype"], case["bits"], 2 * i + 1, (_shift(n, seed, i), inner)))
        Bs.append(_matrix(FAMILIES[i % 4], n, avg, g, case["dtype"], case["bits"], 2 * i + 2, (inner, _shift(n, seed, i + 2))))
    return As, Bs


def _opts(case):
    """Plan options as a user gives them; the learned policy with the committed weights."""
    if case["policy"] == "learned":
        o = Predictor.load(dtype=case["dtype"]).opts()
    else:
        o = {"alloc_policy": case["policy"]}
    for k in ("dense_min_u", "merge_miss"):
        if k in case:
            o[k] = case[k]
    return o


def _new_values(mats, g):
    """Other values of the same structure and sign pattern, in place (what a time step does)."""
    for M in mats:
        M.val.mul_((1.0 + 0.25 * _uniform(M.nnz, g)).to(M.val.dtype))


def _inputs(case, seed):
    g = _gen(seed)
    if case["kind"] == "batch":
        As, Bs = _pairs(case, g, seed)
        return {"A": As, "B": Bs}
    if case["kind"].startswith("galerkin"):
        A = _grid(case["family"], case["n"], g, case["dtype"], case["bits"])
        P, R = _aggregates(case["family"], case["n"], g, case["dtype"], case["bits"])
        return {"R": R, "A": A, "P": P, "g": g}
    if case["kind"] == "train":
        n = case["batch"]
        # features are logarithms of row and column counts; the labels a noisy function of them
        X = torch.rand((n, 8), generator=g, device=DEV) * torch.tensor([10., 18., 8., 8., 8., 4., 20., 20.], device=DEV)
        y = (X[:, 1] * (0.6 + 0.4 * torch.rand(n, generator=g, device=DEV))).contiguous()
        cls = torch.clamp(torch.ceil(y), 0, 15).to(torch.int32)
        p = torch.randn(1921, generator=g, device=DEV) * 0.25
        p[1905:1913] = X.mean(0)
        p[1913:] = X.std(0) + 0.1
        return {"X": X.contiguous(), "cls": cls, "y": y, "params": p}
    k = _shift(case["n"], seed, 0)
    return {"A": _matrix(case["family"], case["n"], case["param"], g, case["dtype"], case["bits"], 1, (k, k)), "g": g}


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    s["kind"] = kind
    if kind == "train":
        s["trainer"] = Trainer(s["params"], lr=3e-3)
        return s
    if kind == "galerkin_graph":
        # room for the results: a row of A*P holds at most the operator's row, and every coarse
        # row reaches at most its 3^dim neighbours
        dim = 2 if case["family"].startswith("lap2d") else 3
        s["stream"] = torch.cuda.Stream(DEV)
        torch.cuda.synchronize()
        s["ap"], s["rap"], s["graph"] = spg.galerkin_device(s["R"], s["A"], s["P"], s["A"].nnz,
                                                            3 ** dim * s["R"].nrows, s["stream"])
        return s
    s["opts"] = _opts(case)
    if kind in ("galerkin_replay", "replay"):
        s["stream"] = torch.cuda.Stream(DEV)
        torch.cuda.synchronize()
        if kind == "replay":
            plan = spg.Plan(s["A"], s["A"], stream=s["stream"], **s["opts"])
            s["C"] = plan.numeric()
            s["graph"] = spg.ReplayGraph([plan])
            mats = [s["A"]]
        else:
            s["C"], p1, p2 = spg.galerkin(s["R"], s["A"], s["P"], stream=s["stream"], **s["opts"])
            s["graph"] = spg.ReplayGraph([p1, p2])
            mats = [s["R"], s["A"], s["P"]]
        torch.cuda.synchronize()
        _new_values(mats, s["g"])
        torch.cuda.synchronize()
    return s


def _out(C):
    return [C.row_ptr, C.col, C.val]


def run(s):
    kind = s["kind"]
    if kind == "product":
        return _out(spg.spgemm(s["A"], s["A"], **s["opts"]))
    if kind == "galerkin":
        return _out(spg.galerkin(s["R"], s["A"], s["P"], **s["opts"])[0])
    if kind == "galerkin_graph":
        s["graph"].launch()
        return _out(s["rap"].result())
    if kind in ("galerkin_replay", "replay"):
        s["graph"].launch()
        return _out(s["C"])
    if kind == "batch":
        return [_out(C) for C in spg.spgemm_batched(s["A"], s["B"], **s["opts"])]
    t = s["trainer"]
    loss = t.step(s["X"], s["cls"], s["y"])
    return {"loss": loss, "grad": t.grad, "params": t.params}


# ---------------- the work of a pass ----------------

def _products(A, B):
    rp = B.row_ptr.to(torch.int64)
    return int((rp[1:] - rp[:-1])[A.col.long()].sum())


def _bytes(M, rows=True):
    return M.val.numel() * (4 + M.val.element_size()) + (M.row_ptr.numel() * M.row_ptr.element_size() if rows else 0)


def work(case):
    if case["kind"] == "train":
        n, macs = case["batch"], 8 * 32 + 32 * 32 + 32 * 17
        # forward, gradients of the weights, and of the activations (not of the features)
        return {"bytes": 40 * n + 4 * 1905 * 8, "flops": 2 * n * (3 * macs - 8 * 32)}
    s = prepare(case, 0)
    kind = case["kind"]
    if kind == "batch":
        prods = sum(_products(a, b) for a, b in zip(s["A"], s["B"]))
        C = spg.spgemm_batched(s["A"], s["B"], **s["opts"])
        return {"bytes": sum(_bytes(M) for M in s["A"] + s["B"] + C), "flops": 2 * prods}
    if kind.startswith("galerkin"):
        AP = spg.spgemm(s["A"], s["P"])
        Ac = spg.spgemm(s["R"], AP)
        prods = _products(s["A"], s["P"]) + _products(s["R"], AP)
        if kind == "galerkin_replay":  # Ac's columns and row pointers are in place: only its values are written
            return {"bytes": sum(_bytes(s[k]) for k in "RAP") + Ac.val.numel() * Ac.val.element_size(), "flops": 2 * prods}
        return {"bytes": sum(_bytes(s[k]) for k in "RAP") + _bytes(Ac), "flops": 2 * prods}
    A = s["A"]
    prods = _products(A, A)
    if kind == "replay":
        return {"bytes": _bytes(A) + s["C"].val.numel() * s["C"].val.element_size(), "flops": 2 * prods}
    C = spg.spgemm(A, A, **s["opts"])
    return {"bytes": _bytes(A) + _bytes(C), "flops": 2 * prods}


# ---------------- the same results in 64 bits ----------------

def _coo64(M):
    rp = M.row_ptr.to(torch.int64)
    return rp, M.col.to(torch.int64), M.val.to(torch.float64)


def _product64(A, B, ncols, chunk=1 << 27):
    """C = A*B of (row_ptr, col, val) triples: the products of a block of rows, sorted and summed."""
    arp, ac, av = A
    brp, bc, bv = B
    blen = brp[1:] - brp[:-1]
    ends = torch.zeros(ac.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(blen[ac], 0, out=ends[1:])
    row_end = ends[arp]  # products before each row
    host = row_end.cpu()
    m = arp.numel() - 1
    counts = torch.zeros(m, dtype=torch.int64, device=DEV)
    cols, vals, r0 = [], [], 0
    while r0 < m:
        r1 = int(torch.searchsorted(host, host[r0] + chunk, right=True)) - 1
        r1 = min(m, max(r1, r0 + 1))
        e0, e1 = int(arp[r0]), int(arp[r1])
        k = ac[e0:e1]
        ln = blen[k]
        tot = int(host[r1] - host[r0])
        if tot:
            ent = torch.repeat_interleave(torch.arange(e1 - e0, device=DEV), ln, output_size=tot)
            q = torch.arange(tot, device=DEV) - (ends[e0:e1] - ends[e0])[ent] + brp[k][ent]
            er = torch.repeat_interleave(torch.arange(r1 - r0, device=DEV), arp[r0 + 1:r1 + 1] - arp[r0:r1],
                                         output_size=e1 - e0)
            v = av[e0:e1][ent] * bv[q]
            key = er[ent] * ncols + bc[q]
            del ent, q
            key, order = torch.sort(key)
            v = v[order]
            del order
            key, inv = torch.unique_consecutive(key, return_inverse=True)
            s = torch.zeros(key.numel(), dtype=torch.float64, device=DEV).index_add_(0, inv, v)
            del inv, v
            rr = torch.div(key, ncols, rounding_mode="floor")
            counts[r0:r1] = torch.bincount(rr, minlength=r1 - r0)
            cols.append(key - rr * ncols)
            vals.append(s)
        r0 = r1
    rp = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=rp[1:])
    z = torch.zeros(0, device=DEV)
    return rp, torch.cat(cols) if cols else z.long(), torch.cat(vals) if vals else z.double()


def exact(case, seed):
    if case["kind"] == "product" and case["family"] == "rmat" and case["n"] > 1 << 18:
        return None  # 6 G products: sorting them takes too long
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "train":
        return _train64(s)
    if kind == "batch":
        return [[None, None, _product64(_coo64(a), _coo64(b), b.ncols)[2]] for a, b in zip(s["A"], s["B"])]
    if kind.startswith("galerkin"):
        mats = [s["R"], s["A"], s["P"]]
        if kind == "galerkin_replay":
            _new_values(mats, s["g"])
        R, A, P = (_coo64(M) for M in mats)
        nc = s["P"].ncols
        return [None, None, _product64(R, _product64(A, P, nc), nc)[2]]
    A = s["A"]
    if kind == "replay":
        _new_values([A], s["g"])
    A64 = _coo64(A)
    return [None, None, _product64(A64, A64, A.ncols)[2]]


def _train64(s):
    """Summed cross-entropy + half squared error, its gradients, and the first Adam step."""
    p = s["params"].double().requires_grad_(True)
    X = s["X"].double()
    w1, b1 = p[:256].view(32, 8), p[256:288]
    w2, b2 = p[288:1312].view(32, 32), p[1312:1344]
    w3, b3 = p[1344:1888].view(17, 32), p[1888:1905]
    h = (X - s["params"][1905:1913].double()) / s["params"][1913:].double()
    h = torch.relu(h @ w1.t() + b1)
    h = torch.relu(h @ w2.t() + b2)
    o = h @ w3.t() + b3
    loss = torch.nn.functional.cross_entropy(o[:, :16], s["cls"].long(), reduction="sum")
    loss = loss + 0.5 * ((o[:, 16] - s["y"].double()) ** 2).sum()
    loss.backward()
    grad = p.grad[:1905]
    gs = grad / X.shape[0]
    new = s["params"].double().clone()
    new[:1905] -= 3e-3 * gs / (gs.abs() + 1e-8)
    return {"loss": loss.detach().reshape(1), "grad": grad, "params": new}
