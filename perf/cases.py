"""The performance cases: what users of the library have it compute, each one
call (or one short sequence of calls) of its public entry points.

Every case is a dict of plain values; ``kind`` names the use:

    one_launch  the one-launch multiply of a small product, result in hand
    multiply    spgemm_1d_multiply of uniform random matrices
    rmat        plan / symbolic / numeric squaring of a skewed-degree graph
    galerkin    A * P_agg, then P_agg^T * (A * P_agg), on a 7-point grid
    refresh     replay of a captured A * P_agg plan after new values of A
    outer       (R^T A) * R by the outer-product 1D algorithm
    similarity  one column chunk of A * A^T, lognormal rows, Zipf columns
    batched     a batch of independent uneven products in one graph launch
    bc          one batched betweenness sweep (masked products)
    host        a multiply whose matrices and result live in host memory

Inputs are drawn on the GPU: a case names one pattern (a graph, a grid, a set of
rows), so that its results have one size, and the seed draws the values (and
the sources of a betweenness batch).  ``exact`` recomputes the double results
with plain torch (expand, sort and add, or dense blocks), without the library.
"""
import json
import math
import os
import zlib

import torch

import paper_2408_14558_gb300 as g

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MODEL = os.path.join(ROOT, "paper_2408_14558_gb300", "models", "nnz_mlp.bin")
DEV = "cuda"


def listed():
    return [
        # The smallest calls: a product that fits L2, called again and again
        # (the 8192 x 8192 configuration with 8 entries per column).
        {"name": "one_launch_8192_f64", "kind": "one_launch", "n": 8192, "d": 8, "values": "f64", "P": 4, "b": 256},
        # The same product through the general call, as a program makes it that
        # does not know its inputs' sizes: launches and host waits count.
        {"name": "multiply_8192_f64", "kind": "multiply", "n": 8192, "d": 8, "values": "f64", "P": 4, "b": 256},
        # Set-up of one algebraic multigrid level: both Galerkin products on a
        # 128^3 grid, short columns only, 32 column blocks.
        {"name": "galerkin_128", "kind": "galerkin", "N": 128, "P": 32, "b": 2048},
        # The same level in a time loop: the patterns stay, the operator's
        # values change, the recorded pass is replayed.
        {"name": "refresh_128", "kind": "refresh", "N": 128, "P": 32, "b": 2048},
        # The right Galerkin multiplication by the outer-product algorithm.
        {"name": "outer_128", "kind": "outer", "N": 128, "P": 32, "b": 2048},
        # The headline: squaring a scale-18 R-MAT graph with weights; C has
        # about 3e9 entries.
        {"name": "rmat_262144_f64", "kind": "rmat", "n": 262144, "ef": 16, "values": "f64", "P": 16, "b": 1024,
         "split": "uniform"},
        # Weighted path counts on a graph whose size is no power of two and no
        # multiple of the blocks, with flop-balanced column blocks.
        {"name": "rmat_100003_i64", "kind": "rmat", "n": 100003, "ef": 12, "values": "i64", "P": 12, "b": 1000,
         "split": "flops"},
        # Item similarity: one of the four column chunks of A * A^T with
        # 100,000 rows, int32 in, int64 out, a nearly dense result.
        {"name": "similarity_100000_i32", "kind": "similarity", "rows": 100000, "features": 1 << 20, "cols": 25000,
         "sizing": "exact", "values": "i32", "P": 4, "b": 1024},
        # The same use at a smaller odd size, sized by the learned model.
        {"name": "similarity_30011_learned", "kind": "similarity", "rows": 30011, "features": 200003, "cols": 15005,
         "sizing": "learned", "values": "i32", "P": 3, "b": 1024},
        # Many small products at once, sizes over two decades.
        {"name": "batched_20_f64", "kind": "batched", "count": 20, "nmin": 1000, "nmax": 200000, "values": "f64"},
        # A betweenness batch: masked products, forward and backward.
        {"name": "bc_65536_1024", "kind": "bc", "n": 65536, "ef": 16, "sources": 1024, "P": 16, "b": 1024},
        # A graph squared from and to page-locked host memory.
        {"name": "host_40009_f64", "kind": "host", "n": 40009, "ef": 16, "values": "f64", "P": 16, "b": 1024,
         "chunks": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["one_launch", "multiply", "galerkin", "refresh", "outer", "rmat", "rmat", "similarity",
                       "batched", "bc", "host"])
    if kind == "one_launch":
        return {"kind": kind, "n": _log(rng, 500, 12000), "d": rng.randint(3, 16),
                "values": rng.choice(["f64", "i32", "i64"]), "P": rng.randint(1, 8), "b": _log(rng, 64, 2048)}
    if kind == "multiply":
        return {"kind": kind, "n": _log(rng, 500, 300000), "d": rng.randint(2, 24),
                "values": rng.choice(["f64", "i32", "i64"]), "P": rng.randint(1, 32), "b": _log(rng, 64, 2048)}
    if kind in ("galerkin", "refresh", "outer"):
        return {"kind": kind, "N": 2 * rng.randint(10, 64), "P": rng.randint(1, 32), "b": _log(rng, 256, 4096)}
    if kind == "rmat":
        return {"kind": kind, "n": _log(rng, 3000, 262144), "ef": rng.randint(4, 16),
                "values": rng.choice(["f64", "i64"]), "P": rng.randint(1, 24), "b": _log(rng, 256, 2048),
                "split": rng.choice(["uniform", "flops"])}
    if kind == "similarity":
        rows = _log(rng, 4000, 100000)
        return {"kind": kind, "rows": rows, "features": _log(rng, 30000, 1 << 20),
                "cols": max(1000, rows // rng.randint(4, 9)), "sizing": rng.choice(["exact", "learned"]),
                "values": rng.choice(["i32", "i32", "f64"]), "P": rng.randint(1, 8), "b": _log(rng, 256, 2048)}
    if kind == "batched":
        return {"kind": kind, "count": rng.randint(2, 20), "nmin": 1000, "nmax": _log(rng, 3000, 200000),
                "values": rng.choice(["f64", "i32"])}
    if kind == "bc":
        return {"kind": kind, "n": _log(rng, 4000, 65536), "ef": rng.randint(4, 16), "sources": _log(rng, 50, 1024),
                "P": rng.randint(1, 16), "b": _log(rng, 256, 2048)}
    return {"kind": kind, "n": _log(rng, 3000, 40009), "ef": rng.randint(4, 16), "values": rng.choice(["f64", "i64"]),
            "P": rng.randint(4, 16), "b": _log(rng, 256, 2048), "chunks": rng.randint(2, 4)}


# ------------------------------------------------------------------- inputs

class _Draws:
    """Random numbers on the GPU: the pattern's from the case, the values' from
    the seed."""

    def __init__(self, case, seed):
        self.gen, self.val = torch.Generator(device=DEV), torch.Generator(device=DEV)
        text = json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True)
        self.gen.manual_seed(zlib.crc32(text.encode()))
        self.val.manual_seed(int(seed))

    def uniform(self, n):
        return torch.rand(n, generator=self.gen, device=DEV, dtype=torch.float64)

    def integers(self, lo, hi, n):
        return torch.randint(lo, hi, (n,), generator=self.gen, device=DEV, dtype=torch.int64)

    def values(self, n, kind):
        if kind == "f64":
            return 2.0 * torch.rand(n, generator=self.val, device=DEV, dtype=torch.float64) - 1.0
        v = torch.randint(1, 5, (n,), generator=self.val, device=DEV, dtype=torch.int64)
        return v.to(torch.int32) if kind == "i32" else v


def _csc(nrows, ncols, key, vals, ptr=torch.int32):
    """CSC of the sorted, distinct keys column * nrows + row."""
    cols = torch.div(key, nrows, rounding_mode="floor")
    colptr = torch.zeros(ncols + 1, dtype=torch.int64, device=DEV)
    colptr[1:] = torch.cumsum(torch.bincount(cols, minlength=ncols), 0)
    return g.DeviceCSC(int(nrows), int(ncols), colptr.to(ptr), (key - cols * nrows).to(torch.int32), vals)


def _distinct(nrows, cols, sampler):
    """Sorted keys col * nrows + row with one distinct sampled row per entry of
    cols; a row that its column already has is drawn again."""
    key = cols * nrows + sampler(cols.numel())
    while True:
        key = torch.sort(key).values
        again = torch.nonzero(key[1:] == key[:-1]).squeeze(1) + 1
        if not again.numel():
            return key
        key[again] = torch.div(key[again], nrows, rounding_mode="floor") * nrows + sampler(again.numel())


def _uniform(n, d, values, r):
    cols = torch.arange(n, device=DEV).repeat_interleave(min(d, n))
    key = _distinct(n, cols, lambda s: r.integers(0, n, s))
    return _csc(n, n, key, r.values(key.numel(), values))


def _rmat(n, ef, values, r):
    """Symmetric R-MAT graph on n vertices (0.57, 0.19, 0.19, 0.05): self loops
    and ids >= n dropped, duplicates merged, A union A^T."""
    ne = ef * n
    row = torch.zeros(ne, dtype=torch.int64, device=DEV)
    col = torch.zeros(ne, dtype=torch.int64, device=DEV)
    for _ in range(max(1, (n - 1).bit_length())):
        u = r.uniform(ne)
        row = 2 * row + (u >= 0.76)
        col = 2 * col + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    keep = (row != col) & (row < n) & (col < n)
    row, col = row[keep], col[keep]
    key = torch.unique(torch.cat([col * n + row, row * n + col]))
    return _csc(n, n, key, r.values(key.numel(), values))


def _rmat_rows(n, d, values, r):
    """Every column has d distinct rows whose bits are 1 with probability 0.24."""
    L = max(1, (n - 1).bit_length())

    def sampler(s):
        out = torch.full((s,), n, dtype=torch.int64, device=DEV)
        while True:
            todo = torch.nonzero(out >= n).squeeze(1)
            if not todo.numel():
                return out
            x = torch.zeros(todo.numel(), dtype=torch.int64, device=DEV)
            for _ in range(L):
                x = 2 * x + (r.uniform(todo.numel()) < 0.24)
            out[todo] = x
    key = _distinct(n, torch.arange(n, device=DEV).repeat_interleave(min(d, n)), sampler)
    return _csc(n, n, key, r.values(key.numel(), values))


def _poisson(N, r):
    """7-point operator with variable coefficients on an N^3 grid (multiples of
    2^-20, so that sums of a few of them are exact)."""
    n = N ** 3
    v = torch.arange(n, device=DEV)
    x, y, z = v // (N * N), (v // N) % N, v % N
    every = torch.ones(n, dtype=torch.bool, device=DEV)
    offs = [(-N * N, x > 0), (-N, y > 0), (-1, z > 0), (0, every), (1, z < N - 1), (N, y < N - 1), (N * N, x < N - 1)]
    key = torch.stack([v * n + v + o for o, _ in offs], 1)
    valid = torch.stack([m for _, m in offs], 1)
    vals = -torch.round((1.0 + 0.5 * r.values(n * 7, "f64")) * 2 ** 20) / 2 ** 20
    vals = vals.view(n, 7)
    vals[:, 3] = 6.0 - vals[:, 3]
    return _csc(n, n, key[valid], vals[valid].contiguous())


def _aggregate(N, value):
    """(P, P^T): 2x2x2 aggregation of the N^3 grid, one entry per fine vertex."""
    M = N // 2
    v = torch.arange(N ** 3, device=DEV)
    agg = ((v // (N * N)) // 2 * M + ((v // N) % N) // 2) * M + (v % N) // 2
    key = torch.sort(agg * N ** 3 + v).values
    vals = torch.full((N ** 3,), value, dtype=torch.float64, device=DEV)
    return _csc(N ** 3, M ** 3, key, vals), _csc(M ** 3, N ** 3, v * M ** 3 + agg, vals.clone())


def _similarity(case, r):
    """A (rows x features: lognormal row lengths, Zipf(1.2) features) and the
    first `cols` columns of A^T."""
    rows, feats = case["rows"], case["features"]
    normal = torch.randn(rows, generator=r.gen, device=DEV, dtype=torch.float64)
    lens = torch.clamp(torch.round(torch.exp(math.log(50.0) - 0.5 + normal)), 1, 500).to(torch.int64)
    cdf = torch.cumsum(torch.arange(1, feats + 1, device=DEV, dtype=torch.float64) ** -1.2, 0)
    cdf /= cdf[-1].clone()
    of = torch.arange(rows, device=DEV).repeat_interleave(lens)
    key = _distinct(feats, of, lambda s: torch.clamp(torch.searchsorted(cdf, r.uniform(s), right=True), max=feats - 1))
    vals = r.values(key.numel(), case["values"])
    At = _csc(feats, rows, key, vals, torch.int64)
    row = torch.div(key, feats, rounding_mode="floor")
    order = torch.argsort((key - row * feats) * rows + row)
    A = _csc(rows, feats, ((key - row * feats) * rows + row)[order], vals[order].contiguous(), torch.int64)
    e = int(At.colptr[case["cols"]])
    B = g.DeviceCSC(feats, case["cols"], At.colptr[: case["cols"] + 1].contiguous(), At.rowidx[:e].contiguous(),
                    At.vals[:e].contiguous())
    return A, B


def _batch(case, r):
    As, Bs = [], []
    for _ in range(case["count"]):
        u = r.uniform(2).tolist()
        n = int(round(math.exp(math.log(case["nmin"]) + u[0] * math.log(case["nmax"] / case["nmin"]))))
        make = _uniform if u[1] < 0.5 else _rmat_rows
        dA, dB = r.integers(4, 33, 2).tolist()
        As.append(make(n, dA, case["values"], r))
        Bs.append(make(n, dB, case["values"], r))
    return As, Bs


def _inputs(case, seed):
    """The matrices of a case (on the GPU)."""
    r, kind = _Draws(case, seed), case["kind"]
    if kind in ("one_launch", "multiply"):
        A = _uniform(case["n"], case["d"], case["values"], r)
        return A, A
    if kind in ("rmat", "host"):
        A = _rmat(case["n"], case["ef"], case["values"], r)
        return A, A
    if kind == "bc":
        A = _rmat(case["n"], case["ef"], "f64", r)
        src = torch.randperm(case["n"], generator=r.val, device=DEV)[: case["sources"]].to(torch.int32)
        return A, src
    if kind in ("galerkin", "refresh"):
        P, PT = _aggregate(case["N"], 1.0 / math.sqrt(8.0))
        return _poisson(case["N"], r), P, PT
    if kind == "outer":
        # R^T A with entries 1/8 is exact, whatever the order of its sums
        R, RT = _aggregate(case["N"], 0.125)
        A = _poisson(case["N"], r)
        key, vals = _product(RT, A)
        return _csc(RT.nrows, A.ncols, key, vals), R
    if kind == "similarity":
        return _similarity(case, r)
    return _batch(case, r)


def _out(C):
    return {"colptr": C.colptr, "rowidx": C.rowidx, "vals": C.vals}


# ----------------------------------------------------------- prepare and run

class _Host:
    """A matrix in page-locked host memory."""

    def __init__(self, M):
        self.nrows, self.ncols = M.nrows, M.ncols
        self.colptr, self.rowidx, self.vals = (t.cpu().pin_memory() for t in (M.colptr, M.rowidx, M.vals))


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "bc":
        s["A"], s["sources"] = _inputs(case, seed)
    elif kind == "batched":
        As, Bs = _inputs(case, seed)
        s["count"], s["batch"] = len(As), g.spgemm_batch_create(As, Bs)
    elif kind == "galerkin":
        s["A"], s["B"], s["PT"] = _inputs(case, seed)
    elif kind == "refresh":
        A, P, _ = _inputs(case, seed)
        s["stream"] = torch.cuda.Stream()
        s["stream"].wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s["stream"]):
            plan = g.spgemm_plan(A, P, case["P"], case["b"])
            g.spgemm_symbolic(plan)
            s["C"] = g.spgemm_numeric(plan)
            g.spgemm_plan_capture(plan, s["C"])
            # the next step's operator, in the arrays that the plan reads
            A.vals.copy_(torch.where(A.vals > 0, 1.0, 0.5) * A.vals)
        s["plan"] = plan
    elif kind == "host":
        A, _ = _inputs(case, seed)
        plan = g.spgemm_plan(A, A, case["P"], case["b"])
        _, nnz = g.spgemm_symbolic(plan)
        g.spgemm_plan_destroy(plan)
        s["A"], s["pool"] = _Host(A), g.HostPool(16 * nnz + 8 * (case["n"] + 1) + 4096)
    else:
        s["A"], s["B"] = _inputs(case, seed)
        if kind == "one_launch":
            s["product"] = g.SmallProduct(s["A"], s["B"], case["P"], case["b"])
        elif kind == "similarity" and case["sizing"] == "learned":
            s["model"] = g.spgemm_model_load(MODEL)
    return s


def run(s):
    case = s["case"]
    kind, P, b = case["kind"], case.get("P"), case.get("b")
    if kind == "one_launch":
        return _out(s["product"].run().C())
    if kind == "multiply":
        return _out(g.spgemm_1d_multiply(s["A"], s["B"], P, b)[0])
    if kind == "rmat":
        plan = g.spgemm_plan(s["A"], s["B"], P, b,
                             split=g.SPG_SPLIT_FLOPS if case["split"] == "flops" else g.SPG_SPLIT_UNIFORM)
        g.spgemm_symbolic(plan)
        C = g.spgemm_numeric(plan)
        g.spgemm_plan_destroy(plan)
        return _out(C)
    if kind == "galerkin":
        AP = g.multiply(s["A"], s["B"], P, b)
        return {"AP": _out(AP), "PTAP": _out(g.multiply(s["PT"], AP, P, b))}
    if kind == "refresh":
        g.spgemm_plan_replay(s["plan"])
        return _out(s["C"])
    if kind == "outer":
        return _out(g.spgemm_outer_multiply(s["A"], s["B"], P, b)[0])
    if kind == "similarity":
        how = dict(sizing=g.SPG_SIZING_LEARNED, model=s["model"]) if case["sizing"] == "learned" else {}
        return _out(g.spgemm_1d_multiply(s["A"], s["B"], P, b, **how)[0])
    if kind == "batched":
        g.spgemm_batch_execute(s["batch"])
        g.spgemm_batch_status(s["batch"])
        return [g.spgemm_batch_result(s["batch"], i) for i in range(s["count"])]
    if kind == "bc":
        score, levels, _ = g.spgemm_bc_batch(s["A"], s["sources"], P, b)
        return {"bc": score, "levels": torch.tensor(levels + [0] * (64 - len(levels)))}
    return _out(g.spgemm_1d_multiply_host(s["A"], s["A"], P, b, chunks=case["chunks"], pool=s["pool"]))


def work(case):
    """Each input and each output once (4 bytes per row id, the value's width,
    the column pointers); one multiplication and one addition per product."""
    kind = case["kind"]

    def size(M):
        return sum(t.numel() * t.element_size() for t in (M.colptr, M.rowidx, M.vals))

    def product(A, B, count_inputs=True):
        plan = g.spgemm_plan(A, B)
        _, nnz = g.spgemm_symbolic(plan)
        flops = 2 * g.spgemm_plan_stats(plan)["products"]
        g.spgemm_plan_destroy(plan)
        ins = size(A) + (size(B) if B is not A else 0)
        return {"bytes": 12 * nnz + 8 * (B.ncols + 1) + (ins if count_inputs else 0), "flops": flops}
    M = _inputs(case, 0)
    if kind == "batched":
        each = [product(A, B) for A, B in zip(*M)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if kind == "bc":
        _, _, st = g.spgemm_bc_batch(M[0], M[1])
        return {"bytes": size(M[0]) + 4 * M[1].numel() + 8 * case["n"],
                "flops": 2 * (st["products_forward"] + st["products_backward"])}
    w = product(M[0], M[1])
    if kind == "galerkin":
        AP = g.multiply(M[0], M[1])
        v = product(M[2], AP, count_inputs=False)
        w = {"bytes": w["bytes"] + v["bytes"] + size(M[2]), "flops": w["flops"] + v["flops"]}
    return w


# -------------------------------------------------------------------- exact

def _expand(A, B, c0, c1):
    """(column - c0, row, value) of every product of columns c0..c1 of A * B."""
    s, e = int(B.colptr[c0]), int(B.colptr[c1])
    k = B.rowidx[s:e].to(torch.int64)
    acp = A.colptr.to(torch.int64)
    lens = acp[k + 1] - acp[k]
    entry = torch.arange(e - s, device=DEV).repeat_interleave(lens)
    at = torch.arange(entry.numel(), device=DEV) - (torch.cumsum(lens, 0) - lens)[entry] + acp[k][entry]
    cnt = B.colptr[c0 + 1:c1 + 1] - B.colptr[c0:c1]
    col = torch.arange(c1 - c0, device=DEV).repeat_interleave(cnt.to(torch.int64))
    return col[entry], A.rowidx[at].to(torch.int64), A.vals[at] * B.vals[s:e][entry]


def _product(A, B, most=1 << 26):
    """Sorted keys column * rows + row and values of A * B, by plain torch."""
    acp, bcp = A.colptr.to(torch.int64), B.colptr.to(torch.int64)
    k = B.rowidx.to(torch.int64)
    upto = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(acp[k + 1] - acp[k], 0)])[bcp]
    dense = int(upto[-1]) * 64 > A.nrows * B.ncols
    width = max(1, (1 << 28) // max(A.nrows, 1)) if dense else B.ncols
    ends, c0 = upto.tolist(), 0
    keys, vals = [], []
    while c0 < B.ncols:
        c1 = c0 + 1
        while c1 < B.ncols and c1 - c0 < width and ends[c1 + 1] - ends[c0] <= most:
            c1 += 1
        col, row, v = _expand(A, B, c0, c1)
        key = col * A.nrows + row
        if dense:
            acc = torch.zeros((c1 - c0) * A.nrows, dtype=v.dtype, device=DEV)
            hit = torch.zeros((c1 - c0) * A.nrows, dtype=torch.bool, device=DEV)
            acc.index_add_(0, key, v)
            hit[key] = True
            at = torch.nonzero(hit).squeeze(1)
            keys.append(at + c0 * A.nrows)
            vals.append(acc[at])
        else:
            at, inv = torch.unique(key, return_inverse=True)
            keys.append(at + c0 * A.nrows)
            vals.append(torch.zeros(at.numel(), dtype=v.dtype, device=DEV).index_add_(0, inv, v))
        c0 = c1
    return torch.cat(keys), torch.cat(vals)


def _values(A, B):
    return {"colptr": None, "rowidx": None, "vals": _product(A, B)[1]}


def _betweenness(A, sources):
    """Brandes' dependencies of all sources at once, on dense n x s arrays."""
    n, s = A.nrows, sources.numel()
    M = torch.sparse_csr_tensor(A.colptr.to(torch.int64), A.rowidx.to(torch.int64),
                                torch.ones(A.rowidx.numel(), dtype=torch.float64, device=DEV), (n, n))
    F = torch.zeros(n, s, dtype=torch.float64, device=DEV)
    F[sources.to(torch.int64), torch.arange(s, device=DEV)] = 1.0
    sigma, level = F.clone(), torch.where(F > 0, 0, -1).to(torch.int32)
    depth = 0
    while True:
        F = torch.where(level < 0, M @ F, 0.0)
        if not bool((F > 0).any()):
            break
        depth += 1
        level[F > 0] = depth
        sigma += F
    delta = torch.zeros_like(sigma)
    for d in range(depth, 0, -1):
        W = torch.where(level == d, (1.0 + delta) / sigma.clamp(min=1.0), 0.0)
        delta += torch.where(level == d - 1, sigma * (M @ W), 0.0)
    delta[level == 0] = 0.0
    return delta.sum(1)


def exact(case, seed):
    kind = case["kind"]
    if kind != "bc" and case.get("values", "f64") != "f64":
        return None            # whole numbers
    M = _inputs(case, seed)
    if kind == "bc":
        return {"bc": _betweenness(*M), "levels": None}
    if kind == "batched":
        return [(None, None, _product(A, B)[1]) for A, B in zip(*M)]
    if kind == "refresh":
        M[0].vals.copy_(torch.where(M[0].vals > 0, 1.0, 0.5) * M[0].vals)
    if kind == "galerkin":
        key, v = _product(M[0], M[1])
        AP = _csc(M[0].nrows, M[1].ncols, key, v)
        return {"AP": {"colptr": None, "rowidx": None, "vals": v}, "PTAP": _values(M[2], AP)}
    return _values(M[0], M[1])
