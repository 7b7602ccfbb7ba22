"""Workloads the library's speed is measured on: what a user has it do, through
its public entry points, over the range of sizes, formats, value types and
matrix structures it is used for.

    listed()            the workloads themselves
    draw(rng)           one more workload of the same ranges
    prepare(case, seed) the device buffers, matrix, plan and workspace a
                        program holds before the call
    run(state)          one pass through the public entry points
    work(case)          the bytes and operations a pass cannot do without
    exact(case, seed)   what run() returns, computed in 64 bits with torch

Matrices are drawn on the GPU from the seed alone:
  uniform    m rows of exactly `per_row` distinct uniform columns
  rmat       R-MAT (a, b, c, d = .57, .19, .19, .05) on 2^scale x 2^scale with
             exactly `nnz` distinct entries, values N(0, 1)
  laplace    2D 5-point Laplacian on a grid x grid mesh (4 and -1)
  geometric  m rows, lengths Geometric(1/mu), distinct uniform columns
"""
import math
import random

import numpy as np
import torch

import paper_2209_07552_gb300 as M

DEV = "cuda"
_FMT = {"csr": M.MSREP_CSR, "csc": M.MSREP_CSC, "coo": M.MSREP_COO,
        "coo_col": M.MSREP_COO_BY_COL, "coo_any": M.MSREP_COO_UNSORTED}
_VAL = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
_BATCH_ROWS = (1e3, 2e5)   # rows of a batched or served matrix, log-uniform
_BATCH_MU = (4.0, 64.0)    # its mean row length


def _spmv(name, kind, fmt, dtype, P, alpha=1.0, beta=0.0, tile=0, **size):
    return dict({"name": name, "op": "spmv", "kind": kind, "fmt": fmt, "dtype": dtype, "P": P,
                 "tile": tile, "alpha": alpha, "beta": beta}, **size)


def listed():
    rmat20 = {"scale": 20, "nnz": 1 << 24}
    return [
        # the smallest call: one SpMV of a 2,000-row matrix inside an
        # iteration of a host-driven solver; latency is all of it
        _spmv("csr_f64_uniform_2k", "uniform", "csr", "f64", 4, m=2000, per_row=10),
        # the headline: double precision over a power-law graph, each format
        # a program may already hold it in
        _spmv("csr_f64_rmat20", "rmat", "csr", "f64", 2368, **rmat20),
        _spmv("csc_f64_rmat20", "rmat", "csc", "f64", 2368, **rmat20),
        _spmv("coo_f64_rmat20", "rmat", "coo", "f64", 2368, **rmat20),
        # a PDE stencil: short equal rows, banded columns (CG, multigrid)
        _spmv("csr_f64_laplace2048", "laplace", "csr", "f64", 2368, grid=2048),
        # graph ranking in single precision
        _spmv("csr_f32_rmat20", "rmat", "csr", "f32", 2368, **rmat20),
        # a ragged sparse layer with 16-bit weights, accumulated into y
        _spmv("csr_bf16_geometric150k", "geometric", "csr", "bf16", 148, alpha=-0.5, beta=0.75,
              m=150001, mu=23.7),
        # a smaller mesh held by columns, single precision, odd sizes
        _spmv("csc_f32_laplace1001", "laplace", "csc", "f32", 592, grid=1001),
        # eight right-hand sides at once (block solvers, personalised ranking)
        {"name": "spmm_f32_k8_rmat20", "op": "spmm", "kind": "rmat", "fmt": "csr", "dtype": "f32",
         "P": 2368, "tile": 0, "alpha": 1.0, "beta": 0.0, "k": 8, **rmat20},
        # 512 independent uneven matrices in one launch
        {"name": "batched_f32_512", "op": "batched", "dtype": "f32", "count": 512},
        # a server's burst: 64 requests of 1-8 vectors on 12 resident
        # matrices, host buffers in, host buffers out
        {"name": "serve_burst_64", "op": "serve", "count": 12, "requests": 64},
        # a matrix arrives: its partition metadata, local pointers and plan
        {"name": "partition_csr_rmat20", "op": "partition", "kind": "rmat", "fmt": "csr",
         "dtype": "f64", "P": 2368, "tile": 0, **rmat20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    pick = rng.random()
    if pick < 0.06:
        return {"op": "serve", "count": rng.randint(2, 12), "requests": rng.randint(8, 64)}
    if pick < 0.14:
        return {"op": "batched", "dtype": rng.choice(("f64", "f32", "bf16")),
                "count": _log(rng, 3, 256)}
    kind = rng.choice(("uniform", "rmat", "rmat", "laplace", "geometric"))
    if kind == "uniform":
        per_row = rng.randint(1, 40)
        size = {"m": _log(rng, 500, 200000), "per_row": per_row}
        rows = size["m"]
    elif kind == "rmat":
        scale = rng.randint(11, 20)
        size = {"scale": scale, "nnz": _log(rng, 2 << scale, 16 << scale)}
        rows = 1 << scale
    elif kind == "laplace":
        size = {"grid": _log(rng, 33, 2048)}
        rows = size["grid"] ** 2
    else:
        m, mu = _log(rng, 1000, 400000), round(rng.uniform(2.0, 64.0), 1)
        size = {"m": m, "mu": min(mu, 16e6 / m)}
        rows = m
    case = {"kind": kind, "dtype": rng.choice(("f64", "f64", "f32", "bf16")),
            "P": _log(rng, 1, min(9472, max(2, rows))),
            "tile": rng.choice((0, 0, 0, 256, 512, 1024)), **size}
    if pick < 0.22:
        return {"op": "partition", "fmt": rng.choice(tuple(_FMT)), **case}
    case["alpha"], case["beta"] = rng.choice(((1.0, 0.0), (1.0, 0.0), (-1.5, 0.75), (2.0, 0.0),
                                              (1.0, 0.5)))
    if pick < 0.42:
        return {"op": "spmm", "fmt": "csr", "k": rng.choice((1, 2, 3, 4, 5, 6, 7, 8)), **case}
    return {"op": "spmv", "fmt": rng.choice(("csr", "csr", "csc", "coo", "coo", "coo_col",
                                             "coo_any")), **case}


# --------------------------------------------------------------------------
# matrices, on the GPU, from the seed alone
# --------------------------------------------------------------------------

def _gen(seed, stream=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + stream)
    return g


def _ptr_of(counts):
    ptr = torch.zeros(counts.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=ptr[1:])
    return ptr.to(torch.int32)


def _distinct_columns(lens, n, g):
    """(ptr, col): row r holds lens[r] distinct sorted uniform columns of n,
    from the order statistics of uniforms (normalised exponential gaps)."""
    m = lens.numel()
    ptr = _ptr_of(lens)
    starts = ptr[:-1].long()
    nnz = int(ptr[-1])
    rows = torch.repeat_interleave(torch.arange(m, device=DEV), lens)
    within = torch.arange(nnz, device=DEV) - starts[rows]
    gap0 = starts + torch.arange(m, device=DEV)       # a row has one gap more than columns
    gaps = torch.empty(nnz + m, dtype=torch.float64, device=DEV).exponential_(generator=g)
    # as integers, whose running sums are the same on every run
    cs = torch.cumsum((gaps * 2**20).long() + 1, 0)
    before = torch.where(gap0 > 0, cs[(gap0 - 1).clamp_min(0)], cs.new_zeros(()))
    total = cs[gap0 + lens] - before
    u = (cs[gap0[rows] + within] - before[rows]).double() / total[rows].double()
    span = (n - lens + 1)[rows]
    col = torch.minimum((u * span).long().clamp_min(0), span - 1) + within
    return ptr, col.to(torch.int32)


def _rmat_keys(scale, nnz, g):
    ta, tab, tabc = 0.57, 0.76, 0.95
    found = None
    while found is None or found.numel() < nnz:
        want = int(nnz * 1.1) + 1024
        rows = torch.zeros(want, dtype=torch.int64, device=DEV)
        cols = torch.zeros(want, dtype=torch.int64, device=DEV)
        for _ in range(scale):
            u = torch.rand(want, generator=g, device=DEV)
            rows = rows * 2 + (u >= tab)
            cols = cols * 2 + (((u >= ta) & (u < tab)) | (u >= tabc))
        keys = (rows << scale) | cols
        found = torch.unique(keys if found is None else torch.cat((found, keys)))
    drop = found.numel() - nnz
    if drop:
        keep = torch.ones(found.numel(), dtype=torch.bool, device=DEV)
        keep[torch.randperm(found.numel(), generator=g, device=DEV)[:drop]] = False
        found = found[keep]
    return found


def _csr(case, seed):
    """m, n, ptr, col (int32) and values (float64) of the case's matrix."""
    g = _gen(seed)
    kind = case["kind"]
    if kind == "rmat":
        s = case["scale"]
        keys = _rmat_keys(s, case["nnz"], g)
        m = n = 1 << s
        ptr = _ptr_of(torch.bincount(keys >> s, minlength=m))
        col = (keys & (n - 1)).to(torch.int32)
        val = torch.randn(col.numel(), dtype=torch.float64, generator=g, device=DEV)
    elif kind == "laplace":
        q = case["grid"]
        m = n = q * q
        r = torch.arange(m, device=DEV)
        i, j = r // q, r % q
        there = torch.stack((i > 0, j > 0, i >= 0, j < q - 1, i < q - 1), 1)
        cols = r[:, None] + torch.tensor([-q, -1, 0, 1, q], device=DEV)
        ptr = _ptr_of(there.sum(1))
        col = cols[there].to(torch.int32)
        val = torch.tensor([-1.0, -1.0, 4.0, -1.0, -1.0], dtype=torch.float64, device=DEV)
        val = val.expand(m, 5)[there].contiguous()
    else:
        m = n = int(case["m"])
        if kind == "uniform":
            lens = torch.full((m,), min(case["per_row"], n), dtype=torch.int64, device=DEV)
        else:
            u = torch.rand(m, dtype=torch.float64, generator=g, device=DEV)
            p = 1.0 / max(case["mu"], 1.0 + 1e-9)
            lens = (torch.log1p(-u) / math.log1p(-p)).long().clamp(0, n - 1) + 1
        ptr, col = _distinct_columns(lens, n, g)
        val = torch.rand(col.numel(), dtype=torch.float64, generator=g, device=DEV) * 2 - 1
    return m, n, ptr, col, val


def _rows_of(ptr):
    n = ptr.numel() - 1
    return torch.repeat_interleave(torch.arange(n, dtype=torch.int32, device=DEV), torch.diff(ptr))


def _matrix(case, seed):
    """The case's matrix as the program holds it: DeviceMatrix in its format."""
    m, n, ptr, col, val = _csr(case, seed)
    fmt, dtype = case["fmt"], case["dtype"]
    v = val.to(_VAL[dtype])
    if fmt == "csr":
        return M.DeviceMatrix(_FMT[fmt], m, n, col.numel(), ptr, col, None, v, dtype)
    row = _rows_of(ptr)
    if fmt in ("csc", "coo_col"):
        order = torch.sort(col, stable=True).indices
        row, col, v = row[order], col[order], v[order]
        if fmt == "csc":
            cp = _ptr_of(torch.bincount(col, minlength=n))
            return M.DeviceMatrix(_FMT[fmt], m, n, row.numel(), cp, row, None, v, dtype)
    elif fmt == "coo_any":
        order = torch.randperm(col.numel(), generator=_gen(seed, 3), device=DEV)
        row, col, v = row[order], col[order], v[order]
    return M.DeviceMatrix(_FMT[fmt], m, n, col.numel(), None, col, row, v, dtype)


def _vectors(case, seed, m, n):
    """x (n) and y (m), or k of each one after another; U(-1, 1)."""
    t = torch.float64 if case["dtype"] == "f64" else torch.float32
    k = case.get("k")
    x = torch.rand(n if k is None else (k, n), dtype=t, generator=_gen(seed, 1), device=DEV)
    y = torch.rand(m if k is None else (k, m), dtype=t, generator=_gen(seed, 2), device=DEV)
    return x * 2 - 1, y * 2 - 1


def _batch_sizes(case):
    """Rows and mean row length of each matrix of a batch or a server: drawn
    from the count alone, so that the sizes belong to the case."""
    r = random.Random(20220918 + case["count"])
    return [(int(math.exp(r.uniform(math.log(_BATCH_ROWS[0]), math.log(_BATCH_ROWS[1])))),
             r.uniform(*_BATCH_MU)) for _ in range(case["count"])]


def _batch_matrices(case, seed):
    for i, (m, mu) in enumerate(_batch_sizes(case)):
        yield _csr({"kind": "geometric", "m": m, "mu": mu}, seed * 1031 + i)


def _batch_vector(seed, i, n, dtype):
    t = torch.float64 if dtype == "f64" else torch.float32
    return torch.rand(n, dtype=t, generator=_gen(seed * 1031 + i, 1), device=DEV) * 2 - 1


def _requests(case):
    """(matrix, k) of each request of a burst."""
    r = random.Random(20220919 + case["requests"])
    return [(r.randrange(case["count"]), r.randint(1, 8)) for _ in range(case["requests"])]


class _HostCSR:
    """A matrix in host memory, as Server.register takes it."""

    def __init__(self, m, n, ptr, col, val):
        self.m, self.n, self.nnz = m, n, col.numel()
        self.row_ptr, self.col_idx = ptr.cpu().numpy(), col.cpu().numpy()
        self.val = val.float().cpu().numpy()


class _Served:
    """A running server with its registered matrices, closed with the state."""

    def __init__(self, mats):
        self.server = M.Server(budget_bytes=8 << 30, arena_bytes=32 << 20, contexts=3)
        self.ids = [self.server.register(a) for a in mats]

    def __del__(self):
        self.server.close()


def _host_vectors(case, seed):
    sizes = _batch_sizes(case)
    return [np.random.default_rng([seed, i]).uniform(-1, 1, (k, sizes[j][0])).astype(np.float32)
            for i, (j, k) in enumerate(_requests(case))]


# --------------------------------------------------------------------------
# state and pass
# --------------------------------------------------------------------------

def prepare(case, seed):
    op = case["op"]
    if op == "batched":
        mats, xs, sizes = [], [], []
        for i, (m, n, ptr, col, val) in enumerate(_batch_matrices(case, seed)):
            mats.append(M.DeviceMatrix(M.MSREP_CSR, m, n, col.numel(), ptr, col, None,
                                       val.to(_VAL[case["dtype"]]), case["dtype"]))
            xs.append(_batch_vector(seed, i, n, case["dtype"]))
            sizes.append(m)
        y = torch.zeros(sum(sizes), dtype=xs[0].dtype, device=DEV)
        batch = M.DeviceBatch(mats, xs, list(y.split(sizes)))
        return {"op": op, "batch": batch, "y": y}
    if op == "serve":
        served = _Served([_HostCSR(*a) for a in _batch_matrices(case, seed)])
        sizes = _batch_sizes(case)
        reqs, xs, ys = [], [], []
        floats = sum(k * sizes[j][0] for j, k in _requests(case))
        arena = M.native.pinned_empty(floats)
        at = 0
        for (j, k), x in zip(_requests(case), _host_vectors(case, seed)):
            px = M.native.pinned_empty(x.shape)
            px[...] = x
            reqs.append((served.ids[j], px, arena[at:at + k * sizes[j][0]]))
            at += k * sizes[j][0]
        return {"op": op, "served": served, "requests": reqs, "y": arena}
    A = _matrix(case, seed)
    part = M.DevicePartition(A, case["P"], tile=case["tile"], local=op == "partition")
    if op == "partition":
        part.local.zero_()  # its unused end, when rows at the ends are empty
        return {"op": op, "A": A, "part": part}
    M.msrep_partition(A, part)
    x, y = _vectors(case, seed, A.m, A.n)
    s = {"op": op, "A": A, "part": part, "x": x, "y": y, "alpha": case["alpha"],
         "beta": case["beta"]}
    if op == "spmm":
        s["ws"] = torch.empty(max(256, M.msrep_spmm_workspace_size(A, part, case["k"])),
                              dtype=torch.uint8, device=DEV)
    else:
        s["ws"] = M.alloc_workspace(A, part)
    return s


def run(s):
    op = s["op"]
    if op == "spmv":
        M.msrep_spmv(s["A"], s["part"], s["alpha"], s["x"], s["beta"], s["y"], workspace=s["ws"])
        return s["y"]
    if op == "spmm":
        M.msrep_spmm(s["A"], s["part"], s["alpha"], s["x"], s["beta"], s["y"], workspace=s["ws"])
        return s["y"]
    if op == "batched":
        s["batch"].run()
        return s["y"]
    if op == "serve":
        server = s["served"].server
        tickets = [server.submit(mid, x, y) for mid, x, y in s["requests"]]
        for t in tickets:
            server.wait(t)
        return s["y"]
    part = s["part"]
    M.msrep_partition(s["A"], part)
    out = [part.start_idx, part.end_idx, part.start_major, part.end_major, part.start_flag]
    return out + [part.local] + ([] if part.local_off is None else [part.local_off])


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def _sizes(case):
    """(m, n, nnz), nnz as the distribution's mean where it is random."""
    kind = case["kind"]
    if kind == "rmat":
        return 1 << case["scale"], 1 << case["scale"], case["nnz"]
    if kind == "laplace":
        q = case["grid"]
        return q * q, q * q, 5 * q * q - 4 * q
    m = int(case["m"])
    if kind == "uniform":
        return m, m, m * min(case["per_row"], m)
    return m, m, int(m * max(case["mu"], 1.0))


def work(case):
    op = case["op"]
    if op in ("batched", "serve"):
        sizes = _batch_sizes(case)
        sv = {"f64": 8, "f32": 4, "bf16": 2}[case.get("dtype", "f32")]
        sx = 8 if sv == 8 else 4
        nnz = [m * mu for m, mu in sizes]
        if op == "batched":
            return {"bytes": sum((sv + 4) * z + 4 * (m + 1) + 2 * sx * m
                                 for (m, _), z in zip(sizes, nnz)), "flops": 2 * sum(nnz)}
        reqs = _requests(case)
        used = {j for j, _ in reqs}
        return {"bytes": sum(8 * nnz[j] + 4 * (sizes[j][0] + 1) for j in used)
                + sum(8 * k * sizes[j][0] for j, k in reqs),
                "flops": sum(2 * k * nnz[j] for j, k in reqs)}
    m, n, nnz = _sizes(case)
    fmt = case["fmt"]
    sv = {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
    sx = 8 if sv == 8 else 4
    if op == "partition":
        meta = 17 * case["P"]
        if fmt in ("csr", "csc"):
            major = m if fmt == "csr" else n
            return {"bytes": 8 * (major + 1) + 8 * case["P"] + meta, "flops": 0}
        return {"bytes": 8 * nnz + meta, "flops": 0}
    k = case.get("k", 1)
    index = 4 * nnz + 4 * (m + 1) if fmt == "csr" else 4 * nnz + 4 * (n + 1) if fmt == "csc" \
        else 8 * nnz
    vectors = sx * k * (n + m * (2 if case["beta"] else 1))
    return {"bytes": sv * nnz + index + vectors, "flops": 2 * k * nnz}


# --------------------------------------------------------------------------
# the same in 64 bits, with torch
# --------------------------------------------------------------------------

def _product(ptr, col, val, x):
    """A x in float64 for one x, the rows' products added with index_add_."""
    rows = _rows_of(ptr).long()
    y = torch.zeros(ptr.numel() - 1, dtype=torch.float64, device=DEV)
    return y.index_add_(0, rows, val * x.double()[col.long()])


def exact(case, seed):
    op = case["op"]
    if op == "partition":
        return None
    if op == "batched":
        return torch.cat([_product(ptr, col, val.to(_VAL[case["dtype"]]).double(),
                                   _batch_vector(seed, i, n, case["dtype"]))
                          for i, (m, n, ptr, col, val) in enumerate(_batch_matrices(case, seed))])
    if op == "serve":
        mats = [(ptr, col, val.float().double())
                for _, _, ptr, col, val in _batch_matrices(case, seed)]
        return np.concatenate([_product(*mats[j], torch.from_numpy(v).to(DEV)).cpu().numpy()
                               for (j, _), x in zip(_requests(case), _host_vectors(case, seed))
                               for v in x])
    m, n, ptr, col, val = _csr(case, seed)
    val = val.to(_VAL[case["dtype"]]).double()
    x, y = _vectors(case, seed, m, n)
    if op == "spmm":
        ax = torch.stack([_product(ptr, col, val, v) for v in x])
    else:
        ax = _product(ptr, col, val, x)
    return case["alpha"] * ax + (case["beta"] * y.double() if case["beta"] else 0.0)
