"""Edges of the k-vector tile kernel and of the low-precision sums.

The kernel keeps a tile's finished rows in a buffer of 88 rows and walks a
tile with more row ends once per 88 of them; FP64 with eight vectors takes
two passes of four.  Integer data make every sum exact, so the oracle's
product must come out bit for bit, whatever the order; on other data every
column must equal msrep_spmv of its x bit for bit.
"""
import numpy as np
import pytest

from helpers import oracle_spmv
from paper_2209_07552_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _short_rows(m, per_row, seed):
    """Rows of `per_row` nonzeros, every fifth one empty."""
    g = np.random.default_rng(seed)
    rows = np.repeat(np.array([r for r in range(m) if r % 5 != 3]), per_row)
    cols = np.concatenate([np.sort(g.choice(m, per_row, replace=False))
                           for _ in range(rows.size // per_row)])
    return I.csr_from_triplets(m, m, rows, cols, g.uniform(-1, 1, rows.size))


@pytest.mark.parametrize("k", [1, 2, 3, 8])
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("per_row", [1, 2, 5])
def test_tiles_with_many_row_ends(per_row, dtype, k):
    import torch

    import paper_2209_07552_gb300 as M
    a = _short_rows(3000, per_row, seed=per_row)
    ai, _ = I.integer_twin(a, seed=2)
    xt = torch.float64 if dtype == "f64" else torch.float32
    for tile in (256, 512, 1024):
        for alpha, beta in ((1.0, 0.0), (1.5, -0.25)):
            A = M.DeviceMatrix.from_host(a, "csr", dtype)
            part = M.DevicePartition(A, 3, tile=tile)
            M.msrep_partition(A, part)
            X = torch.from_numpy(np.stack([I.vector(a.n, 10 + v) for v in range(k)])).to("cuda", xt)
            Y0 = torch.from_numpy(np.stack([I.y_vector(a.m, 20 + v) for v in range(k)])).to("cuda", xt)
            Y = Y0.clone()
            M.msrep_spmm(A, part, alpha, X, beta, Y)
            ws = M.alloc_workspace(A, part)
            for v in range(k):
                y = Y0[v].clone()
                M.msrep_spmv(A, part, alpha, X[v], beta, y, workspace=ws)
                assert torch.equal(Y[v], y), (tile, alpha, v)
        Ai = M.DeviceMatrix.from_host(ai, "csr", dtype)
        pi = M.DevicePartition(Ai, 3, tile=tile)
        M.msrep_partition(Ai, pi)
        xi = np.stack([I.integer_twin(a, seed=30 + v)[1] for v in range(k)])
        Yi = torch.full((k, a.m), float("nan"), dtype=xt, device="cuda")
        M.msrep_spmm(Ai, pi, 1.0, torch.from_numpy(xi).to("cuda", xt), 0.0, Yi)
        for v in range(k):
            assert np.array_equal(Yi[v].cpu().numpy().astype(np.float64),
                                  oracle_spmv(ai, "csr", xi[v])), (tile, v)


@pytest.mark.parametrize("fmt", ["csr", "coo", "spmm"])
def test_low_precision_infinities_and_nan(fmt):
    """A compensated binary32 sum that meets an infinity keeps it (its
    compensation is NaN and must not reach y): +inf and -inf alone, NaN from
    their sum and from a NaN, and other rows untouched."""
    import torch

    import paper_2209_07552_gb300 as M
    n = 700
    rows, cols = [], []
    for r in range(40):                                   # short rows
        cs = [0, 10 + r, 100 + r] if r % 4 else [10 + r, 200 + r]
        rows += [r] * len(cs)
        cols += cs
    rows += [40] * 600                                    # a row over several tiles
    cols += list(range(600))
    rows += [41, 41, 42, 42, 43]
    cols += [0, 1, 1, 5, 2]
    a = I.csr_from_triplets(44, n, rows, cols, np.ones(len(rows)))
    x = np.ones(n, np.float32)
    x[0], x[1], x[2] = np.inf, -np.inf, np.nan
    A = M.DeviceMatrix.from_host(a, "coo" if fmt == "coo" else "csr", "f32")
    part = M.DevicePartition(A, 3, tile=256)
    M.msrep_partition(A, part)
    xd = torch.from_numpy(x).cuda()
    if fmt == "spmm":
        Y = torch.empty((3, a.m), dtype=torch.float32, device="cuda")
        M.msrep_spmm(A, part, 1.0, torch.stack([xd, xd, xd]), 0.0, Y)
        ys = [t.cpu().numpy() for t in Y]
    else:
        y = torch.empty(a.m, dtype=torch.float32, device="cuda")
        M.msrep_spmv(A, part, 1.0, xd, 0.0, y, workspace=M.alloc_workspace(A, part))
        ys = [y.cpu().numpy()]
    want = np.array([np.inf if r % 4 else 2.0 for r in range(40)]
                    + [np.nan, np.nan, -np.inf, np.nan], np.float32)
    for y in ys:
        assert np.array_equal(y, want, equal_nan=True), y
