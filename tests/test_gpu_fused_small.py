"""One-launch SpMV of small problems (CSR and row-sorted COO of at most 64
tiles: one cluster of blocks runs the tiles and merges the split rows behind a
cluster barrier) on both sides of that limit.

Rows of several hundred nonzeros span tiles and thread blocks, so the merge
reads partials other blocks wrote.  Integer data make every sum exact: y must
equal the oracle's bit for bit, also when the call is replayed from a CUDA
graph with other x values.
"""
import numpy as np
import pytest

from helpers import oracle_spmv
from paper_2209_07552_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TILE = 256


def _rows(m, nnz, seed):
    g = np.random.default_rng(seed)
    per = np.diff(np.concatenate(([0], np.sort(g.integers(0, nnz + 1, m - 1)), [nnz])))
    rows = np.repeat(np.arange(m), per)
    cols = np.concatenate([np.sort(g.choice(20000, k, replace=False)) for k in per])
    return I.csr_from_triplets(m, 20000, rows, cols, np.ones(rows.size))


@pytest.mark.parametrize("fmt", ["csr", "coo"])
@pytest.mark.parametrize("tiles", [2, 8, 9, 33, 63, 64, 65, 66])
def test_small_problems_match_the_oracle(fmt, tiles):
    import torch

    import paper_2209_07552_gb300 as M
    m = 40
    for P in (1, 3):
        # the plan counts (m + nnz) // tile + P + 1 tiles at most (CSR)
        nnz = max(1, (tiles - P - 1) * TILE - m) if fmt == "csr" else max(1, (tiles // P) * P * TILE)
        a, x = I.integer_twin(_rows(m, nnz, tiles), seed=tiles + P)
        y0 = np.arange(m, dtype=np.float64) - 7
        for dtype in ("f64", "f32"):
            xt = torch.float64 if dtype == "f64" else torch.float32
            A = M.DeviceMatrix.from_host(a, fmt, dtype)
            part = M.DevicePartition(A, P, tile=TILE)
            M.msrep_partition(A, part)
            ws = M.alloc_workspace(A, part)
            xd = torch.from_numpy(x).to("cuda", xt)
            for alpha, beta in ((1.0, 0.0), (2.0, 3.0)):
                y = torch.from_numpy(y0).to("cuda", xt)
                M.msrep_spmv(A, part, alpha, xd, beta, y, workspace=ws)
                want = oracle_spmv(a, fmt, x, alpha, beta, y0)
                assert np.array_equal(y.cpu().numpy().astype(np.float64), want), (P, dtype, alpha)


@pytest.mark.parametrize("fmt", ["csr", "coo"])
def test_small_problem_replayed_from_a_graph(fmt):
    import torch

    import paper_2209_07552_gb300 as M
    a, x = I.integer_twin(_rows(40, 9000, 3), seed=4)
    A = M.DeviceMatrix.from_host(a, fmt, "f64")
    part = M.DevicePartition(A, 2, tile=TILE)
    M.msrep_partition(A, part)
    ws = M.alloc_workspace(A, part)
    xd = torch.from_numpy(x).cuda()
    y = torch.empty(a.m, dtype=torch.float64, device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    M.msrep_spmv(A, part, 1.0, xd, 0.0, y, workspace=ws, stream=s)
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        M.msrep_spmv(A, part, 1.0, xd, 0.0, y, workspace=ws, stream=s)
        M.msrep_spmv(A, part, 2.0, xd, 1.0, y, workspace=ws, stream=s)
    for trial in range(2):
        xn = I.integer_twin(a, seed=50 + trial)[1]
        xd.copy_(torch.from_numpy(xn))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(y.cpu().numpy(), 3.0 * oracle_spmv(a, fmt, xn)), trial
