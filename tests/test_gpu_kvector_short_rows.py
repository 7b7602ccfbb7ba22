"""msrep_spmm on rows of few nonzeros, whose tiles have more row ends than the
k-vector kernel's row buffer holds, and on one vector, which the SpMV kernels
take.

Rows on both sides of what the buffers hold (a tile of 1024 items with rows of
3 nonzeros has 256 ends, of 4 to 5 some 190, of 6 to 7 some 141, of one 512),
mixed with rows that span tiles and rows without nonzeros.  Every column must
equal msrep_spmv of its x bit for bit; with integer data it must equal the
oracle's product.
"""
import numpy as np
import pytest

from helpers import oracle_spmv
from paper_2209_07552_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _matrix(lens, n, seed):
    g = np.random.default_rng(seed)
    lens = np.asarray(lens)
    rows = np.repeat(np.arange(lens.size), lens)
    cols = np.concatenate([np.sort(g.choice(n, k, replace=False)) for k in lens] or [[]])
    return I.csr_from_triplets(lens.size, n, rows, cols.astype(np.int64),
                               g.uniform(-1, 1, rows.size))


def _lens(pattern, m):
    return np.resize(pattern, m)


CASES = {
    "one": _lens([1], 5000),
    "two": _lens([2], 3000),
    "three": _lens([3], 3000),
    "four_five": _lens([4, 4, 5], 3000),
    "six_seven": _lens([6, 6, 6, 7], 2000),
    # rows over several tiles and empty ones between rows of one nonzero
    "spans": np.concatenate([_lens([1], 700), [1500], _lens([1, 1, 1, 0], 900), [0] * 40, [1300],
                             _lens([1], 1111), [3]]),
}


def _compare(a, dtype, tile, P, k, alpha, beta):
    import torch

    import paper_2209_07552_gb300 as M
    xt = torch.float64 if dtype == "f64" else torch.float32
    A = M.DeviceMatrix.from_host(a, "csr", dtype)
    part = M.DevicePartition(A, P, tile=tile)
    M.msrep_partition(A, part)
    X = torch.from_numpy(np.stack([I.vector(a.n, 10 + v) for v in range(k)])).to("cuda", xt)
    Y0 = torch.from_numpy(np.stack([I.y_vector(a.m, 20 + v) for v in range(k)])).to("cuda", xt)
    Y = Y0.clone()
    M.msrep_spmm(A, part, alpha, X, beta, Y)
    ws = M.alloc_workspace(A, part)
    for v in range(k):
        y = Y0[v].clone()
        M.msrep_spmv(A, part, alpha, X[v], beta, y, workspace=ws)
        assert torch.equal(Y[v], y), (tile, P, k, alpha, v)


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("name", list(CASES))
def test_short_rows(name, dtype):
    import torch

    import paper_2209_07552_gb300 as M
    a = _matrix(CASES[name], 6000, seed=len(name))
    ai, _ = I.integer_twin(a, seed=2)
    xt = torch.float64 if dtype == "f64" else torch.float32
    Ai = M.DeviceMatrix.from_host(ai, "csr", dtype)
    for tile in (256, 512, 1024):
        for P in (1, 3):
            for k in (1, 2, 3, 8):
                for alpha, beta in ((1.0, 0.0), (1.5, -0.25)):
                    _compare(a, dtype, tile, P, k, alpha, beta)
        part = M.DevicePartition(Ai, 2, tile=tile)
        M.msrep_partition(Ai, part)
        for k in (2, 4, 8):
            xi = np.stack([I.integer_twin(a, seed=30 + v)[1] for v in range(k)])
            Y = torch.full((k, a.m), float("nan"), dtype=xt, device="cuda")
            M.msrep_spmm(Ai, part, 1.0, torch.from_numpy(xi).to("cuda", xt), 0.0, Y)
            for v in range(k):
                assert np.array_equal(Y[v].cpu().numpy().astype(np.float64),
                                      oracle_spmv(ai, "csr", xi[v])), (tile, k, v)


@pytest.mark.parametrize("mostly_short", [True, False])
def test_served_short_rows(mostly_short):
    """Matrices of short and of long rows share a server's launches."""
    import torch

    import paper_2209_07552_gb300 as M
    mats = [_matrix(CASES[n], 6000, seed=3) for n in ("one", "two", "spans")]
    mats.append(_matrix(_lens([40], 600 if mostly_short else 6000), 6000, seed=4))
    g = I.rng(71, 1)
    with M.Server(budget_bytes=2 << 30, arena_bytes=8 << 20, contexts=1) as S:
        ids = [S.register(a) for a in mats]
        X = [g.uniform(-1, 1, (8, a.n)).astype(np.float32) for a in mats]
        tickets = [(j, k, S.submit(ids[j], X[j][:k])) for k in (2, 3, 8, 1) for j in range(len(mats))]
        got = [(j, k, S.wait(t).copy()) for j, k, t in tickets]
    for j, k, y in got:
        A = M.DeviceMatrix.from_host(mats[j], "csr", "f32")
        part = M.DevicePartition(A, 1)
        M.msrep_partition(A, part)
        ws = M.alloc_workspace(A, part)
        for v in range(k):
            want = torch.empty(mats[j].m, dtype=torch.float32, device="cuda")
            M.msrep_spmv(A, part, 1.0, torch.from_numpy(X[j][v]).cuda(), 0.0, want, workspace=ws)
            assert np.array_equal(y[v], want.cpu().numpy()), (j, k, v)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("k", [1, 2, 9])
def test_y_over_x(dtype, k):
    """Y may lie over X: each pass reads its vectors before it writes."""
    import torch

    import paper_2209_07552_gb300 as M
    a, _ = I.integer_twin(_matrix(_lens([3, 9, 1], 4000), 4000, seed=5), seed=6)
    xt = torch.float64 if dtype == "f64" else torch.float32
    A = M.DeviceMatrix.from_host(a, "csr", dtype)
    part = M.DevicePartition(A, 3)
    M.msrep_partition(A, part)
    x = np.stack([I.integer_twin(a, seed=40 + v)[1] for v in range(k)])
    Z = torch.from_numpy(x).to("cuda", xt)
    M.msrep_spmm(A, part, 1.0, Z, 0.0, Z)
    for v in range(k):
        assert np.array_equal(Z[v].cpu().numpy().astype(np.float64), oracle_spmv(a, "csr", x[v])), v


@pytest.mark.parametrize("k", [1, 2, 8])
def test_no_nonzeros(k):
    import torch

    import paper_2209_07552_gb300 as M
    a = I.csr_from_triplets(700, 90, [], [], [])
    A = M.DeviceMatrix.from_host(a, "csr", "f32")
    part = M.DevicePartition(A, 2)
    M.msrep_partition(A, part)
    Y0 = torch.from_numpy(np.stack([I.y_vector(a.m, v) for v in range(k)])).to("cuda", torch.float32)
    Y = Y0.clone()
    M.msrep_spmm(A, part, 2.0, torch.ones((k, a.n), device="cuda"), -0.5, Y)
    assert torch.equal(Y, -0.5 * Y0)
