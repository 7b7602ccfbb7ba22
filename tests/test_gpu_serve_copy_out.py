"""y of a request of at least four vectors and 2 MB goes to the caller's buffer
through a copy kernel at the launch's end, any other y is written there by the
SpMV kernels; the copy kernel's list shares its room with the one that brings
x of one-vector requests in.  Requests on both sides of the limits, with mapped
and pageable buffers, share launches; every y equals msrep_spmm's bit for bit.
"""
import numpy as np
import pytest

from paper_2209_07552_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LIMIT = (2 << 20) // 4      # floats


def _solo(M, a, X):
    import torch
    A = M.DeviceMatrix.from_host(a, "csr", "f32")
    part = M.DevicePartition(A, max(1, -(-a.nnz // (1 << 20))))
    M.msrep_partition(A, part)
    Y = torch.full((X.shape[0], a.m), float("nan"), dtype=torch.float32, device="cuda")
    M.msrep_spmm(A, part, 1.0, torch.from_numpy(X).cuda(), 0.0, Y)
    return Y.cpu().numpy()


@pytest.mark.parametrize("pinned", [True, False])
def test_copied_and_direct_results_share_launches(pinned):
    import paper_2209_07552_gb300 as M
    ms = [LIMIT // 4, LIMIT // 4 - 1, LIMIT // 8 + 1]
    mats = [I.geometric_matrix(m, 2.5, m, np.float32) for m in ms]
    g = I.rng(61, 1)
    X = [g.uniform(-1, 1, (8, a.n)).astype(np.float32) for a in mats]
    want = [_solo(M, a, x) for a, x in zip(mats, X)]
    reqs = [(j, k) for k in (1, 3, 4, 8, 1, 5) for j in range(len(mats))]
    with M.Server(budget_bytes=4 << 30, arena_bytes=64 << 20, contexts=1,
                  max_items=len(reqs)) as S:
        ids = [S.register(a) for a in mats]
        for _ in range(2):
            tickets = []
            for j, k in reqs:
                x = X[j][:k].copy()
                y = np.full(k * mats[j].m, np.nan, np.float32)
                if pinned:
                    x, y = M.native.pinned_empty(x.shape), M.native.pinned_empty(y.shape)
                    x[:], y[:] = X[j][:k], np.nan
                tickets.append(S.submit(ids[j], x, y))
            for (j, k), t in zip(reqs, tickets):
                assert np.array_equal(S.wait(t), want[j][:k]), (j, k)
