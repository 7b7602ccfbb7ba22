"""Requests that queue while a launch is in flight are packed into the next
one, of at most max_items requests whatever their numbers of vectors: a burst
of one-vector and k-vector requests that passes the limit in total, but not for
either kind, takes several launches and every request is answered, bit for bit
as when it is alone.
"""
import numpy as np
import pytest

from paper_2209_07552_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_items", [1, 4, 5])
def test_mixed_burst_over_the_item_limit(max_items):
    import paper_2209_07552_gb300 as M
    big = I.rmat(scale=16, nnz=1_500_000, seed=33)
    a = I.geometric_matrix(3000, 9.0, 6, np.float32)
    g = I.rng(51, 1)
    X = g.uniform(-1, 1, (3, a.n)).astype(np.float32)
    with M.Server(budget_bytes=2 << 30, arena_bytes=8 << 20, contexts=1,
                  max_items=max_items) as S:
        bid, mid = S.register(big), S.register(a)
        alone = S.wait(S.submit(mid, X)).copy()
        before = S.stats()["launches"]
        # the single context is busy with a large request while the others queue
        hold = S.submit(bid, np.ones((8, big.n), np.float32))
        ks = [1, 2, 1, 3, 1, 2, 3, 1]
        tickets = [S.submit(mid, X[:k]) for k in ks]
        S.wait(hold)
        for k, t in zip(ks, tickets):
            assert np.array_equal(S.wait(t), alone[:k]), k
        assert S.stats()["launches"] - before >= 1 + -(-len(ks) // max_items)
