"""Row-block partitions (MSREP_PART_ROW_BLOCK) of row-sorted COO with the
bulk-copy staging kernels (MSREP_STREAM_TMA).

Every partition is cut into the same number of tiles, so row blocks of uneven
rows give tiles longer than a shared-memory stage holds; those are read from
global memory.  Integer data make every sum exact: y must equal the oracle's
bit for bit, and on other data the direct kernels' y bit for bit (both run the
same sums).
"""
import numpy as np
import pytest

import oracle as O
from helpers import gpu_spmv, oracle_spmv
from paper_2209_07552_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _uneven(m, long_every, long_len, seed):
    """Rows of one nonzero, every long_every-th of long_len."""
    g = np.random.default_rng(seed)
    lens = np.where(np.arange(m) % long_every == 0, long_len, 1)
    n = 2 * long_len
    rows = np.repeat(np.arange(m), lens)
    cols = np.concatenate([np.sort(g.choice(n, k, replace=False)) for k in lens])
    return I.csr_from_triplets(m, n, rows, cols, g.uniform(-1, 1, rows.size))


def _longest_tile(a, P, tile):
    """Nonzeros of the longest of the tiles the partitions are cut into."""
    p = O.partition_coo_row_block(I.csr_to_coo(a).row_idx, a.m, P, False)
    G = -(-(-(-a.nnz // P)) // tile)
    spans = np.asarray(p["end_idx"], np.int64) - np.asarray(p["start_idx"], np.int64) + 1
    return max((g + 1) * L // G - g * L // G for L in spans for g in range(G))


# one tile a warp, and more tiles than the grid has warps, so that long and
# short tiles follow one another through a warp's stages
@pytest.mark.parametrize("m,long_every,long_len,P", [(40, 39, 3001, 16), (20000, 97, 1003, 6000)])
@pytest.mark.parametrize("tile", [256, 512])
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
def test_row_block_tiles_longer_than_a_stage(dtype, tile, m, long_every, long_len, P):
    import paper_2209_07552_gb300 as M
    a = _uneven(m, long_every, long_len, seed=m)
    assert _longest_tile(a, P, tile) > tile + 16   # a stage's entries
    ai, xi = I.integer_twin(a, seed=3)
    y0 = np.arange(m, dtype=np.float64) % 11 - 5
    kw = dict(tile=tile, val_dtype=dtype, part_flags=M.MSREP_PART_ROW_BLOCK)
    for alpha, beta in ((1.0, 0.0), (2.0, 3.0)):
        y = gpu_spmv(ai, "coo", P, xi, alpha, beta, y0, flags=M.MSREP_STREAM_TMA, **kw)
        assert np.array_equal(y, oracle_spmv(ai, "coo", xi, alpha, beta, y0)), (alpha, beta)
    x = I.vector(a.n, 4)
    assert np.array_equal(gpu_spmv(a, "coo", P, x, flags=M.MSREP_STREAM_TMA, **kw),
                          gpu_spmv(a, "coo", P, x, **kw))
    assert M.native.msrep_device_status() == 0
