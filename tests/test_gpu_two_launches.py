"""Low-precision sums of CSR and row-sorted COO by the kernels that large
problems use: one launch for the tiles and one that merges split rows.  Problems
of at most 64 tiles otherwise run in one launch of a cluster, so the small
matrices here take more partitions than that, or one thread block a partition.
The one-launch form must give the same y, bit for bit.
"""
import numpy as np
import pytest

from helpers import gpu_spmv
from paper_2209_07552_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PER_PARTITION = 0x80      # MSREP_SCHED_PER_PARTITION
COMP_NONE = 0x20          # MSREP_COMP_NONE
# (partitions, flags): one launch; more than 64 tiles; a block a partition
ROUTES = [(3, 0), (70, 0), (3, PER_PARTITION), (70, PER_PARTITION)]


def _cancelling(length, rows):
    """Rows of (2^24, 1, -2^24) repeated: with x = 1 the row's sum is
    length / 3, and plain binary32 accumulation loses every 1."""
    pat = np.tile(np.array([2.0**24, 1.0, -(2.0**24)]), length // 3)
    return I.csr_from_triplets(rows, length, np.repeat(np.arange(rows), length),
                               np.tile(np.arange(length), rows), np.tile(pat, rows))


@pytest.mark.parametrize("fmt", ["csr", "coo"])
@pytest.mark.parametrize("length,rows", [(900, 4), (60, 40), (3, 2000)])
def test_every_row_is_compensated(fmt, length, rows):
    """Long rows, short ones, and rows of three nonzeros, most of which no tile
    or partition splits."""
    a = _cancelling(length, rows)
    for dt in ("f32", "bf16"):
        for P, flags in ROUTES:
            for tile in (256, 512):
                kw = dict(val_dtype=dt, tile=tile)
                y = gpu_spmv(a, fmt, P, np.ones(a.n), flags=flags, **kw)
                assert np.array_equal(y, np.full(rows, length / 3.0)), (dt, P, flags, tile)
        plain = gpu_spmv(a, fmt, 1, np.ones(a.n), val_dtype=dt, tile=512, flags=COMP_NONE)
        assert not np.array_equal(plain, np.full(rows, length / 3.0)), dt


@pytest.mark.parametrize("fmt", ["csr", "coo"])
def test_infinities_and_nan(fmt):
    """A compensated sum that meets an infinity keeps it, and NaN where two
    infinities of both signs or a NaN meet; other rows are untouched."""
    rows = [r for r in range(60) for _ in range(3)] + [60] * 600 + [61, 61, 62, 62, 63]
    cols = [c for r in range(60) for c in ((0 if r % 4 else 9), 10 + r, 100 + r)]
    cols += list(range(600)) + [0, 1, 1, 5, 2]
    a = I.csr_from_triplets(64, 700, rows, cols, np.ones(len(rows)))
    x = np.ones(700)
    x[0], x[1], x[2] = np.inf, -np.inf, np.nan
    want = np.array([np.inf if r % 4 else 3.0 for r in range(60)]
                    + [np.nan, np.nan, -np.inf, np.nan])
    for P, flags in ROUTES:
        y = gpu_spmv(a, fmt, P, x, val_dtype="f32", tile=256, flags=flags)
        assert np.array_equal(y, want, equal_nan=True), (P, flags)


@pytest.mark.parametrize("fmt", ["csr", "coo"])
@pytest.mark.parametrize("dt", ["f64", "f32", "bf16"])
def test_routes_agree(fmt, dt):
    """The same partitions and tiles in one launch and by two."""
    a = I.rmat(scale=10, nnz=6000, seed=9)
    x, y0 = I.vector(a.n, 1), I.y_vector(a.m, 2)
    for P in (1, 5):
        for alpha, beta in ((1.0, 0.0), (1.5, -0.5)):
            kw = dict(alpha=alpha, beta=beta, y0=y0, val_dtype=dt, tile=256)
            assert np.array_equal(gpu_spmv(a, fmt, P, x, **kw),
                                  gpu_spmv(a, fmt, P, x, flags=PER_PARTITION, **kw)), (P, alpha)
