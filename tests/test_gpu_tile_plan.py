"""The tile plan of CSR and CSC partitions, entry for entry.

Up to 3072 partitions, and not too many tiles or rows, every block sums the
lengths of all partitions itself, 256 of them a row; otherwise a kernel before
it does.  A warp finds its first tile's partition and looks at the next 32.  The
cases lie on both sides of those limits, with partitions without tiles and with
nearly all of them; the offsets of local pointers can be had alone.

All entries are integers and must equal the rule's: partition i spans the
diagonals [D_i, D_i+1) of the merge path, cut into ceil(length / tile) even
stretches, whose coordinates consume a row's end before the next nonzero.
"""
import numpy as np
import pytest

from paper_2209_07552_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _sparse_ends(m, nnz, seed):
    """nnz one-nonzero rows, half among the first of m rows, half among the last."""
    g = np.random.default_rng(seed)
    half = nnz // 2
    rows = np.sort(np.concatenate([g.choice(nnz, half, replace=False),
                                   m - 1 - g.choice(nnz, nnz - half, replace=False)]))
    return I.csr_from_triplets(m, m, rows, g.integers(0, m, nnz), np.ones(nnz))


def _ragged(m, nnz, seed):
    g = np.random.default_rng(seed)
    rows = np.sort((m * g.random(nnz) ** 3).astype(np.int64))
    key = np.unique(rows * m + g.integers(0, m, nnz))
    return I.csr_from_triplets(m, m, key // m, key % m, np.ones(key.size))


def _want(ptr, nnz, P, tile):
    """(tile_off, tile_row, tile_k)"""
    ptr = np.asarray(ptr, np.int64)
    m = ptr.size - 1
    s = np.arange(P + 1, dtype=np.int64) * nnz // P
    R = np.searchsorted(ptr, s, side="right") - 1     # last row with ptr[row] <= s
    R[0], R[P] = 0, m
    D = s + R
    D[0] = 0
    G = -(-np.diff(D) // tile)
    off = np.concatenate(([0], np.cumsum(G)))
    part = np.repeat(np.arange(P), G)
    g = np.arange(off[-1]) - off[part]
    d = D[part] + g * np.diff(D)[part] // G[part]
    r = np.searchsorted(ptr + np.arange(m + 1), d, side="right") - 1
    r = np.clip(r, R[part], R[part + 1])
    return off, np.append(r, m), np.append(d - r, nnz)


def _got(part, P, m, nnz, tile):
    """The same arrays out of the plan buffer (each aligned to 256 bytes)."""
    raw = part.plan.cpu().numpy()
    up = lambda n: (n + 255) // 256 * 256
    tmax = (m + nnz) // tile + P + 1
    o = up(8 * (P + 1)) + up(4 * (P + 1))
    off = raw[o:o + 4 * (P + 1)].view(np.int32)
    o += up(4 * (P + 1))
    T = int(off[-1])
    row = raw[o:o + 4 * (T + 1)].view(np.int32)
    o += up(4 * (tmax + 1))
    return off, row, raw[o:o + 4 * (T + 1)].view(np.int32)


@pytest.mark.parametrize("name,m,nnz", [("ragged", 30000, 35500), ("ragged", 3000, 200000),
                                        ("ends", 2600000, 3000), ("ends", 40000000, 500),
                                        ("ends", 5000, 600),
                                        ("ragged", 50, 7)])
@pytest.mark.parametrize("fmt", ["csr", "csc"])
def test_tile_plan(fmt, name, m, nnz):
    import paper_2209_07552_gb300 as M
    a = (_ragged if name == "ragged" else _sparse_ends)(m, nnz, seed=m)
    ptr = a.row_ptr if fmt == "csr" else I.csr_to_csc(a).col_ptr
    A = M.DeviceMatrix.from_host(a, fmt, "f64")
    for P in (1, 2, 31, 32, 33, 255, 256, 257, 1000, 3072, 3073, 6000) if m < 10**7 else (1, 592):
        for local in (False, True):
            part = M.DevicePartition(A, P, tile=256, local=local)
            part.plan.fill_(0x7f)      # what a caller's buffer may hold
            M.msrep_partition(A, part)
            for got, want in zip(_got(part, P, m, a.nnz, 256), _want(ptr, a.nnz, P, 256)):
                assert np.array_equal(got, want), (P, local)
        off = part.local_off.cpu().numpy()
        spans = part.end_major.cpu().numpy().astype(np.int64) - part.start_major.cpu().numpy() + 2
        assert np.array_equal(off, np.concatenate(([0], np.cumsum(spans)))), P
        for plan in (part.c.plan, None):
            part.local_off.fill_(-1)
            part.c.local, part.c.plan = None, plan
            M.msrep_partition(A, part)
            assert np.array_equal(part.local_off.cpu().numpy(), off), (P, plan is None)


def test_tile_plan_of_full_last_block():
    """A number of tiles that fills its last plan block leaves the closing
    entry to a block of its own."""
    import paper_2209_07552_gb300 as M
    for tiles in (256, 512):
        m = tiles * 128
        rows = np.arange(m)
        a = I.csr_from_triplets(m, m, rows, rows, np.ones(m))
        A = M.DeviceMatrix.from_host(a, "csr", "f64")
        for P in (1, tiles):
            part = M.DevicePartition(A, P, tile=256)
            part.plan.fill_(0x7f)
            M.msrep_partition(A, part)
            got = _got(part, P, m, m, 256)
            assert got[0][-1] == tiles
            for g, w in zip(got, _want(a.row_ptr, m, P, 256)):
                assert np.array_equal(g, w), (tiles, P)
