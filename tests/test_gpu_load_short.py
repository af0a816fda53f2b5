"""The CSC copy bit for bit on both sides of the rule that takes rows with fewer
than 2 entries per 1024 columns to the entry-by-entry transpose, and where that
one can go wrong: rows longer than one of its tiles (4096 entries), tiles of 64
rows, more rows per strip than it stages at a time (1024), a column that every
row holds, columns that share a hash slot, empty rows, fewer rows than strips."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2509_20012_gb300 import fredopt
    return fredopt


def lists(case):
    rng = np.random.default_rng(31)
    if case == "long_rows":
        n, rows = 70001, 900
        cols = [np.sort(rng.choice(n, 3, replace=False)) for _ in range(rows)]
        for r, k in ((0, 4096), (1, 4097), (450, 9001), (451, 8192), (899, 12289)):
            cols[r] = np.sort(rng.choice(n, k, replace=False))
    elif case == "many_rows":
        n, rows = 3000, 330000
        c = np.sort(rng.integers(0, n, (rows, 2)), axis=1)
        cols = [x[:1] if x[0] == x[1] else x for x in c]
    elif case == "shared_column":
        n, rows = 5000, 20000
        cols = [np.unique([77, 4999, *rng.integers(0, n, 3)]) for _ in range(rows)]
    elif case == "hash_slots":  # columns whose first slots are the last, the first and the second one
        n, rows = (1 << 21) + 5, 3000
        slot = (np.arange(n, dtype=np.uint64) * 2654435761 % (1 << 32)) >> 19
        c = np.flatnonzero((slot == 8191) | (slot <= 1))
        cols = [np.sort(rng.choice(c, 5, replace=False)) for _ in range(rows)]
    elif case == "few_rows":
        n, rows = 100000, 7
        cols = [np.sort(rng.choice(n, 40 * r, replace=False)) for r in range(rows)]
    elif case == "below_line":
        n, rows = 4096, 5000  # four groups
        cols = [np.sort(rng.choice(n, 7, replace=False)) for _ in range(rows)]
    else:  # at the line, with the edges of the groups in every row
        n, rows = 4097, 5000  # five groups
        cols = [np.unique([0, 1023, 1024, 2047, 2048, 4095, 4096, *rng.integers(0, n, 9)]) for _ in range(rows)]
    for r in rng.choice(rows, rows // 9, replace=False):
        if len(cols[r]) < 100:
            cols[r] = cols[r][:0]
    return n, cols


@pytest.mark.parametrize("case", ["long_rows", "many_rows", "shared_column", "hash_slots", "few_rows", "below_line",
                                  "at_line"])
@pytest.mark.parametrize("fmt,index32,rows", [("fp32", False, "all"), ("bf16", True, "roi")])
def test_csc_bit_exact(lib, case, fmt, index32, rows):
    n, cols = lists(case)
    if case == "hash_slots" and fmt != "fp32":
        pytest.skip("one format is enough for the largest table")
    lens = np.array([len(c) for c in cols])
    rp = np.zeros(len(cols) + 1, np.int64)
    rp[1:] = np.cumsum(lens)
    col = np.concatenate(cols).astype(np.int32)
    k = np.arange(len(col))
    D = (1 + k % 251).astype(np.float32)  # exact in 8 bits, whatever the row's scale
    L = (1 + k % 241).astype(np.float32)
    mask = (1 + np.arange(len(cols)) % 3 * (np.arange(len(cols)) % 5 > 0)).astype(np.uint32)
    order = np.concatenate([np.flatnonzero(lens > 0), np.flatnonzero(lens == 0)])  # every row lies in a structure
    dev = np.empty(len(cols), np.int64)
    dev[order] = np.arange(len(cols))
    row = np.repeat(dev, lens)
    at = np.argsort(col, kind="stable")
    with lib.Handle(0) as h:
        h.load_influence(rp, col, D, L, mask, n, fmt=fmt, rows=rows, index32=index32)
        cp, r, d, l = h.get_csc()
    np.testing.assert_array_equal(np.diff(cp), np.bincount(col, minlength=n))
    np.testing.assert_array_equal(r, row[at])
    np.testing.assert_array_equal(d, D[at])
    np.testing.assert_array_equal(l, L[at])
