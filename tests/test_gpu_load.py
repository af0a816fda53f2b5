"""The CSC copy that the plan load builds, bit for bit, at the sizes where the
tiled transpose can go wrong: columns at the edges of its column groups (1024
or 4096 wide), rows and columns longer than a tile, more columns than the
shared-memory histogram holds, and rows so short that the groups' starts are
found by bisection instead of a table."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2509_20012_gb300 import fredopt
    return fredopt


def pattern(case):
    rng = np.random.default_rng(23)
    if case == "group_edges":  # the same few columns in every row: runs over many tiles
        n, rows = 3073, 20000
        cols = [[5, 1023, 1024, 2047, 2048, 3071, 3072]] * rows
    elif case == "full_rows":  # every column in every row
        n, rows = 2500, 37
        cols = [np.arange(n)] * rows
    elif case == "one_column":
        n, rows = 1, 9000
        cols = [[0] if r % 7 else [] for r in range(rows)]
    elif case == "many_columns_short_rows":  # 4096-wide groups, bisection, global histogram
        n, rows = 70001, 5000
        cols = [np.sort(rng.choice(n, 1 + r % 5, replace=False)) for r in range(rows)]
        cols[17] = [4095, 4096, 65535, 65536, 70000]
    else:  # ragged rows, one of them longer than the others by far
        n, rows = 9000, 700
        cols = [np.sort(rng.choice(n, k, replace=False)) for k in rng.integers(0, 90, rows)]
        cols[351] = np.arange(0, n, 2)
    rp = np.zeros(rows + 1, np.int64)
    rp[1:] = np.cumsum([len(c) for c in cols])
    col = np.concatenate([np.asarray(c, np.int32) for c in cols])
    D = rng.uniform(0.1, 1.0, len(col)).astype(np.float32)
    L = (D * rng.uniform(1.0, 9.0, len(col))).astype(np.float32)
    return n, rp, col, D, L


@pytest.mark.parametrize("fmt", ["fp32", "bf16"])
@pytest.mark.parametrize("case", ["group_edges", "full_rows", "one_column", "many_columns_short_rows", "ragged"])
def test_csc_bit_exact_at_tile_edges(lib, case, fmt):
    n, rp, col, D, L = pattern(case)
    mask = np.ones(len(rp) - 1, np.uint32)
    lens = np.diff(rp)
    rp2 = np.zeros_like(rp)  # device order: rows with nonzeros first
    rp2[1:] = np.cumsum(np.concatenate([lens[lens > 0], lens[lens == 0]]))
    with lib.Handle(0) as h:
        h.load_influence(rp, col, D, L, mask, n, fmt=fmt)
        cp, row, gD, gL = h.get_csc()
    if fmt == "bf16":  # storage rounds each value to 8 significant bits, to nearest even
        def bf16(v):
            u = v.view(np.uint32)
            return ((u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000).astype(np.uint32).view(np.float32)
        D, L = bf16(D), bf16(L)
    ref = oracle.transpose_csr(rp2, col, n, D, L)
    for got, want in zip((cp, row, gD, gL), ref):
        np.testing.assert_array_equal(got, want)
