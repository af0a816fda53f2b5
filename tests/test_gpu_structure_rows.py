"""Volume statistics from the pass over the structure rows alone: they equal
the statistics of the full per-voxel maps bit for bit, whatever share of the
structure's voxels has influence entries (none, some, all) and whatever the
storage, row set and launch shapes."""
import numpy as np
import pytest

import phantom

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2509_20012_gb300 import fredopt
    return fredopt


@pytest.mark.parametrize("rows,fmt,shared", [("all", "fp32", False), ("all", "fp16", True), ("roi", "bf16", False)])
@pytest.mark.parametrize("where", ["empty_rows", "mixed", "all_rows"])
def test_statistics_equal_those_of_the_maps(lib, rows, fmt, shared, where):
    n_vox, n, empty = 700, 129, 90
    rp, col, D, L = phantom.random_csr(n_vox, n, 0.3, seed=3, empty_rows=empty)
    mask = np.zeros(n_vox, np.uint32)
    lo, hi = {"empty_rows": (5, 60), "mixed": (40, 333), "all_rows": (0, n_vox)}[where]
    mask[lo:hi] = 4
    mask[hi - 3:hi] |= 1
    w = np.random.default_rng(1).uniform(0.0, 2.0, n).astype(np.float32)
    fracs = [0.01, 0.3, 0.5, 0.98, 1.0]
    with lib.Handle(0) as h:
        h.load_influence(rp, col, D, L, mask, n, fmt=fmt, rows=rows, shared=shared)
        maps = {q: h.quantity_map(w, q) for q in ("DOSE", "CDL", "LETD")}
        edges = {q: np.linspace(0.0, float(m.max()) + 1.0, 41).astype(np.float32) for q, m in maps.items()}
        reqs = [dict(quantity=q, struct_bit=b, edges=edges[q], fracs=fracs) for q in maps for b in (0, 2)]
        got = h.volume_stats(reqs, w)
    for r, g in zip(reqs, got):
        v = np.sort(maps[r["quantity"]][(mask >> r["struct_bit"]) & 1 == 1])[::-1]
        assert g["n_voxels"] == len(v)
        np.testing.assert_array_equal(g["counts"], np.histogram(v, r["edges"])[0])  # no value on the last edge
        k = [min(max(int(np.ceil(f * len(v) - 1e-9 * max(1.0, f * len(v)))), 1), len(v)) for f in fracs]
        np.testing.assert_array_equal(g["at_volume"], v[np.array(k) - 1])
