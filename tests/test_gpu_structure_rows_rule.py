"""The statistics' pass over the structure rows alone and over every row, on both
sides of the rule between them (nonzeros and rows of the structures against those
of the plan): equal to the statistics of the full per-voxel maps, and a later full
pass is not disturbed by an earlier one over few rows."""
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


@pytest.mark.parametrize("rows,fmt", [("all", "fp32"), ("all", "bf16"), ("roi", "fp16")])
@pytest.mark.parametrize("n,density", [(1500, 0.4), (60, 0.1)])
def test_both_passes(lib, rows, fmt, n, density):
    n_vox = 1201
    rp, col, D, L = phantom.random_csr(n_vox, n, density, seed=n, empty_rows=30)
    rng = np.random.default_rng(4)
    ws = rng.uniform(0.0, 2.0, (2, n)).astype(np.float32)
    for every in (0, 300, 40, 3, 1):  # every k-th row in a structure (0: none with nonzeros)
        mask = np.zeros(n_vox, np.uint32)
        if every:
            mask[::every] = rng.choice(np.array([1, 2, 3], np.uint32), len(mask[::every]))
        mask[:20] = 2  # rows without nonzeros
        with lib.Handle(0) as h:
            h.load_influence(rp, col, D, L, mask, n, fmt=fmt, rows=rows)
            for w in ws:  # statistics first: nothing of the map's pass is there yet
                edges = np.linspace(0.0, 3e3, 33).astype(np.float32)
                got = h.volume_stats([dict(quantity=q, struct_bit=b, edges=edges, fracs=[0.2, 0.9])
                                      for q in ("DOSE", "LETD") for b in (0, 1)], w)
                maps = {q: h.quantity_map(w, q) for q in ("DOSE", "LETD")}
                for (q, b), g in zip([(q, b) for q in ("DOSE", "LETD") for b in (0, 1)], got):
                    v = np.sort(maps[q][(mask >> b) & 1 == 1])[::-1]
                    assert g["n_voxels"] == len(v)
                    np.testing.assert_array_equal(g["counts"], np.histogram(v, edges)[0])
                    if len(v):
                        k = [min(max(int(np.ceil(f * len(v) - 1e-9)), 1), len(v)) for f in (0.2, 0.9)]
                        np.testing.assert_array_equal(g["at_volume"], v[np.array(k) - 1])
                    else:
                        assert np.all(np.isnan(g["at_volume"]))
