"""Block-iterative sweep at the row and column lengths where its kernels take
another split: 1, 2, 4 or 8 warps per row (mean row below 192, 512 and 1024
nonzeros), 8 or 32 lanes per column (mean column entries per block up to 12),
ragged last blocks, empty rows and rows outside every structure, 32-bit
indices.  Tolerance as for any sweep against the FP64 oracle: 2e-5 relative L2."""
import numpy as np
import pytest

import oracle
import phantom

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2509_20012_gb300 import fredopt
    return fredopt


@pytest.mark.parametrize("n_cols,density,n_blocks", [(700, 0.03, 5), (700, 0.4, 63), (901, 0.7, 2), (2003, 0.75, 7),
                                                     (130, 0.6, 200)])
@pytest.mark.parametrize("norm,index32,rows", [("all", False, "all"), ("violated", True, "roi")])
def test_sweep_splits(lib, n_cols, density, n_blocks, norm, index32, rows):
    n_vox = 331
    rp, col, D, L = phantom.random_csr(n_vox, n_cols, density, seed=n_cols, empty_rows=9)
    rng = np.random.default_rng(n_blocks)
    mask = rng.choice(np.array([0, 1, 2, 3, 4], np.uint32), n_vox)
    x = rng.uniform(0.2, 2.0, n_cols).astype(np.float32)
    d = float(np.median(oracle.forward(oracle.build_problem(rp, col, D, L, n_cols, mask, [], []), x)[0][9:]))
    cons = [dict(struct_bit=0, kind="DOSE_MIN", bound=1.1 * d, priority=1.0),
            dict(struct_bit=0, kind="DOSE_MAX", bound=1.3 * d, priority=0.7),
            dict(struct_bit=1, kind="CDL_MAX", bound=0.2 * d, priority=2.0),
            dict(struct_bit=2, kind="LETD_MAX", bound=5.0, priority=0.3),
            dict(struct_bit=1, kind="LETD_MIN", bound=6.5, priority=1.0)]
    P = oracle.build_problem(rp, col, D, L, n_cols, mask, cons, [])
    R = oracle.constraint_rows(P)
    with lib.Handle(0) as h:
        h.load_influence(rp, col, D, L, mask, n_cols, rows=rows, index32=index32)
        h.set_constraints(cons)
        w = h.sweep_step(x, n_blocks, relaxation=1.0, prio_scale=0.9, norm=norm)
    ref = oracle.block_iterative_sweep(R, x.astype(np.float64), 1.0, oracle.sweep_blocks(P, R, n_blocks),
                                       prio_scale=0.9, norm=norm)
    assert np.linalg.norm(w - ref) <= 2e-5 * np.linalg.norm(ref)
