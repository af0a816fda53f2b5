"""Sweep blocks that the streaming forward product takes with the rows between their
structure rows (many nonzeros, or many short rows per block), and neighbouring ones
that the sweep's own row kernel takes; structure rows alone and among others,
whole-GPU and shared launch shapes.  Tolerance as for any sweep: 2e-5 relative L2."""
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


def make(name):
    rng = np.random.default_rng(8)
    if name == "long":  # 24 million nonzeros in 17 thousand rows
        n_vox, n = 17003, 2001
        rp, col, D, L = phantom.random_csr(n_vox, n, 0.7, seed=8, empty_rows=21)
    else:  # 400 thousand rows of at most 6; "wide": the fluence does not fit shared memory
        n_vox, n = 400007, 61 if name == "short" else 60001
        c = np.sort(rng.integers(0, n, (n_vox, 6)), axis=1)
        keep = np.ones(c.shape, bool)
        keep[:, 1:] = c[:, 1:] != c[:, :-1]
        keep[:21] = False
        rp = np.zeros(n_vox + 1, np.int64)
        rp[1:] = np.cumsum(keep.sum(1))
        col = c[keep].astype(np.int32)
        D = rng.uniform(0.01, 1.0, len(col)).astype(np.float32)
        L = (D * rng.uniform(0.5, 12.0, len(col))).astype(np.float32)
    mask = rng.choice(np.array([0, 1, 2, 3], np.uint32), n_vox, p=[0.02, 0.4, 0.3, 0.28])
    x = rng.uniform(0.2, 2.0, n).astype(np.float32)
    d = float(np.median(oracle.forward(oracle.build_problem(rp, col, D, L, n, mask, [], []), x)[0][21:]))
    cons = [dict(struct_bit=0, kind="DOSE_MIN", bound=1.1 * d, priority=1.0),
            dict(struct_bit=1, kind="CDL_MAX", bound=0.2 * d, priority=2.0),
            dict(struct_bit=1, kind="LETD_MAX", bound=5.0, priority=0.3)]
    return rp, col, D, L, mask, n, x, cons


@pytest.fixture(scope="module")
def plans():
    return {name: make(name) for name in ("long", "short", "wide")}


@pytest.mark.parametrize("name,fmt,n_blocks", [("long", "fp32", 1), ("long", "fp32", 2), ("long", "bf16", 1),
                                               ("long", "fp16", 5), ("short", "fp32", 1), ("short", "fp32", 3),
                                               ("short", "bf16", 2), ("short", "fp32", 40), ("wide", "fp32", 2)])
@pytest.mark.parametrize("norm", ["all", "violated"])
def test_streamed_blocks(lib, plans, name, fmt, n_blocks, norm):
    rp, col, D, L, mask, n, x, cons = plans[name]
    out = {}
    for rows, shared in (("roi", False), ("all", True)):
        with lib.Handle(0) as h:
            h.load_influence(rp, col, D, L, mask, n, fmt=fmt, rows=rows, shared=shared)
            h.set_constraints(cons)
            out[rows] = h.sweep_step(x, n_blocks, norm=norm)
            np.testing.assert_array_equal(h.sweep_step(x, n_blocks, norm=norm), out[rows])  # deterministic
            w, *_ = h.superiorize(x, 1, 0.99, 1.0, sweep_blocks=n_blocks, cimmino_norm=norm, reductions=0)
            np.testing.assert_array_equal(w, out[rows])  # the solve's sweep, from a captured graph
    assert np.linalg.norm(out["roi"] - out["all"]) <= 2e-5 * np.linalg.norm(out["all"])
    if fmt == "fp32":
        P = oracle.build_problem(rp, col, D, L, n, mask, cons, [])
        R = oracle.constraint_rows(P)
        ref = oracle.block_iterative_sweep(R, x.astype(np.float64), 1.0, oracle.sweep_blocks(P, R, n_blocks), norm=norm)
        for got in out.values():
            assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)
