"""The block weights of a sweep follow the constraint table, the number of
blocks and c_cdl, through which a cDL row's norm, and with it its place in the
weights, can vanish: c_cdl^2 |L_i|^2 is 0 for c_cdl = 1e-200."""
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


N_VOX, N = 5003, 90
RP, COL, D, L = phantom.random_csr(N_VOX, N, 0.1, seed=2, empty_rows=40)
MASK = np.random.default_rng(2).choice(np.array([1, 2, 3], np.uint32), N_VOX)
X = np.random.default_rng(3).uniform(0.2, 2.0, N).astype(np.float32)
TABLES = [[dict(struct_bit=0, kind="DOSE_MAX", bound=2.0, priority=1.0),
           dict(struct_bit=1, kind="CDL_MAX", bound=0.1, priority=3.0)],
          [dict(struct_bit=0, kind="DOSE_MAX", bound=2.0, priority=0.25),
           dict(struct_bit=1, kind="CDL_MAX", bound=0.1, priority=7.0),
           dict(struct_bit=1, kind="LETD_MAX", bound=4.0, priority=0.5)]]


def reference(lib, table, c, blocks):
    """A fresh handle that has seen nothing else."""
    with lib.Handle(0) as h:
        h.load_influence(RP, COL, D, L, MASK, N)
        h.begin(X, 0.99, 1.0, c_cdl=c)
        h.set_constraints(TABLES[table])
        return h.sweep_step(X, blocks)


def test_weights_follow_every_change(lib):
    ref = {}
    with lib.Handle(0) as h:
        h.load_influence(RP, COL, D, L, MASK, N)
        c = 0.04
        for table, new_c, blocks in ((0, None, 1), (0, None, 3), (1, None, 3), (1, 1e-200, 3), (0, None, 1),
                                     (0, None, 4), (1, 0.04, 4), (1, 0.02, 4000), (0, None, 4000), (1, None, 2)):
            h.set_constraints(TABLES[table])
            if new_c is not None:
                c = new_c
                h.begin(X, 0.99, 1.0, c_cdl=c)
            for _ in range(2):
                got = h.sweep_step(X, min(blocks, lib.MAX_SWEEP_BLOCKS))
                key = (table, c, blocks)
                if key not in ref:
                    ref[key] = reference(lib, table, c, min(blocks, lib.MAX_SWEEP_BLOCKS))
                np.testing.assert_array_equal(got, ref[key], err_msg=str(key))
    assert not np.array_equal(ref[1, 0.04, 3], ref[0, 0.04, 3])


def test_solve_uses_the_weights_of_its_own_c(lib):
    with lib.Handle(0) as h:
        h.load_influence(RP, COL, D, L, MASK, N)
        h.set_constraints(TABLES[0])
        runs = [h.superiorize(X, 3, 0.99, 1.0, c_cdl=1e-200, sweep_blocks=2, reductions=0)[0] for _ in range(2)]
    np.testing.assert_array_equal(runs[0], runs[1])
