"""A single sweep over other blocks beside a begun solve that sweeps its own, in
plain launches and in a batch graph: the solve ends as if nothing had been between."""
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


@pytest.mark.parametrize("batch", [False, True])
def test_single_sweep_beside_a_solve(lib, batch):
    pl = phantom.tiny_plan()
    x = np.random.default_rng(2).uniform(0.5, 1.5, pl.n_spots).astype(np.float32)
    with lib.Handle(0) as ref:
        ref.load_plan(pl)
        swept = {n: ref.sweep_step(x, n) for n in (7, 1, 300)}
        w_ref = ref.superiorize(pl.w0, 6, pl.alpha, pl.relaxation, sweep_blocks=4)[0]
    with lib.Handle(0) as h:
        h.load_plan(pl)
        h.begin(pl.w0, pl.alpha, pl.relaxation, sweep_blocks=4, use_graphs=0)
        b = lib.Batch([h], depth=2) if batch else None
        for n in (7, 1, 300):
            if batch:
                b.iterate(2)
            else:
                h.iterate(2)
            np.testing.assert_array_equal(h.sweep_step(x, n), swept[n])
        if batch:
            b.sync()
            b.close()
        np.testing.assert_array_equal(h.end()[0], w_ref)
