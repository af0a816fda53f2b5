"""Rows of very small and very large values in 16-bit storage.  Scaling D and L
by 2^k and the point by 2^-k scales every step of a feasibility step or sweep by
a power of two, so the result is exactly 2^-k times the unscaled one, as long as
nothing on the way leaves the FP32 range."""
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


@pytest.mark.parametrize("fmt", ["bf16", "fp16"])
def test_steps_scale_exactly(lib, fmt):
    pl = phantom.tiny_plan()
    x = np.random.default_rng(5).uniform(0.2, 2.0, pl.n_spots).astype(np.float32)
    ref = None
    for k in (0, 70, -70):
        s = np.float32(2.0 ** k)
        with lib.Handle(0) as h:
            h.load_influence(pl.row_ptr, pl.col, pl.D * s, pl.L * s, pl.mask, pl.n_spots, fmt=fmt)
            h.set_constraints(pl.constraints)
            out = [h.feasibility_step(x / s, norm=n) * s for n in ("all", "violated")]
            out.append(h.sweep_step(x / s, 8) * s)
        ref = ref or out
        for got, want in zip(out, ref):
            assert not np.array_equal(want, x)  # the step moves the point
            np.testing.assert_array_equal(got, want, err_msg=f"2^{k}")
