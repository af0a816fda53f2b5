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


@pytest.mark.parametrize("fmt", ["bf16", "fp16"])
def test_coefficients_at_the_edges_of_the_fp32_range(lib, fmt):
    """One nonzero per row: the step's change of each spot is the row's coefficient times
    the stored value, (b - v) / d / W, for values d from 2^-124 to 2^120 and points x = 1 / d
    for which it stays in the FP32 range, so unscaled coefficients from far below to far
    above it.  (FP16 storage holds d as 2^13 to 2^14 times a scale, and the FP32 product
    with x must not overflow: from 2^-108 on.)"""
    exps = np.arange(-124 if fmt == "bf16" else -108, 124, 4)
    n = len(exps)
    d = (1.5 * 2.0 ** exps).astype(np.float32)  # one value per row, exact in 16 bits
    x = (2.0 ** -exps.astype(np.float64)).astype(np.float32)
    rp, col = np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32)
    with lib.Handle(0) as h:
        h.load_influence(rp, col, d, d, np.ones(n, np.uint32), n, fmt=fmt)
        h.set_constraints([dict(struct_bit=0, kind="DOSE_MIN", bound=2.0, priority=1.0)])
        got = [h.feasibility_step(x, norm="violated"), h.sweep_step(x, 1, norm="violated")]
    want = x.astype(np.float64) * (1.0 + 0.5 / 1.5 / n)  # v = 1.5, (2 - 1.5) / 1.5 of x, over n violated rows
    for w in got:
        np.testing.assert_allclose(w, want, rtol=1e-6)
