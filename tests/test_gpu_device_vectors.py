"""Vectors that lie on the device give what the same vectors give as host arrays."""
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


def cuda(x):
    import torch
    return torch.from_numpy(x).cuda()


@pytest.mark.parametrize("n", [1, 255, 2250, 20001])
def test_begin(lib, n):
    """beta0 (a sum over w0, default 0.1 ||w0||) and the solve bit for bit; the
    error of the first bad element."""
    rp, col, D, L = phantom.random_csr(400, n, min(1.0, 60.0 / n), seed=n)
    rng = np.random.default_rng(n)
    mask = rng.choice(np.array([0, 1, 2], np.uint32), 400)
    w0 = rng.uniform(0.1, 2.0, n).astype(np.float32)
    with lib.Handle(0) as h:
        h.load_influence(rp, col, D, L, mask, n)
        h.set_constraints([dict(struct_bit=0, kind="DOSE_MAX", bound=1.0, priority=1.0)])
        h.set_objective([dict(struct_bit=1, quantity="CDL", target=0.0, weight=1.0)])
        a = h.superiorize(w0, 5, 0.99, 1.0)
        b = h.superiorize(cuda(w0), 5, 0.99, 1.0)
        assert a[3]["beta0"] == b[3]["beta0"] == 0.1 * np.sqrt(np.cumsum(w0.astype(np.float64) ** 2)[-1])
        for x, y in zip(a[:3], b[:3]):
            np.testing.assert_array_equal(x, y.cpu().numpy())
        for bad, code in (((-1.0, np.nan), -1), ((np.nan, -1.0), -4), ((np.inf, 0.0), -4), ((-0.0, -1e-30), -1)):
            w = w0.copy()
            w[n // 2], w[n - 1] = bad
            if n == 1:  # the second value is the only one
                code = -4 if not np.isfinite(bad[1]) else -1 if bad[1] < 0 else None
            for x in (w, cuda(w)):
                if code is None:
                    h.begin(x, 0.99, 1.0)
                    continue
                with pytest.raises(lib.FredoptError) as e:
                    h.begin(x, 0.99, 1.0)
                assert e.value.code == code
