"""The double-float sums (row moments, final pass) against exact ones: within
(3 n / 128 + 40) 2^-48 of the sum of the products' magnitudes for a row of n
nonzeros, the bound derived at df_dot4.  The products of two FP32 numbers are
exact in FP64 and math.fsum adds them exactly."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LENGTHS = (1, 3, 4, 5, 127, 128, 129, 257, 1000, 4097, 20000, 57000)


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2509_20012_gb300 import fredopt
    return fredopt


def values(kind, k, rng):
    v = rng.uniform(0.01, 1.0, k)
    if kind == "mixed":
        v *= rng.choice([-1.0, 1.0], k)
    elif kind == "wide":
        v *= 2.0 ** rng.integers(-30, 30, k) * rng.choice([-1.0, 1.0], k)
    elif kind == "cancelling":  # every value again with the other sign, and a small rest
        h = k // 2
        v[h:2 * h] = -v[:h]
    return v.astype(np.float32)


def bound(n, magnitudes):
    return (3 * n / 128 + 40) * 2.0 ** -48 * magnitudes


@pytest.mark.parametrize("kind", ["positive", "mixed", "wide", "cancelling"])
def test_sums_within_the_bound(lib, kind):
    n = max(LENGTHS)
    rng = np.random.default_rng(len(kind))
    D = [np.abs(values("positive", k, rng)) for k in LENGTHS]
    L = [values(kind, k, rng) for k in LENGTHS]
    cols = [np.sort(rng.choice(n, k, replace=False)).astype(np.int32) for k in LENGTHS]
    x = rng.uniform(0.2, 2.0, n).astype(np.float32)
    if kind == "cancelling":  # in the products too
        x[:] = x[0]
    rp = np.zeros(len(LENGTHS) + 1, np.int64)
    rp[1:] = np.cumsum(LENGTHS)
    mask = (1 << np.arange(len(LENGTHS))).astype(np.uint32)
    with lib.Handle(0) as h:
        h.load_influence(rp, np.concatenate(cols), np.concatenate(D), np.concatenate(L), mask, n)
        dd, ll, dl = h.get_moments()
        for i, k in enumerate(LENGTHS):
            d, l, xi = D[i].astype(np.float64), L[i].astype(np.float64), x[cols[i]].astype(np.float64)
            for got, a, b in ((dd[i], d, d), (ll[i], l, l), (dl[i], d, l)):
                assert abs(got - math.fsum(a * b)) <= bound(k, np.sum(np.abs(a * b)))
            # (D x)_i and (L x)_i in FP64, from the final check: the violation of a bound
            # of 0 (dose and cDL with c = 1; at least or at most, by the sign)
            for kinds, a in ((("DOSE_MIN", "DOSE_MAX"), d), (("CDL_MIN", "CDL_MAX"), l)):
                exact = math.fsum(a * xi)
                up = exact > 0
                h.set_constraints([dict(struct_bit=i, kind=kinds[up], bound=0.0, priority=1.0)])
                h.begin(x, 0.99, 1.0, c_cdl=1.0, use_graphs=0)
                viol = h.end()[3]["max_violation"][lib.KINDS[kinds[up]]]
                assert abs(viol - abs(exact)) <= bound(k, np.sum(np.abs(a * xi)))
