"""The host part of the projected eigensolver (bisection, inverse iteration and
its acceptance test), called in the library without a GPU: pairs it accepts are
as close as a library eigensolve's, residuals within 32 and overlaps within
1,000 units of rounding (neighbours 1e-3 |T| apart are not orthogonalised
against each other); what it cannot bring there it refuses.  Spectra from random
to many-fold degenerate, with couplings at the rounding of the diagonal."""
import ctypes

import numpy as np
import pytest

EPS = np.finfo(float).eps
KINDS = {
    "random": lambda r, m: (r.standard_normal(m), r.standard_normal(m - 1)),
    "banded": lambda r, m: (1 + 10 * r.random(m), 0.1 * r.standard_normal(m - 1)),
    "wilkinson": lambda r, m: (np.abs(np.arange(m) - m / 2.0), np.ones(m - 1)),
    "threefold": lambda r, m: (np.floor(3 * r.random(m)), 1e-9 * r.standard_normal(m - 1)),
    "nearly-equal": lambda r, m: (np.ones(m), np.where(r.random(m - 1) < 0.3, 0.0,
                                                       1e-15 * r.standard_normal(m - 1))),
    "graded": lambda r, m: (10 ** (-8 * r.random(m)), 1e-3 * 10 ** (-8 * r.random(m - 1))),
    "blocks": lambda r, m: (4 + (np.arange(m) % 3) * 1e-13,
                            np.where(np.arange(m - 1) % 4 == 0, 0.0, 0.5)),
}


@pytest.fixture(scope="module")
def solve():
    from paper_1904_05575_gb300 import build
    fn = ctypes.CDLL(build.build())._ZN3bse18tridiagonal_lowestEiPKdS1_iPdS2_
    fn.restype = ctypes.c_bool
    dp = ctypes.POINTER(ctypes.c_double)

    def call(d, e, k):
        m = len(d)
        d, e = np.ascontiguousarray(d, float), np.append(e, 0.0)
        lam, z = np.zeros(m), np.zeros((k, m))
        p = lambda x: x.ctypes.data_as(dp)  # noqa: E731
        return fn(m, p(d), p(e), k, p(lam), p(z)), lam[:k], z
    return call


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("m", [3, 8, 33, 96, 192, 512])
def test_accepted_pairs(solve, kind, m):
    accepted = 0
    for seed in range(40 if m < 512 else 8):
        r = np.random.default_rng(seed)
        d, e = KINDS[kind](r, m)
        ok, lam, z = solve(d, e, min(m, 64 if seed % 2 else 16))
        if not ok:
            continue
        accepted += 1
        # in extended precision, so that the check adds no rounding of its own
        d, e, lam, z = (x.astype(np.longdouble) for x in (d, e, lam, z))
        row = np.abs(d) + np.append(np.abs(e), 0) + np.append(0, np.abs(e))
        norm = row.max()
        t = z * d - lam[:, None] * z
        t[:, :-1] += z[:, 1:] * e
        t[:, 1:] += z[:, :-1] * e
        assert np.abs(t).max() <= 34 * EPS * norm
        assert np.abs(z @ z.T - np.eye(len(lam))).max() <= 1003 * EPS
    assert accepted > 0
