"""The screening inversion without pivots at the edge of what it may take: the
exact eps is similar to a matrix with all eigenvalues >= 1, but the X of the
tensor cores carries their rounding, and a large v on two almost proportional
plane waves G brings that rounding to the size of the pivot.  X as the library
forms it follows from a call with v = 1 (well conditioned: w = (1 + 2 kappa X)^-1),
and v of the second G is set so that the second pivot of eps would be about zero
(left to the pivoted LU) or clearly above 1/2 (taken without pivots).

Which of the two served the call is what is asserted: X is rounding there, and w
with it (condition numbers of 1e12 and more), whoever inverts.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HA = 27.211386245988
OM, NK, NV, NC, NG = 250.0, 2, 3, 4, 6


@pytest.fixture(scope="module")
def bse():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1904_05575_gb300 import build
    build.build()
    import paper_1904_05575_gb300 as m
    m.load()
    return m


def _screen(bse, m, v, e_v, e_c, prec):
    """w and whether the library's LU formed it."""
    import torch
    g = lambda x: torch.as_tensor(np.ascontiguousarray(x)).cuda()  # noqa: E731
    w = torch.empty((NG, NG), dtype=torch.complex128, device="cuda")
    bse.bse_phase_timing(True)
    bse.bse_rpa_screening(g(e_v), g(e_c), g(m), g(v), OM, w, precision=prec)
    torch.cuda.synchronize()
    bse.bse_phase_timing(False)
    return w.cpu().numpy(), "rpa_lu" in bse.bse_phase_report()


@pytest.mark.parametrize("prec", [2, 3], ids=["bf16x6", "bf16x3"])
def test_pivots_at_the_rounding_of_x(bse, prec):
    two = 2.0 * HA / (NK * OM)
    served = {False: 0, True: 0}
    for seed in range(8):
        r = np.random.default_rng(seed)
        e_v, e_c = -3.0 * r.random((NK, NV)), 1.0 + 3.0 * r.random((NK, NC))
        m = r.standard_normal((NK, NV, NC, NG)) + 1j * r.standard_normal((NK, NV, NC, NG))
        m[..., 1] = m[..., 0] * (0.7 + 0.3j)
        w, lu = _screen(bse, m, np.ones(NG), e_v, e_c, prec)
        assert not lu
        X = (np.linalg.inv(w) - np.eye(NG)) / two
        v = np.ones(NG)
        v[0] = 1e12
        # what is left of X11 behind the first pivot: zero but for rounding
        rest = (X[1, 1] - two * v[0] * X[1, 0] * X[0, 1] / (1.0 + two * v[0] * X[0, 0])).real
        for pivot in (1e-3, 0.9, 3.0):
            if (pivot - 1.0) * rest <= 0.0:
                continue   # this sign of the rounding cannot give that pivot
            v[1] = (pivot - 1.0) / (two * rest)
            w, lu = _screen(bse, m, v, e_v, e_c, prec)
            served[lu] += 1
            assert lu == (pivot < 0.5)
            assert np.isfinite(w).all()
    assert served[True] > 0 and served[False] > 0
