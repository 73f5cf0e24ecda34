"""A screening that no inversion can give (a NaN among the pair elements, an infinite
v) is an error and leaves w as it was, whichever inversion met it first."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("ng", [2, 17, 160])
@pytest.mark.parametrize("what", ["nan", "inf"])
@pytest.mark.parametrize("prec", [0, 2])
def test_error_leaves_w(bse, ng, what, prec):
    import torch
    r = np.random.default_rng(ng)
    m = r.standard_normal((2, 2, 3, ng)) + 1j * r.standard_normal((2, 2, 3, ng))
    e_v, e_c, v = -3.0 * r.random((2, 2)), 1.0 + 3.0 * r.random((2, 3)), 0.1 + r.random(ng)
    if what == "nan":
        m[0, 0, 0, 0] = np.nan
    else:
        v[ng // 2] = np.inf
    g = lambda x: torch.as_tensor(x).cuda()  # noqa: E731
    w = torch.full((ng, ng), 3.0 - 4.0j, dtype=torch.complex128, device="cuda")
    with pytest.raises(bse.BSEError) as err:
        bse.bse_rpa_screening(g(e_v), g(e_c), g(m), g(v), 250.0, w, precision=prec)
    assert err.value.status == bse.BSE_ERR_CUDA
    assert (w == 3.0 - 4.0j).all()
