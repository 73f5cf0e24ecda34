"""w = v eps^-1 at the sizes where the block Gauss-Jordan inversion can go wrong
(one row, one pivot block, a remainder, several columns per block), on inputs
with v = 0 (a zero row and column of w), and on matrices it leaves to the
pivoted LU (a negative v; columns that do not fit shared memory); against
numpy in FP64.  Bound 1e-11 of the largest |w|: condition numbers here stay
below 1e3 and the FP64 products are accurate to a few 1e-16."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HA = 27.211386245988


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


@pytest.mark.parametrize("ng", [1, 15, 16, 17, 152, 153, 457, 1300])
@pytest.mark.parametrize("v_form", ["positive", "zeros", "negative"])
def test_screening_inverse(bse, ng, v_form):
    import torch
    r = np.random.default_rng(ng)
    nk, nv, nc, om = 2, 3, 4, 250.0
    e_v, e_c = -3.0 * r.random((nk, nv)), 1.0 + 3.0 * r.random((nk, nc))
    m = (r.standard_normal((nk, nv, nc, ng)) + 1j * r.standard_normal((nk, nv, nc, ng))) / np.sqrt(ng)
    v = 0.1 + 10.0 * r.random(ng)
    if v_form == "zeros":
        v[::5] = 0.0
    if v_form == "negative":
        v[ng // 2] = -0.05
    t = (m / np.sqrt(e_c[:, None, :] - e_v[:, :, None])[..., None]).reshape(-1, ng)
    eps = np.eye(ng) + 2.0 * HA / (nk * om) * (t.conj().T @ t) * v[None, :]
    ref = v[:, None] * np.linalg.inv(eps)
    g = lambda x: torch.as_tensor(np.ascontiguousarray(x)).cuda()  # noqa: E731
    w = torch.empty((ng, ng), dtype=torch.complex128, device="cuda")
    bse.bse_rpa_screening(g(e_v), g(e_c), g(m), g(v), om, w)
    assert np.abs(w.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
