"""eps by Lanczos at the ends of the FP64 range: a recursion that ends after one
step (rho an eigenvector) with delta and omega towards zero, omega up to 1e60;
rho scaled by 1e-157 to 1e152 (eps - 1 is proportional to |rho|^2; subnormal
sums to 1e-3).  A = diag(e), so eps has a closed form.  Bound 1e-10 of the largest |eps| (the
coefficients are sums of at most 5 terms and the recursion ends exactly)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
E = np.arange(1.0, 6.0)
PREF, VC = 4 * np.pi * 27.211386245988 * 2.0, 100.0


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


def _eps(bse, rho, omega, delta):
    import torch
    g = lambda x, t: torch.as_tensor(np.asarray(x), dtype=t).cuda()  # noqa: E731
    out = torch.empty(len(omega), dtype=torch.complex128, device="cuda")
    bse.bse_spectrum_lanczos(5, g(np.diag(E), torch.complex128), None, g(rho, torch.complex128),
                             4 * np.pi, VC, g(omega, torch.float64), delta, out, tol=1e-8)
    return out.cpu().numpy()


def _closed(rho, omega, delta):
    z2 = (np.asarray(omega) + 1j * delta) ** 2
    return 1.0 - PREF / VC * (np.asarray(rho) ** 2 * E / (z2[:, None] - E ** 2)).sum(1)


@pytest.mark.parametrize("delta", [1e-3, 1e-15, 1e-20, 1e-25, 1e-60])
def test_ended_recursion_near_zero_frequency(bse, delta):
    rho = np.array([1.0, 0, 0, 0, 0])
    omega = [0.0, 1e-30, 1e-20, 0.5]
    eps, ref = _eps(bse, rho, omega, delta), _closed(rho, omega, delta)
    assert np.abs(eps - ref).max() < 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("omega", [1e3, 1e10, 1e19, 1e20, 1e40, 1e60])
def test_large_frequencies(bse, omega):
    rho = np.ones(5)
    eps, ref = _eps(bse, rho, [omega, 2 * omega], 0.1), _closed(rho, [omega, 2 * omega], 0.1)
    assert np.isfinite(eps).all()
    assert np.abs(eps.real - ref.real).max() < 1e-10


@pytest.mark.parametrize("scale", [1e-157, 1e-155, 1e-152, 1e-120, 1e120, 1e150, 1e152])
def test_small_and_large_rho(bse, scale):
    omega, one = [0.5, 2.0, 7.0], np.ones(5)
    eps, ref = _eps(bse, scale * one, omega, 0.1), _closed(one, omega, 0.1)
    if scale > 1.0:
        assert np.abs((eps - 1.0) / scale / scale - (ref - 1.0)).max() < 1e-10 * np.abs(ref).max()
    else:   # eps - 1 is lost in the real part
        assert np.abs(eps.real - 1.0).max() < 1e-10
        rel = 1e-3 if scale < 1e-153 else 1e-10
        assert np.abs(eps.imag / scale / scale - ref.imag).max() < rel * np.abs(ref.imag).max()
