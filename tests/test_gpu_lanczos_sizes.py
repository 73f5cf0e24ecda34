"""eps by the Lanczos recursion at the sizes where its row split can go wrong:
one row, fewer rows than SMs, a last block with fewer rows, more than 32 rows
per block, K segments that end inside a tile; against a closed form.

A = diag(e) + w w^H and B = 0 give (z^2 - A^2)^-1 A = ((z - A)^-1 - (z + A)^-1) / 2,
each resolvent by Sherman-Morrison.  The recursion stops when eps changes by
less than 1e-10 between checks; the bounds are those of the spectrum test
(FP64 products 1e-7, split products 1e-5 of the largest |eps|)."""
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


def _case(n, seed=5):
    r = np.random.default_rng(seed)
    e = np.sort(r.uniform(1.0, 7.0, n))
    w = (r.standard_normal(n) + 1j * r.standard_normal(n)) * np.sqrt(0.3 / n)
    rho = r.standard_normal(n) + 1j * r.standard_normal(n)
    return e, w, rho


def _eps_closed(e, w, rho, omega, delta, c_q, vc):
    y = np.conj(rho)

    def resolvent(z):   # y^H (z - diag(e) - w w^H)^-1 y
        g = 1.0 / (z[:, None] - e)
        ww = (g * np.abs(w) ** 2).sum(1)
        yw, wy = (g * np.conj(y) * w).sum(1), (g * np.conj(w) * y).sum(1)
        return (g * np.abs(y) ** 2).sum(1) + yw * wy / (1.0 - ww)

    z = omega + 1j * delta
    q = 0.5 * (resolvent(z) + resolvent(-z))   # -(z + A)^-1 = (-z - A)^-1
    return 1.0 - c_q * 27.211386245988 * 2.0 / vc * q


@pytest.mark.parametrize("with_b", [False, True], ids=["tda", "full"])
@pytest.mark.parametrize("n,prec", [(1, 0), (2, 0), (33, 0), (152, 0), (153, 0), (1025, 0), (4900, 0),
                                    (40, 2), (193, 2), (1025, 2), (4900, 2)])
def test_lanczos_sizes(bse, n, prec, with_b):
    import torch
    e, w, rho = _case(n)
    ld = n + (3 if n % 2 else 0)
    A = torch.zeros((n, ld), dtype=torch.complex128, device="cuda")
    wt = torch.as_tensor(w).cuda()
    A[:, :n] = wt.conj()[:, None] * wt[None, :]      # row c of the tensor: column c of w w^H
    A[:, :n].diagonal().add_(torch.as_tensor(e).cuda())
    B = torch.zeros_like(A) if with_b else None
    omega = np.linspace(0.0, 10.0, 301)
    eps = torch.empty(omega.size, dtype=torch.complex128, device="cuda")
    bse.bse_spectrum_lanczos(n, A, B, torch.as_tensor(rho).cuda(), 4 * np.pi, 100.0 * n,
                             torch.as_tensor(omega).cuda(), 0.05, eps, tol=1e-10,
                             matvec_precision=prec)
    ref = _eps_closed(e, w, rho, omega, 0.05, 4 * np.pi, 100.0 * n)
    bound = 1e-7 if prec == 0 else 1e-5
    assert np.abs(eps.cpu().numpy() - ref).max() < bound * np.abs(ref).max()


@pytest.mark.parametrize("n,prec", [(31, 2), (257, 2), (2100, 2), (1025, 0)])
def test_lanczos_repeats_bit_for_bit(bse, n, prec):
    import torch
    e, w, rho = _case(n)
    wt = torch.as_tensor(w).cuda()
    A = wt.conj()[:, None] * wt[None, :]
    A.diagonal().add_(torch.as_tensor(e).cuda())
    omega = torch.linspace(0.0, 10.0, 301, dtype=torch.float64, device="cuda")
    eps = [torch.empty(301, dtype=torch.complex128, device="cuda") for _ in range(3)]
    for x in eps:
        bse.bse_spectrum_lanczos(n, A, torch.zeros_like(A), torch.as_tensor(rho).cuda(), 4 * np.pi,
                                 100.0 * n, omega, 0.05, x, tol=1e-10, matvec_precision=prec)
    assert torch.equal(eps[0], eps[1]) and torch.equal(eps[0], eps[2])
