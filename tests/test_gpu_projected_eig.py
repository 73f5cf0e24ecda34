"""The Davidson solve's own eigensolver of the projected problem: degenerate
excitons (each energy three times, the wanted ones cutting through a triple),
small bases and a basis of several hundred vectors, against numpy.  Residual
tolerance 1e-6 eV: energies to 1e-8 eV as in the Davidson tests."""
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


@pytest.mark.parametrize("n0,copies,nev", [(1, 3, 1), (2, 2, 2), (40, 3, 7), (150, 1, 12), (300, 2, 20)],
                         ids=str)
@pytest.mark.parametrize("full", [False, True], ids=["tda", "full"])
def test_degenerate_and_small(bse, n0, copies, nev, full):
    import torch
    r = np.random.default_rng(n0)

    def herm(scale):
        z = r.standard_normal((n0, n0)) + 1j * r.standard_normal((n0, n0))
        return (z + z.conj().T) * scale / np.sqrt(n0)

    A0 = np.diag(r.uniform(2.0, 6.0, n0)) + herm(0.05)
    B0 = herm(0.03)
    A, B = np.kron(A0, np.eye(copies)), np.kron(B0, np.eye(copies))
    if full:
        L = np.linalg.cholesky(A0 - B0)
        e0 = np.sqrt(np.linalg.eigvalsh(L.conj().T @ (A0 + B0) @ L))
    else:
        e0 = np.linalg.eigvalsh(A0)
    ref = np.sort(np.repeat(e0, copies))[:nev]
    n = n0 * copies
    t = lambda x: torch.as_tensor(np.ascontiguousarray(x.T)).cuda()  # noqa: E731
    E = torch.empty(nev, dtype=torch.float64, device="cuda")
    X = torch.empty((nev, n), dtype=torch.complex128, device="cuda")
    bse.bse_lowest_excitons(n, t(A), t(B) if full else None, nev, E, X, tol_ev=1e-6, max_iter=300)
    assert np.abs(E.cpu().numpy() - ref).max() < 1e-8
    x = X.cpu().numpy()                       # rows: X+Y; (X+Y)^H (X-Y) = 1, X-Y = (A+B)(X+Y)/E
    P = A + B if full else A
    xm = (P @ x.T) / E.cpu().numpy()[None, :]
    assert np.abs(x.conj() @ xm - np.eye(nev)).max() < 1e-6
