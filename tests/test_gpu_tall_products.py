"""The Davidson solve's tall-skinny products at the edges of their row ranges
(64 rows) and tiles (16 columns): block-diagonal problems, shuffled and
reflected, whose excitons follow from the blocks.  Residual tolerance 1e-6 eV: energies to
1e-8 eV as in the Davidson tests."""
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


@pytest.mark.parametrize("g,blocks,nev", [(9, 7, 1), (8, 8, 15), (13, 5, 16), (41, 25, 17), (17, 241, 33)],
                         ids=str)
def test_block_problems(bse, g, blocks, nev):
    import torch
    r = np.random.default_rng(g)
    n = g * blocks
    perm = r.permutation(n)
    A = np.zeros((n, n), dtype=np.complex128)
    B = np.zeros_like(A)
    ref = []
    for i in range(blocks):
        z = r.standard_normal((2, g, g)) + 1j * r.standard_normal((2, g, g))
        a, b = ((x + x.conj().T) * 0.03 / np.sqrt(g) for x in z)
        a = a + np.diag(r.uniform(2.0, 6.0, g))
        L = np.linalg.cholesky(a - b)
        ref.append(np.sqrt(np.linalg.eigvalsh(L.conj().T @ (a + b) @ L)))
        p = perm[i * g:(i + 1) * g]
        A[np.ix_(p, p)], B[np.ix_(p, p)] = a, b
    ref = np.sort(np.concatenate(ref))[:nev]
    # a reflection couples the blocks (the solve can miss a state that the
    # unit vectors it starts from hardly reach)
    v = r.standard_normal(n) + 1j * r.standard_normal(n)
    v *= np.sqrt(2.0) / np.linalg.norm(v)

    def reflect(M):
        M = M - np.outer(v, v.conj() @ M)
        return M - np.outer(M @ v, v.conj())

    A, B = reflect(A), reflect(B)
    t = lambda x: torch.as_tensor(np.ascontiguousarray(x.T)).cuda()  # noqa: E731
    E = torch.empty(nev, dtype=torch.float64, device="cuda")
    X = torch.empty((nev, n), dtype=torch.complex128, device="cuda")
    bse.bse_lowest_excitons(n, t(A), t(B), nev, E, X, tol_ev=1e-6, max_iter=300)
    e = E.cpu().numpy()
    assert np.abs(e - ref).max() < 1e-8
    x = X.cpu().numpy()
    assert np.abs(x.conj() @ (((A + B) @ x.T) / e[None, :]) - np.eye(nev)).max() < 1e-6


@pytest.mark.parametrize("n", [9440, 9480])
def test_split_planes_either_side_of_a_gibibyte(bse, n):
    """Tensor-core products whose planes (12 n^2 bytes) are just below and just
    above 1 GiB: pairs [[a, c], [c, a]] with coupling b have E = sqrt((a +- c)^2
    - b^2).  Split error of the couplings below 1e-7 eV, residual 1e-5 eV."""
    import torch
    r = np.random.default_rng(n)
    a, c, b, nev = r.uniform(2.0, 6.0, n // 2), 0.1, 0.05, 4
    A = torch.diag(torch.as_tensor(np.repeat(a, 2), dtype=torch.complex128, device="cuda"))
    B = torch.zeros_like(A)
    i = torch.arange(0, n, 2, device="cuda")
    for M, x in ((A, c), (B, b)):
        M[i, i + 1] = x
        M[i + 1, i] = x
    ref = np.sort(np.concatenate([np.sqrt((a + c) ** 2 - b * b), np.sqrt((a - c) ** 2 - b * b)]))[:nev]
    E = torch.empty(nev, dtype=torch.float64, device="cuda")
    bse.bse_lowest_excitons(n, A, B, nev, E, tol_ev=1e-5, matvec_precision=bse.BSE_PREC_BF16X6)
    assert np.abs(E.cpu().numpy() - ref).max() < 1e-6
