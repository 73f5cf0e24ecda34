"""Bounded device waits of the calls without a plan, made to run out without a
fault: with a budget of a few clock cycles every block but the last to arrive
at an exchange, and every wait for an operand copy, gives up.  The call returns
BSE_ERR_TIMEOUT, the context stays usable and the same call with the default
budget gives the result it gave before, bit for bit.  The phase records show
where the launches with those waits serve a call and where the library does."""
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


def _matrices(n, seed=1):
    """A, B with A +- B positive definite (diagonal 2 .. 6, couplings of about 0.05)."""
    import torch
    r = np.random.default_rng(seed)
    out = []
    for scale in (0.05, 0.03):
        z = r.standard_normal((n, n)) + 1j * r.standard_normal((n, n))
        out.append((z + z.conj().T) * scale / np.sqrt(n))
    out[0] += np.diag(r.uniform(2.0, 6.0, n))
    return [torch.as_tensor(np.ascontiguousarray(x.T)).cuda() for x in out]


def _lanczos(bse, n, prec):
    import torch
    A, B = _matrices(n)
    rho = torch.as_tensor(np.random.default_rng(2).standard_normal(n) + 0.3j).cuda()
    omega = torch.linspace(0.0, 10.0, 101, dtype=torch.float64, device="cuda")
    eps = torch.empty(101, dtype=torch.complex128, device="cuda")

    def call():
        bse.bse_spectrum_lanczos(n, A, B, rho, 4 * np.pi, 100.0 * n, omega, 0.1, eps,
                                 matvec_precision=prec)
        return eps.clone()
    return call


def _excitons(bse, n, prec):
    import torch
    A, B = _matrices(n)
    E = torch.empty(3, dtype=torch.float64, device="cuda")

    def call():
        bse.bse_lowest_excitons(n, A, B, 3, E, tol_ev=1e-5, max_iter=100, matvec_precision=prec)
        return E.clone()
    return call


def _screening(bse, ng, prec):
    import torch
    r = np.random.default_rng(ng)
    g = lambda x: torch.as_tensor(x).cuda()  # noqa: E731
    m = g(r.standard_normal((2, 3, 4, ng)) + 1j * r.standard_normal((2, 3, 4, ng))) / np.sqrt(ng)
    args = (g(-3.0 * r.random((2, 3))), g(1.0 + 3.0 * r.random((2, 4))), m, g(0.1 + r.random(ng)))
    w = torch.empty((ng, ng), dtype=torch.complex128, device="cuda")

    def call():
        bse.bse_rpa_screening(*args, 250.0, w, precision=prec)
        return w.clone()
    return call


@pytest.mark.parametrize("prec", [0, 2], ids=["fp64", "bf16x6"])
@pytest.mark.parametrize("make,n", [(_lanczos, 300), (_excitons, 300), (_screening, 100)],
                         ids=["lanczos", "excitons", "screening"])
def test_wait_runs_out_then_recovers(bse, make, n, prec):
    import torch
    call = make(bse, n, prec)
    before = call()
    assert torch.isfinite(torch.view_as_real(before) if before.is_complex() else before).all()
    bse.bse_set_wait_limit(1e-9)
    try:
        with pytest.raises(bse.BSEError) as err:
            call()
    finally:
        bse.bse_set_wait_limit(2.0)
    assert err.value.status == bse.BSE_ERR_TIMEOUT
    assert torch.equal(call(), before)


def test_another_thread_keeps_its_own_limit(bse):
    import threading
    import torch
    call = _lanczos(bse, 300, 0)
    before = call()
    bse.bse_set_wait_limit(1e-9)
    try:
        got = []
        t = threading.Thread(target=lambda: got.append(call()))
        t.start()
        t.join()
    finally:
        bse.bse_set_wait_limit(2.0)
    assert torch.equal(got[0], before)


def _phases(bse, call):
    import torch
    bse.bse_phase_timing(True)
    call()
    torch.cuda.synchronize()
    bse.bse_phase_timing(False)
    return bse.bse_phase_report()


@pytest.mark.parametrize("nev,library", [(3, False), (33, True)])
def test_which_eigensolve_serves_the_projection(bse, nev, library):
    """Up to 64 pairs (two per exciton) of up to 512 vectors: this library's."""
    import torch
    A, B = _matrices(300)
    E = torch.empty(nev, dtype=torch.float64, device="cuda")
    ph = _phases(bse, lambda: bse.bse_lowest_excitons(300, A, B, nev, E, tol_ev=1e-5, max_iter=100))
    assert ("davidson_zheevd" in ph) == library


@pytest.mark.parametrize("ng,library", [(1, False), (152, False), (1000, False), (1300, True)])
def test_which_inversion_serves_the_screening(bse, ng, library):
    """The unpivoted inversion while a block's columns fit shared memory, else LU."""
    assert ("rpa_lu" in _phases(bse, _screening(bse, ng, 0))) == library


@pytest.mark.parametrize("warm", [False, True], ids=["cold", "warm"])
def test_expired_product_is_a_timeout_not_a_statement_on_the_input(bse, warm):
    """The products of a solve whose waits run out are whatever the workspace
    held.  An earlier solve leaves a matrix there whose projection is not positive
    definite; the next, of a positive definite matrix, must report the wait."""
    import torch
    n, k = 300, 4
    good = _matrices(n)[0]
    bad = torch.full((n, n), -10.0, dtype=torch.complex128, device="cuda")
    bad.diagonal().copy_(torch.linspace(2.0, 6.0, n).cuda())
    E = torch.empty(k, dtype=torch.float64, device="cuda")
    start = torch.eye(n, dtype=torch.complex128, device="cuda")[:2 * k].contiguous() if warm else None

    def call(A):
        bse.bse_lowest_excitons(n, A, None, k, E, tol_ev=1e-5, max_iter=100, matvec_precision=2,
                                start=start)

    with pytest.raises(bse.BSEError) as err:
        call(bad)
    assert err.value.status == bse.BSE_ERR_NOT_PD
    bse.bse_set_wait_limit(1e-9)
    try:
        with pytest.raises(bse.BSEError) as err:
            call(good)
    finally:
        bse.bse_set_wait_limit(2.0)
    assert err.value.status == bse.BSE_ERR_TIMEOUT
    call(good)
    assert torch.isfinite(E).all()
