"""FP64 Lanczos steps: the sums that the blocks exchange in device memory are
read after every block has written them, so that each run gives the same bits.
From two blocks to one per SM, one row per block and many; several runs each,
against A = diag(e) (no exchange error: the resolvent sum has a closed form).
Bound 1e-9 of the largest |eps| (tolerance of the recursion 1e-10)."""
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


@pytest.mark.parametrize("n", [2, 47, 151, 304, 1300])
def test_fp64_runs_agree_bit_for_bit(bse, n):
    import torch
    r = np.random.default_rng(n)
    e, rho = r.uniform(1.0, 7.0, n), r.standard_normal(n) + 1j * r.standard_normal(n)
    omega, delta, vc = np.linspace(0.0, 10.0, 201), 0.2, 100.0 * n
    A = torch.diag(torch.as_tensor(e).cuda().to(torch.complex128))
    rt, wt = torch.as_tensor(rho).cuda(), torch.as_tensor(omega).cuda()
    out = []
    for _ in range(6):
        eps = torch.empty(omega.size, dtype=torch.complex128, device="cuda")
        bse.bse_spectrum_lanczos(n, A, torch.zeros_like(A), rt, 4 * np.pi, vc, wt, delta, eps,
                                 tol=1e-10)
        out.append(eps)
    assert all(torch.equal(out[0], x) for x in out[1:])
    z = omega + 1j * delta
    q = (np.abs(rho) ** 2 * e / (z[:, None] ** 2 - e ** 2)).sum(1)
    ref = 1.0 - 4 * np.pi * 27.211386245988 * 2.0 / vc * q
    assert np.abs(out[0].cpu().numpy() - ref).max() < 1e-9 * np.abs(ref).max()
