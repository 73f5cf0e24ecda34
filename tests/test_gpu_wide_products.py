"""Tensor-core products of blocks wider than the split-K partial sums allow (512
MiB: 52 columns at 12,803 rows): one tile runs over all of K.  A warm start from
61 vectors makes two such products, with a ragged last row tile, K step and
column tile; after one iteration the Ritz values of the 122 vectors are compared
with those of FP64 products.  They differ by at most the products' error, 1e-7
(BF16x6) of the off-diagonal part: 1e-6 eV asserted for an off-diagonal norm
of about 1 eV."""
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


@pytest.mark.parametrize("full", [False, True], ids=["tda", "full"])
def test_whole_k_block(bse, full):
    import torch
    n, nev, k0 = 12803, 16, 61
    g = torch.Generator(device="cuda").manual_seed(3)

    def herm(scale):
        z = torch.randn((n, n), dtype=torch.complex64, device="cuda", generator=g)
        z = z + z.conj().T
        return (z * (scale / n ** 0.5)).to(torch.complex128)

    A = herm(0.25)
    A.diagonal().copy_(2.0 + 6.0 * torch.rand(n, dtype=torch.float64, device="cuda", generator=g))
    B = herm(0.05) if full else None
    start = torch.randn((k0, n), dtype=torch.complex64, device="cuda", generator=g).to(torch.complex128)
    E = {}
    for prec in (0, 2):
        E[prec] = torch.zeros(nev, dtype=torch.float64, device="cuda")
        with pytest.raises(bse.BSEError) as err:
            bse.bse_lowest_excitons(n, A, B, nev, E[prec], tol_ev=1e-12, max_iter=1,
                                    matvec_precision=prec, start=start)
        assert err.value.status == bse.BSE_ERR_NO_CONV
    assert (E[0] > 0).all()
    assert (E[0] - E[2]).abs().max() < 1e-6
