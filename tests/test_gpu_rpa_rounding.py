"""Rounding of the unpivoted screening inversion against the library's pivoted LU on
the same problem: one more G without pair elements and with v < 0 sends a call to
the LU and leaves the other rows and columns of eps as they were.  The reference is
the same formula in extended precision, the inverse by Newton steps from the FP64
one.  Pair elements and v fall off with |G| and v is large at G = 0, as in a
screening near q = 0.  The mean error of four inputs must not exceed 1.25 times
that of the LU (the errors vary by about a tenth from input to input)."""
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


def _inverse_ext(eps, first):
    inv, e = first.astype(np.clongdouble), eps.astype(np.clongdouble)
    for _ in range(2):
        inv = inv + inv @ (np.eye(len(e)) - e @ inv)
    return inv


@pytest.mark.parametrize("ng", [60, 150, 250])
def test_error_against_lu(bse, ng):
    import torch
    nk, nv, nc, om = 8, 4, 6, 270.0
    g = lambda x: torch.as_tensor(np.ascontiguousarray(x)).cuda()  # noqa: E731
    ours, lu = [], []
    for seed in range(4):
        r = np.random.default_rng(seed)
        g2 = 0.9 * np.arange(ng) ** (2.0 / 3.0)
        m = r.standard_normal((nk, nv, nc, ng)) + 1j * r.standard_normal((nk, nv, nc, ng))
        m *= 0.3 / (1.0 + g2)
        e_v, e_c = -3.0 * r.random((nk, nv)), 1.0 + 3.0 * r.random((nk, nc))
        v = 4.0 * np.pi / (g2 + 0.003)
        m1, v1 = np.concatenate([m, np.zeros((nk, nv, nc, 1))], -1), np.append(v, -1e-30)
        w = []
        for x, y, library in ((m, v, False), (m1, v1, True)):
            out = torch.empty((len(y), len(y)), dtype=torch.complex128, device="cuda")
            bse.bse_phase_timing(True)
            bse.bse_rpa_screening(g(e_v), g(e_c), g(x), g(y), om, out)
            torch.cuda.synchronize()
            bse.bse_phase_timing(False)
            assert ("rpa_lu" in bse.bse_phase_report()) == library
            w.append(out.cpu().numpy()[:ng, :ng])

        def eps_of(real, cplx):
            gap = e_c.astype(real)[:, None, :] - e_v.astype(real)[:, :, None]
            t = (m.astype(cplx) / np.sqrt(gap)[..., None]).reshape(-1, ng)
            kappa2 = real(2.0) * real(HA) / (real(nk) * real(om))
            return np.eye(ng) + kappa2 * (t.conj().T @ t) * v.astype(real)[None, :]

        first = np.linalg.inv(eps_of(np.float64, np.complex128))
        ref = v[:, None] * _inverse_ext(eps_of(np.longdouble, np.clongdouble), first)
        norm = np.linalg.norm(ref.astype(complex))
        err = lambda x: float(np.linalg.norm((x - ref).astype(complex)) / norm)  # noqa: E731
        ours.append(err(w[0]))
        lu.append(err(w[1]))
    print(ng, np.mean(ours), np.mean(lu))
    assert np.mean(ours) <= 1.25 * np.mean(lu)
