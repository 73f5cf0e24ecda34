"""Device memory that stays in use after a split-precision screening: at most the
1 GiB of workspace that the pool may keep, whatever the number of transitions
(they go in chunks), and 8 bytes per transition.  64 MiB allowance for the pool's
block size and the library's small buffers.  The result of several chunks, the
last one shorter, against numpy (BF16x6: 1e-6 of the largest |w|)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
GIB, SLACK = 1 << 30, 64 << 20


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


def test_workspace_after_the_call(bse):
    import torch
    ng = 200
    g = torch.Generator(device="cuda").manual_seed(1)

    def inputs(nk, nv, nc):
        rand = lambda *s: torch.rand(s, dtype=torch.float64, device="cuda", generator=g)  # noqa: E731
        m = torch.randn((nk, nv, nc, ng), dtype=torch.complex64, device="cuda", generator=g)
        return -3.0 * rand(nk, nv), 1.0 + 3.0 * rand(nk, nc), (0.01 * m).to(torch.complex128), rand(ng)

    w = torch.empty((ng, ng), dtype=torch.complex128, device="cuda")
    call = lambda a: bse.bse_rpa_screening(*a, 250.0, w, precision=2)  # noqa: E731
    # 16,000 and 160,000 transitions (0.1 and 0.99 GiB), 400,000 and 451,000 (2.5 and
    # 2.8 GiB of workspace at once)
    small, below, above = inputs(40, 20, 20), inputs(400, 20, 20), inputs(1000, 20, 20)
    ragged = inputs(1000, 11, 41)
    torch.cuda.empty_cache()
    call(small)      # library handles, module load
    free = [torch.cuda.mem_get_info()[0]]
    for a in (below, above, ragged):
        call(a)
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
    assert free[0] - min(free) <= GIB + SLACK
    for a in (above, ragged):
        call(a)
        e_v, e_c, m, v = (x.cpu().numpy() for x in a)
        t = (m / np.sqrt(e_c[:, None, :] - e_v[:, :, None])[..., None]).reshape(-1, ng)
        eps = np.eye(ng) + 2.0 * 27.211386245988 / (len(e_v) * 250.0) * (t.conj().T @ t) * v[None, :]
        ref = v[:, None] * np.linalg.inv(eps)
        assert np.abs(w.cpu().numpy() - ref).max() < 1e-6 * np.abs(ref).max()
