"""Device memory that stays in use after a split-precision screening: at most the
1 GiB that the pool may keep, whatever the number of transitions; a workspace
above that is given back on return.  64 MiB allowance for the pool's block size
and the library's small buffers."""
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
    # 16,000, 160,000 and 400,000 transitions: planes of 0.1, 0.96 and 2.4 GB,
    # partial sums of 0.01, 0.1 and 0.25 GB
    small, below, above = inputs(40, 20, 20), inputs(400, 20, 20), inputs(1000, 20, 20)
    torch.cuda.empty_cache()
    call(small)      # library handles, module load
    used = [torch.cuda.mem_get_info()[0]]
    for a in (above, below, above):
        call(a)
        torch.cuda.synchronize()
        used.append(torch.cuda.mem_get_info()[0])
    free0, after_above, after_below, after_all = used
    assert free0 - after_above <= SLACK            # given back
    assert free0 - after_below <= GIB + SLACK      # kept for the next call, bounded
    assert after_below - after_all <= SLACK        # and not added to
    # the pool's memory and the device's give the same result
    w1 = w.clone()
    call(above)
    assert torch.equal(w, w1)
    e_v, e_c, m, v = (x.cpu().numpy() for x in below)
    call(below)
    t = (m / np.sqrt(e_c[:, None, :] - e_v[:, :, None])[..., None]).reshape(-1, ng)
    eps = np.eye(ng) + 2.0 * 27.211386245988 / (400 * 250.0) * (t.conj().T @ t) * v[None, :]
    ref = v[:, None] * np.linalg.inv(eps)
    assert np.abs(w.cpu().numpy() - ref).max() < 1e-6 * np.abs(ref).max()
