"""Calls whose launches wait for their own blocks, from several host threads on
streams of different priority at once (FP64 Lanczos, screening inversion,
projected eigensolver), beside tensor-core builds: every result is that of the
call by itself, bit for bit, and no wait runs out."""
import threading

import numpy as np
import pytest

import bse_inputs as bi

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


def _jobs(bse):
    import torch
    g = torch.Generator(device="cuda").manual_seed(5)
    rand = lambda *s: torch.rand(s, dtype=torch.float64, device="cuda", generator=g)  # noqa: E731
    cn = lambda *s: torch.randn(s, dtype=torch.complex64, device="cuda",  # noqa: E731
                                generator=g).to(torch.complex128)

    def lanczos(n):
        z = cn(n, n)
        A = (z + z.conj().T) * (0.05 / n ** 0.5)
        A.diagonal().copy_(2.0 + 4.0 * rand(n))
        B, rho, om = 0.3 * A, cn(n), torch.linspace(0.0, 10.0, 201, dtype=torch.float64, device="cuda")
        B.diagonal().zero_()

        def run(stream):
            eps = torch.empty(201, dtype=torch.complex128, device="cuda")
            bse.bse_spectrum_lanczos(n, A, B, rho, 12.0, 100.0 * n, om, 0.1, eps, stream=stream)
            return eps

        def excitons(stream):
            E = torch.empty(3, dtype=torch.float64, device="cuda")
            bse.bse_lowest_excitons(n, A, B, 3, E, tol_ev=1e-6, stream=stream)
            return E
        return run, excitons

    m, e_v, e_c, v = cn(8, 4, 4, 400), -3.0 * rand(8, 4), 1.0 + rand(8, 4), rand(400)

    def screening(stream):
        w = torch.empty((400, 400), dtype=torch.complex128, device="cuda")
        bse.bse_rpa_screening(e_v, e_c, m, v, 250.0, w, stream=stream)
        return w

    d = bse.upload_problem(bi.make_problem(bi.BSEConfig("thr", grid=2, nv=4, nc=6, ng=59, w_scale=0.1)))
    plan = bse.Plan([bse.make_problem_struct(d)], precision=bse.BSE_PREC_BF16X6)

    def build(stream):
        plan.execute(stream)
        plan.status(stream)
        return d["A"].clone()
    big, exc = lanczos(1024)
    small, _ = lanczos(200)
    return [big, small, screening, exc, build]


def test_concurrent_calls(bse):
    import torch
    jobs = _jobs(bse)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        ref = [j(torch.cuda.current_stream()) for j in jobs]
    torch.cuda.synchronize()
    errors = []

    def work(i):
        stream = torch.cuda.Stream(priority=-(i % 3))
        try:
            with torch.cuda.stream(stream):
                for _ in range(6):
                    out = jobs[i](stream)
                    stream.synchronize()
                    if not torch.equal(out, ref[i]):
                        errors.append((i, "differs"))
        except Exception as e:  # noqa: BLE001
            errors.append((i, str(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert errors == []
    assert all(np.isfinite(torch.view_as_real(r).cpu().numpy() if r.is_complex() else r.cpu().numpy()).all()
               for r in ref)
