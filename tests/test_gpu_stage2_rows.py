"""The CUDA-core second contraction with one X row per thread, at the sizes
where its tiles, ring and row pairs can go wrong: an odd T side (boxes start on
an odd row), more X rows than one tile, a T side of several tiles, one chunk
of plane waves, fewer chunks than the ring, a remainder; whole builds,
Hermitian plans and k-row slabs, against the oracle (BF16x6: 1e-6 relative
Frobenius of A - E^ip and of B, the tolerance of the build tests)."""
import numpy as np
import pytest

import bse_inputs as bi
from oracle import bse_oracle as O

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


# (grid, nv, nc, ng): pair blocks nv^2 x nc^2 and (nv nc)^2
SHAPES = [(2, 3, 5, 59),     # 25 x 9 (odd T side)
          (2, 4, 6, 17),     # 36 x 16, three chunks
          (1, 3, 13, 9),     # 169 x 9: two x tiles; 39 x 39
          (1, 3, 14, 5),     # 196 x 9; 42 x 42: three t tiles; one chunk
          (2, 4, 12, 33),    # 144 x 16; 48 x 48
          (1, 5, 10, 1)]     # 100 x 25: two odd t tiles; NG = 1


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("form", ["whole", "hermitian", "slab"])
def test_stage2_rows(bse, shape, form):
    grid, nv, nc, ng = shape
    nk = grid ** 3
    if form == "slab" and nk == 1:
        pytest.skip("one k row")
    p = bi.make_problem(bi.BSEConfig("rows", grid=grid, nv=nv, nc=nc, ng=ng, w_scale=0.1))
    d = bse.upload_problem(p)
    if form == "slab":
        kb, kn = 1, nk - 3
        d["m_vv"], d["m_cc"] = d["m_vv"][kb:kb + kn].contiguous(), d["m_cc"][kb:kb + kn].contiguous()
        st = bse.make_problem_struct(d, k_begin=kb, k_count=kn)
    else:
        kb, kn = 0, nk
        st = bse.make_problem_struct(d)
    plan = bse.Plan([st], precision=bse.BSE_PREC_BF16X6, hermitian=form == "hermitian")
    plan.execute()
    plan.execute()
    plan.status()
    plan.close()
    n, nb = nk * nv * nc, nv * nc
    rows = slice(kb * nb, (kb + kn) * nb)
    A_ref, B_ref = O.build_A_B(p)
    e = (p["e_c"][:, None, :] - p["e_v"][:, :, None]).reshape(-1)
    for M, R, sub in ((d["A"], A_ref, np.diag(e)), (d["B"], B_ref, 0.0)):
        got, ref = (bse.matrix_to_numpy(M, n) - sub)[rows], (R - sub)[rows]
        assert np.linalg.norm(got - ref) < 1e-6 * np.linalg.norm(ref)
