"""The CUDA-core second contraction on both sides of the rule between tiles and
one X row per thread (it weighs what the pairs of a launch save): whole builds
of 27 and 64 k points, whose many pairs take the one-row form, with odd T
sides, several x and t tiles, one chunk of plane waves and remainders, and
k-row slabs of one row of the same problems, whose few pairs take the tiles.
Against the oracle (BF16x6: 1e-6 relative Frobenius of A - E^ip and of B, the
tolerance of the build tests)."""
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
SHAPES = [(4, 3, 5, 11),     # 25 x 9: one-row form from 3,145 pairs
          (3, 3, 13, 9),     # 169 x 9: two x tiles
          (3, 3, 15, 1),     # 225 x 9; 45 x 45: t tiles starting on odd rows; NG = 1
          (3, 14, 3, 25),    # the same with the sides swapped; 42 x 42; a remainder
          (3, 4, 12, 33)]    # 144 x 16; 48 x 48


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_both_sides_of_the_rule(bse, shape):
    grid, nv, nc, ng = shape
    nk = grid ** 3
    p = bi.make_problem(bi.BSEConfig("form", grid=grid, nv=nv, nc=nc, ng=ng, w_scale=0.1))
    A_ref, B_ref = O.build_A_B(p)
    e = (p["e_c"][:, None, :] - p["e_v"][:, :, None]).reshape(-1)
    n, nb = nk * nv * nc, nv * nc
    for kb, kn, hermitian in ((0, nk, False), (0, nk, True), (nk - 2, 1, False)):
        d = bse.upload_problem(p)
        d["m_vv"], d["m_cc"] = d["m_vv"][kb:kb + kn].contiguous(), d["m_cc"][kb:kb + kn].contiguous()
        st = bse.make_problem_struct(d) if kn == nk else bse.make_problem_struct(d, k_begin=kb, k_count=kn)
        plan = bse.Plan([st], precision=bse.BSE_PREC_BF16X6, hermitian=hermitian)
        plan.execute()
        plan.execute()
        plan.status()
        plan.close()
        rows = slice(kb * nb, (kb + kn) * nb)
        for M, R, sub in ((d["A"], A_ref, np.diag(e)), (d["B"], B_ref, 0.0)):
            got, ref = (bse.matrix_to_numpy(M, n) - sub)[rows], (R - sub)[rows]
            assert np.linalg.norm(got - ref) < 1e-6 * np.linalg.norm(ref)
