"""A plan of more problems than one split launch takes jobs (24; five to six
per problem here): every problem's A and B against the oracle, 1e-6 relative
Frobenius as in the build tests."""
import numpy as np
import pytest

import bse_inputs as bi
from oracle import bse_oracle as O

pytestmark = pytest.mark.gpu


def test_plan_of_nine_problems():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1904_05575_gb300 as bse
    wins = [(2, 3), (3, 2), (1, 4), (2, 2), (3, 5), (4, 1), (2, 6), (3, 3), (1, 1)]
    cfg = bi.BSEConfig("nine", grid=2, nv=2, nc=2, ng=27, q_abs=tuple(0.1 * i for i in range(9)),
                       windows=tuple(wins), w_scale=0.1)
    ps = [bi.make_problem(cfg, q_index=i) for i in range(9)]
    ds = [bse.upload_problem(p) for p in ps]
    plan = bse.Plan([bse.make_problem_struct(d) for d in ds], precision=bse.BSE_PREC_BF16X6)
    plan.execute()
    plan.status()
    plan.close()
    for p, d in zip(ps, ds):
        n = p["nk"] * p["nv"] * p["nc"]
        for got, ref in zip((d["A"], d["B"]), O.build_A_B(p)):
            assert np.linalg.norm(bse.matrix_to_numpy(got, n) - ref) < 1e-6 * np.linalg.norm(ref)
