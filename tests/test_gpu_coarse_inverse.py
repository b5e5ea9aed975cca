"""The V-cycle's coarsest solve: a one-level hierarchy is the inverse of the pressure operator, compared with a dense
solve at sizes around a panel (8 columns), a warp (32 rows) and a CTA (1024 rows)."""
import numpy as np
import pytest

import synth
from tests.helpers import stencil_to_dense

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 1, 1), (7, 1, 1), (2, 2, 2), (3, 3, 1), (11, 3, 1), (5, 7, 3), (16, 8, 4),
                                  (16, 8, 8), (5, 41, 5)])
def test_one_level_vcycle_is_the_dense_solve(dims):
    """The operator's condition number times the FP64 rounding unit bounds both solves' difference (factor 10 for the
    growth of n operations)."""
    torch = pytest.importorskip("torch")
    from tests.helpers import build_library
    build_library()
    import paper_1602_05901_gb300 as rsv
    p = synth.make_problem(*dims, seed=17)
    A = rsv.Matrix(*dims, precision="fp64")
    A.set_values(p.vals)
    s = rsv.Solver(A)
    s.setup("cpr", gmg_max_levels=1)
    levels, _, a7 = s.cpr_info()
    assert levels == [dims]
    M = stencil_to_dense(*dims, a7[0])
    b = np.random.default_rng(3).standard_normal(A.nb)
    x = torch.zeros(A.nb, dtype=torch.float64, device="cuda")
    s.vcycle(torch.from_numpy(b).cuda(), x)
    torch.cuda.synchronize()
    ref = np.linalg.solve(M, b)
    err = np.linalg.norm(x.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err <= 10 * A.nb ** 0.5 * np.linalg.cond(M) * 2.0 ** -53, err
