"""Block ILU(0) tile sweeps at the shapes where a tile, a step group or the residency ends: fewer pencils than a
tile, one more than a tile, odd step counts, and more tiles than are resident at once (a CTA then takes several)."""
import numpy as np
import pytest

import oracle
import synth
from tests.helpers import per_entry_ratio, report_ratio

pytestmark = pytest.mark.gpu

DIMS = [(1, 8, 4), (1, 9, 5), (2, 7, 3), (3, 17, 9), (6, 33, 4), (5, 4, 33), (70, 9, 8), (4, 248, 124)]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dims", DIMS)
def test_ilu_apply_at_tile_edges(dims, precision):
    """Per entry against the oracle on the same (FP32-rounded for mixed) matrix, with the bounds of the other
    block ILU(0) parity tests: 1e-10 in FP64, 1e-3 in FP32."""
    torch = pytest.importorskip("torch")
    from tests.helpers import build_library
    build_library()
    import paper_1602_05901_gb300 as rsv
    p = synth.make_problem(*dims, seed=91)
    A = rsv.Matrix(*dims)
    A.set_values(p.vals)
    s = rsv.Solver(A, precision=precision)
    s.setup("bilu0")
    r = np.random.default_rng(92).standard_normal(p.n)
    dtype, bound = (torch.float64, 1e-10) if precision == "fp64" else (torch.float32, 1e-3)
    if precision == "mixed":
        p.vals = p.vals.astype(np.float32).astype(np.float64)
        r = r.astype(np.float32).astype(np.float64)
    rd = torch.from_numpy(r).cuda().to(dtype)
    zd = torch.full_like(rd, float("nan"))
    for _ in range(2):  # the second apply starts from the first one's edge buffers
        s.apply(rd, zd)
    torch.cuda.synchronize()
    _, z = oracle.System.from_problem(p, pc="bilu0").pc_apply(r)
    ratio = report_ratio(f"ilu_tiles_{precision}_{dims}", per_entry_ratio(zd.double().cpu().numpy(), z), bound)
    assert ratio <= bound


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dims", [(3, 17, 9), (70, 9, 8), (41, 40, 21)])
def test_ilu_apply_repeats_bit_for_bit(precision, dims):
    """The order of a cell's operations is fixed, so whatever the timing of the hand-offs between warps and tiles is, every
    apply gives the same bits."""
    torch = pytest.importorskip("torch")
    from tests.helpers import build_library
    build_library()
    import paper_1602_05901_gb300 as rsv
    p = synth.make_problem(*dims, seed=93)
    A = rsv.Matrix(*dims)
    A.set_values(p.vals)
    s = rsv.Solver(A, precision=precision)
    s.setup("bilu0")
    r = torch.from_numpy(np.random.default_rng(94).standard_normal(p.n)).cuda()
    r = r if precision == "fp64" else r.float()
    first, z = torch.empty_like(r), torch.empty_like(r)
    s.apply(r, first)
    for _ in range(100):
        s.apply(r, z.fill_(float("nan")))
        assert torch.equal(z, first)
