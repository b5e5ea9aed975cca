"""Buffers that a solver keeps from one preconditioner setup to the next."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rsv():
    from tests.helpers import build_library
    build_library()
    import paper_1602_05901_gb300 as m
    return m


def _apply(torch, s, r):
    z = torch.full_like(r, float("nan"))
    s.apply(r, z)
    torch.cuda.synchronize()
    return z


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_coarsening_changes_on_one_solver(rsv, precision):
    """Both pressure hierarchies of a grid of at most gmg_max_coarse cells have one geometric level, but only the geometric
    one keeps that level's dense inverse: setups in turn on one solver give the same bits as on a solver of their own."""
    torch = pytest.importorskip("torch")
    p = synth.make_problem(9, 8, 6, seed=31)
    A = rsv.Matrix(p.nx, p.ny, p.nz)
    A.set_values(p.vals)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    r = torch.from_numpy(np.random.default_rng(32).standard_normal(p.n)).cuda().to(dtype)
    setups = {"amg": dict(coarsening="amg", gmg_max_levels=8, gmg_max_coarse=64), "gmg": {}}
    alone = {}
    for name, kw in setups.items():
        s = rsv.Solver(A, precision=precision)
        s.setup("cpr", **kw)
        alone[name] = _apply(torch, s, r)
    s = rsv.Solver(A, precision=precision)
    for name in ("amg", "gmg", "amg", "gmg"):
        s.setup("cpr", **setups[name])
        assert torch.equal(_apply(torch, s, r), alone[name]), name
