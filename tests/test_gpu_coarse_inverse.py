"""The V-cycle's coarsest solve: a one-level hierarchy is the inverse of the pressure operator, compared with a dense
solve at sizes around a panel (8 columns), a warp (32 rows) and a CTA (1024 rows)."""
from fractions import Fraction

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


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def _lu_inverse(M):
    """Inverse by LU with partial pivoting (smallest row on ties) and forward and back substitution of the unit vectors,
    in plain order; every a - l u is rounded once, every quotient is the rounded quotient."""
    n = len(M)
    A = [[float(v) for v in row] for row in M]
    order = list(range(n))
    for k in range(n):
        p = max(range(k, n), key=lambda i: (abs(A[i][k]), -i))
        A[k], A[p] = A[p], A[k]
        order[k], order[p] = order[p], order[k]
        for i in range(k + 1, n):
            A[i][k] /= A[k][k]
            for q in range(k + 1, n):
                A[i][q] = _fma(-A[i][k], A[k][q], A[i][q])
    X = np.empty((n, n))
    for j in range(n):
        x = [1.0 if o == j else 0.0 for o in order]
        for k in range(n):
            for i in range(k + 1, n):
                x[i] = _fma(-A[i][k], x[k], x[i])
        for k in range(n - 1, -1, -1):
            x[k] /= A[k][k]
            for i in range(k):
                x[i] = _fma(-A[i][k], x[k], x[i])
        X[:, j] = x
    return X


@pytest.mark.parametrize("dims", [(7, 1, 1), (3, 3, 1), (5, 2, 2), (11, 3, 1), (5, 3, 3)])
def test_inverse_rounds_like_plain_elimination(dims):
    """Bit for bit: panels and parallel updates change no operation and no order."""
    torch = pytest.importorskip("torch")
    import paper_1602_05901_gb300 as rsv
    p = synth.make_problem(*dims, seed=19)
    A = rsv.Matrix(*dims, precision="fp64")
    A.set_values(p.vals)
    s = rsv.Solver(A)
    s.setup("cpr", gmg_max_levels=1)
    _, _, a7 = s.cpr_info()
    ref = _lu_inverse(stencil_to_dense(*dims, a7[0]))
    x = torch.zeros(A.nb, dtype=torch.float64, device="cuda")
    for j in range(A.nb):
        s.vcycle(torch.eye(A.nb, dtype=torch.float64, device="cuda")[j].contiguous(), x)
        assert np.array_equal(x.cpu().numpy(), ref[:, j]), j


def test_singular_pressure_operator_is_refused():
    """A closed chain without accumulation: the pressure operator's rows sum to zero, and its elimination (multipliers of -1)
    ends with a pivot of exactly zero, whatever the transmissibility; 1/49 is not a power of two.  The block factor's last
    pivot is rounding, not zero, so the pressure operator alone is what reports it."""
    import paper_1602_05901_gb300 as rsv
    n, t = 20, 49.0
    A = rsv.Matrix(n, 1, 1, precision="fp64")
    vals = np.zeros((len(A.col_idx), 3, 3))
    for c in range(n):
        for q in range(A.row_ptr[c], A.row_ptr[c + 1]):
            if A.col_idx[q] == c:
                vals[q] = np.diag([t * (A.row_ptr[c + 1] - A.row_ptr[c] - 1), 1.0, 1.0])
            else:
                vals[q, 0, 0] = -t
    A.set_values(vals)
    s = rsv.Solver(A)
    s.setup("bilu0")
    with pytest.raises(rsv.RsvError) as e:
        s.setup("cpr")
    assert e.value.status == rsv.RSV_ESINGULAR
