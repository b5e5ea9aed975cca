"""One GMRES cycle on systems around the sizes where the Gram-Schmidt kernels change their grid (one row per thread up to
152 x 256 unknowns): the residual after m steps against textbook GMRES (modified Gram-Schmidt, twice) in FP64."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _textbook(torch, A, dinv, b, m):
    """||b - A x_m|| / ||b|| of right-preconditioned GMRES with block Jacobi from x = 0."""
    n = b.numel()
    V = torch.zeros(m + 1, n, dtype=torch.float64, device="cuda")
    H = np.zeros((m + 1, m))
    beta = b.norm()
    V[0] = b / beta
    w = torch.zeros_like(b)
    for j in range(m):
        A.spmv(torch.einsum("cij,cj->ci", dinv, V[j].view(-1, 3)).reshape(-1).contiguous(), w)
        u = w.clone()
        for _ in range(2):
            for i in range(j + 1):
                h = torch.dot(u, V[i])
                H[i, j] += float(h)
                u -= h * V[i]
        H[j + 1, j] = float(u.norm())
        V[j + 1] = u / H[j + 1, j]
    e = np.zeros(m + 1)
    e[0] = 1.0
    y = np.linalg.lstsq(H, e, rcond=None)[0]
    return float(np.linalg.norm(e - H @ y))


# (nx, ny, nz, m): one CTA, three full ones, the last size of the small grid with eight groups of basis vectors, and the
# first size of the full grid
CASES = [(5, 3, 2, 12), (16, 16, 1, 30), (24, 20, 27, 64), (26, 20, 25, 64), (20, 20, 10, 33)]


@pytest.mark.parametrize("case", CASES, ids=["{}x{}x{}_m{}".format(*c) for c in CASES])
def test_gmres_cycle_small_systems(case):
    torch = pytest.importorskip("torch")
    import paper_1602_05901_gb300 as rsv
    nx, ny, nz, m = case
    p = synth.make_problem(nx, ny, nz, seed=11)
    A = rsv.Matrix(nx, ny, nz)
    A.set_values(p.vals)
    s = rsv.Solver(A, solver="gmres", restart=m, rtol=1e-15, maxit=m)
    s.setup("bjacobi")
    b = torch.from_numpy(p.b).cuda()
    x = torch.zeros_like(b)
    _, info = s.solve(b, x)
    assert info["iters"] == m
    ref = _textbook(torch, A, torch.from_numpy(s.dinv()).cuda(), b, m)
    # both bases are orthogonal to a few units of rounding per vector (2^-53 m sqrt(m) < 1e-13), and the least residual
    # moves by no more than that relative to ||b||; one more order for the update x = M^-1 V y
    assert abs(info["true_relres"] - ref) <= 1e-12, (info["true_relres"], ref)
