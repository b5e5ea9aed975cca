"""FP64 -> FP32 and FP32 -> FP64 conversions in integer arithmetic (matrix copy, factor input) against the hardware-defined ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rsv():
    from tests.helpers import build_library
    build_library()
    import paper_1602_05901_gb300 as m
    return m


def _values():
    """Doubles around everything that rounding to FP32 decides: ties with even and odd last bits and their neighbours, carries
    across a power of two, every exponent from below the smallest subnormal to above the largest float, random bits."""
    e = np.arange(-152, 130)
    head = np.array([1.0, 1.0 + 2.0 ** -23, 1.5, 2.0 - 2.0 ** -22, 2.0 - 2.0 ** -23])
    rest = np.array([0.0, 2.0 ** -24, 2.0 ** -24 - 2.0 ** -52, 2.0 ** -24 + 2.0 ** -52, 2.0 ** -25, 3 * 2.0 ** -25])
    v = np.ldexp((head[:, None] + rest).ravel()[None, :], e[:, None]).ravel()
    r = np.random.default_rng(41)
    v = np.concatenate([v, np.ldexp(1.0 + r.random(2000), r.integers(-155, 132, 2000))])
    return np.concatenate([v, -v])


def _chain(rsv, precision, column):
    """A chain of cells whose diagonal blocks hold `column` in their first columns and ones elsewhere on the diagonal; the
    count of matrix entries is no multiple of four."""
    n = len(column) // 3
    while 9 * (3 * n - 2) % 4 == 0:
        n -= 1
    A = rsv.Matrix(n, 1, 1, precision=precision)
    vals = np.zeros((len(A.col_idx), 3, 3))
    rows = np.repeat(np.arange(n), np.diff(A.row_ptr))
    vals[A.col_idx == rows, :, 0] = column[:3 * n].reshape(n, 3)
    return A, n, vals


@pytest.mark.parametrize("source", ["host", "device", "device, 8 bytes off a 16-byte boundary"])
def test_matrix_copies_are_the_correctly_rounded_values(rsv, source):
    """A times the vector that picks the first columns: one product with 1 per entry, exact in either precision."""
    torch = pytest.importorskip("torch")
    column = np.concatenate([_values(), [np.inf, -np.inf, np.nan]])
    column = np.concatenate([column[-3:], column])
    A, n, vals = _chain(rsv, "mixed", column)
    if source == "host":
        A.set_values(vals)
    else:
        buf = torch.zeros(vals.size + 1, dtype=torch.float64, device="cuda")
        t = buf[1:] if "off" in source else buf[:-1]
        assert (t.data_ptr() % 16 == 8) == ("off" in source)
        t.copy_(torch.from_numpy(vals.ravel()))
        A.set_values(t)
    pick = torch.zeros(3 * n, dtype=torch.float64, device="cuda")
    pick[::3] = 1.0
    with np.errstate(over="ignore"):
        ref32 = column[:3 * n].astype(np.float32)
    for x, ref in ((pick, column[:3 * n]), (pick.float(), ref32)):
        y = torch.empty_like(x)
        A.spmv(x, y)
        assert np.array_equal(y.cpu().numpy(), ref, equal_nan=True)


def test_factor_input_is_the_widened_float(rsv):
    """A diagonal block diag(v, 1, 1) without neighbours' entries: its inverse's first entry is the rounded 1 / v, with v
    the FP32 value widened exactly."""
    with np.errstate(over="ignore"):
        v = _values().astype(np.float32)
    v = v[np.isfinite(v) & (v != 0)].astype(np.float64)
    column = np.zeros(3 * len(v))
    column[::3] = v
    A, n, vals = _chain(rsv, "mixed", column)
    diag = np.repeat(np.arange(n), np.diff(A.row_ptr)) == A.col_idx
    vals[diag, 1, 1] = vals[diag, 2, 2] = 1.0
    A.set_values(vals)
    s = rsv.Solver(A, precision="mixed")
    s.setup("bilu0")
    assert np.array_equal(s.dinv().reshape(n, 3, 3)[:, 0, 0], 1.0 / v[:n])
