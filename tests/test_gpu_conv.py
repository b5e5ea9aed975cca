"""Tensor-core convolutions (forward, input gradient, weight gradient) against the FP64 oracle.

Both sides use the same BF16 operands; the GPU accumulates exact BF16
products in FP32, so the bound used is the classical one for a recursive FP32
sum of K terms, |err| <= K * 2^-24 * sum|terms| (doubled for margin), taken
element by element from the oracle's sum of absolute products.
"""
import ctypes

import numpy as np
import pytest

from oracle import unet as U

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24


@pytest.fixture(scope="module")
def rsv():
    import paper_1602_05901_gb300 as rsv
    return rsv


def _bf16(torch, a):
    """(device BF16 tensor, the same values as float64 numpy)."""
    t = torch.tensor(np.ascontiguousarray(a), dtype=torch.float32).to(torch.bfloat16)
    return t.cuda(), t.float().double().numpy()


def _p(t):
    return ctypes.c_void_p(t.data_ptr()) if t is not None else None


def _vol(rng, nz, ny, nx, c, ld=None, scale=1.0):
    ld = ld or c
    a = np.zeros((nz, ny, nx, ld))
    a[..., :c] = rng.standard_normal((nz, ny, nx, c)) * scale
    return a


FWD_CASES = [
    # (nx, ny, nz, taps, ci, co, ldx, relu, bias)
    (16, 8, 4, 1, 64, 32, 64, False, False),      # plain GEMM, 4 tiles
    (20, 12, 6, 27, 32, 32, 40, False, False),    # BK = 32, ragged tiles (120 of 128 rows used), ldx > ci
    (16, 16, 8, 27, 128, 256, 128, True, True),   # coarsest U-Net level, BN = 256
    (8, 8, 4, 27, 384, 128, 384, True, True),     # concatenated input, 3 K blocks of 128
    (32, 8, 5, 27, 64, 96, 64, True, True),       # BN = 96, ragged z
    (24, 4, 3, 27, 96, 192, 104, False, True),    # ci = 96 (BK = 32), BN = 192, ragged x tiles
]


@pytest.mark.parametrize("case", FWD_CASES, ids=[f"{c[0]}x{c[1]}x{c[2]}_t{c[3]}_ci{c[4]}_co{c[5]}" for c in FWD_CASES])
def test_conv_fwd_matches_oracle(rsv, case):
    torch = pytest.importorskip("torch")
    nx, ny, nz, taps, ci, co, ldx, relu, use_bias = case
    rng = np.random.default_rng(sum(case[:6]))
    xt, xh = _bf16(torch, _vol(rng, nz, ny, nx, ci, ldx))
    w = rng.standard_normal((co, taps, ci)) * np.sqrt(2.0 / (taps * ci))
    wt, wh = _bf16(torch, w)
    bias = rng.standard_normal(co).astype(np.float32) * 0.1 if use_bias else None
    bt = torch.tensor(bias).cuda() if use_bias else None
    y32 = torch.full((nz * ny * nx, co), float("nan"), device="cuda")
    ldy = co + 32
    yb = torch.zeros((nz * ny * nx, ldy), dtype=torch.bfloat16, device="cuda")
    st = rsv.rsv_conv3d_fwd(None, nx, ny, nz, taps, ci, co, _p(xt), ldx, _p(wt), _p(bt), int(relu), None, 0,
                            ctypes.c_void_p(yb.data_ptr() + 64), ldy, _p(y32))
    assert st == rsv.RSV_OK, rsv.status_string(st)
    x = xh[..., :ci]
    if taps == 27:
        ref = U.conv3(x, wh)
        absref = U.conv3(np.abs(x), np.abs(wh))
    else:
        ref = x @ wh[:, 0, :].T
        absref = np.abs(x) @ np.abs(wh[:, 0, :]).T
    if use_bias:
        ref = ref + bias
        absref = absref + np.abs(bias)
    if relu:
        ref = np.maximum(ref, 0)
    got = y32.cpu().double().numpy().reshape(ref.shape)
    tol = 2 * (taps * ci + 1) * U32 * absref + 1e-30
    assert np.all(np.abs(got - ref) <= tol), np.max(np.abs(got - ref) / tol)
    # BF16 output: the round-to-nearest of the FP32 result, at channel offset 32 of rows of ldy
    gb = yb.float().cpu().double().numpy().reshape(nz, ny, nx, ldy)[..., 32:32 + co]
    assert np.array_equal(gb, U.bf16_round(got))
    assert np.all(yb.float().cpu().numpy().reshape(nz, ny, nx, ldy)[..., :32] == 0)


def test_conv_dgrad_with_relu_mask(rsv):
    torch = pytest.importorskip("torch")
    nx, ny, nz, ci, co = 16, 8, 4, 96, 32
    rng = np.random.default_rng(5)
    gyt, gyh = _bf16(torch, _vol(rng, nz, ny, nx, co))
    w = rng.standard_normal((co, 27, ci)) * 0.1
    wt, wh = _bf16(torch, w)
    mask = rng.standard_normal((nz, ny, nx, ci))
    mt, mh = _bf16(torch, mask)
    gx32 = torch.full((nz * ny * nx, ci), float("nan"), device="cuda")
    st = rsv.rsv_conv3d_dgrad(None, nx, ny, nz, ci, co, _p(gyt), co, _p(wt), _p(mt), ci, None, 0, _p(gx32))
    assert st == rsv.RSV_OK, rsv.status_string(st)
    ref = U.conv3_dgrad(gyh, wh) * (mh > 0)
    absref = U.conv3_dgrad(np.abs(gyh), np.abs(wh))
    got = gx32.cpu().double().numpy().reshape(ref.shape)
    assert np.all(np.abs(got - ref) <= 2 * 27 * co * U32 * absref + 1e-30)
    assert np.all(got[mh <= 0] == 0)


WG_CASES = [
    # (nx, ny, nz, taps, ci, co)
    (16, 8, 6, 27, 32, 32),
    (8, 8, 4, 27, 96, 32),
    (16, 4, 4, 1, 64, 32),
    (16, 16, 8, 27, 128, 256),
    (24, 5, 3, 27, 64, 96),      # no 64-voxel box fits: the voxel-major copy path
    (16, 8, 8, 27, 192, 64),     # ci > co: rows = (tap, output channel), N = 192
    (16, 8, 4, 27, 384, 128),    # ci > co: two N tiles of 192
    (32, 4, 3, 27, 96, 32),      # ci > co with ragged z chunks
]


@pytest.mark.parametrize("case", WG_CASES, ids=[f"{c[0]}x{c[1]}x{c[2]}_t{c[3]}_ci{c[4]}_co{c[5]}" for c in WG_CASES])
def test_conv_wgrad_matches_oracle(rsv, case):
    torch = pytest.importorskip("torch")
    nx, ny, nz, taps, ci, co = case
    rng = np.random.default_rng(100 + sum(case))
    ldx = ci + 8
    xt, xh = _bf16(torch, _vol(rng, nz, ny, nx, ci, ldx))
    gyt, gyh = _bf16(torch, _vol(rng, nz, ny, nx, co))
    gw = torch.full((co, taps, ci), float("nan"), device="cuda")
    gb = torch.full((co,), float("nan"), device="cuda")
    st = rsv.rsv_conv3d_wgrad(None, nx, ny, nz, taps, ci, co, _p(xt), ldx, _p(gyt), co, _p(gw), _p(gb))
    assert st == rsv.RSV_OK, rsv.status_string(st)
    x = xh[..., :ci]
    if taps == 27:
        ref, absref = U.conv3_wgrad(gyh, x), U.conv3_wgrad(np.abs(gyh), np.abs(x))
    else:
        ref = (gyh.reshape(-1, co).T @ x.reshape(-1, ci))[:, None, :]
        absref = (np.abs(gyh).reshape(-1, co).T @ np.abs(x).reshape(-1, ci))[:, None, :]
    nvox = nx * ny * nz
    got = gw.cpu().double().numpy()
    assert np.all(np.abs(got - ref) <= 2 * nvox * U32 * absref + 1e-30), np.nanmax(np.abs(got - ref) / absref)
    gbr = gyh.reshape(-1, co).sum(axis=0)
    assert np.allclose(gb.cpu().double().numpy(), gbr, rtol=0, atol=2 * nvox * U32 * np.abs(gyh).reshape(-1, co).sum(0).max())


def test_conv_argument_checks(rsv):
    torch = pytest.importorskip("torch")
    x = torch.zeros(64 * 40, dtype=torch.bfloat16, device="cuda")
    w = torch.zeros(32 * 40, dtype=torch.bfloat16, device="cuda")
    y = torch.zeros(64 * 32, dtype=torch.float32, device="cuda")
    # ci not a multiple of 32, taps not 1 or 27, misaligned leading dimension
    assert rsv.rsv_conv3d_fwd(None, 4, 4, 4, 1, 40, 32, _p(x), 40, _p(w), None, 0, None, 0, None, 0, _p(y)) == rsv.RSV_EINVAL
    assert rsv.rsv_conv3d_fwd(None, 4, 4, 4, 9, 32, 32, _p(x), 32, _p(w), None, 0, None, 0, None, 0, _p(y)) == rsv.RSV_EINVAL
    assert rsv.rsv_conv3d_fwd(None, 4, 4, 4, 1, 32, 32, _p(x), 36, _p(w), None, 0, None, 0, None, 0, _p(y)) == rsv.RSV_EINVAL
    assert rsv.rsv_conv3d_wgrad(None, 6, 4, 4, 27, 32, 32, _p(x), 32, _p(x), 32, _p(y), None) == rsv.RSV_EINVAL


# The folded form's edges: rows that do not fill a tile (24 x 5 = 120, 40 x 3), an odd count of tile rows in y, a tile
# row of one voxel row (nx = 128), weights resident and streamed, and its neighbours that take the general kernel
# (nx not a multiple of 8, one tile in y, more than 128 voxels in x).
FOLD_CASES = [
    (24, 11, 3, 32, 32), (40, 7, 2, 64, 64), (128, 3, 3, 32, 32), (128, 2, 2, 96, 32), (64, 5, 3, 64, 32),
    (8, 33, 2, 192, 64), (64, 4, 70, 32, 32), (20, 13, 3, 32, 32), (16, 8, 3, 32, 64), (136, 3, 2, 32, 32),
]


@pytest.mark.parametrize("case", FOLD_CASES, ids=[f"{c[0]}x{c[1]}x{c[2]}_ci{c[3]}_co{c[4]}" for c in FOLD_CASES])
def test_conv_narrow_layers_match_oracle(rsv, case):
    """Same bound as above: K = 27 ci exact products summed in FP32, plus the bias."""
    torch = pytest.importorskip("torch")
    nx, ny, nz, ci, co = case
    rng = np.random.default_rng(sum(case))
    xt, xh = _bf16(torch, _vol(rng, nz, ny, nx, ci))
    wt, wh = _bf16(torch, rng.standard_normal((co, 27, ci)) * np.sqrt(2.0 / (27 * ci)))
    bias = rng.standard_normal(co).astype(np.float32) * 0.1
    y32 = torch.full((nz * ny * nx, co), float("nan"), device="cuda")
    st = rsv.rsv_conv3d_fwd(None, nx, ny, nz, 27, ci, co, _p(xt), ci, _p(wt), _p(torch.tensor(bias).cuda()), 0, None, 0,
                            None, 0, _p(y32))
    assert st == rsv.RSV_OK, rsv.status_string(st)
    ref = U.conv3(xh, wh) + bias
    absref = U.conv3(np.abs(xh), np.abs(wh)) + np.abs(bias)
    got = y32.cpu().numpy().reshape(ref.shape)
    assert np.all(np.abs(got - ref) <= 2 * (27 * ci + 1) * U32 * absref)


# More pairs of tiles than CTAs, so that a CTA walks along z and over the end of a column: boxes of three planes kept
# (weights resident: 32 channels; through a ring: 64), one box at a time (rows of 128 voxels, several channel blocks).
WALK_CASES = [
    (32, 40, 40, 32, 32), (40, 21, 50, 32, 64), (16, 66, 40, 64, 64), (64, 10, 60, 64, 32), (128, 4, 90, 64, 64),
    (128, 3, 90, 64, 32), (32, 33, 40, 128, 64), (64, 7, 80, 96, 32),
]


@pytest.mark.parametrize("case", WALK_CASES, ids=[f"{c[0]}x{c[1]}x{c[2]}_ci{c[3]}_co{c[4]}" for c in WALK_CASES])
def test_conv_narrow_layers_walk(rsv, case):
    test_conv_narrow_layers_match_oracle(rsv, case)


# The weight gradient by whole rows of a plane: odd and single rows, rows of 8 and 128 voxels, two shared-memory stages
# (128 x 64 channels), every block of rows (128, 64, 32 channels) in both roles, more channels than a thread block
# has in the bias gradient; a leading dimension that 16-byte loads cannot take; rows too long for it.
ROW_CASES = [
    # (nx, ny, nz, ci, co, extra ldx)
    (8, 1, 1, 32, 32, 8),
    (8, 5, 3, 32, 512, 0),
    (24, 7, 5, 96, 64, 0),
    (40, 3, 9, 64, 64, 8),
    (120, 3, 2, 32, 64, 0),
    (104, 3, 2, 64, 64, 0),
    (128, 4, 2, 64, 64, 0),
    (128, 3, 3, 32, 32, 0),
    (64, 21, 4, 64, 128, 0),
    (16, 6, 5, 128, 96, 0),
    (24, 5, 3, 64, 32, 4),
    (136, 3, 2, 32, 32, 0),
]


@pytest.mark.parametrize("case", ROW_CASES, ids=["{}x{}x{}_ci{}_co{}_pad{}".format(*c) for c in ROW_CASES])
def test_conv_wgrad_rows(rsv, case):
    torch = pytest.importorskip("torch")
    nx, ny, nz, ci, co, pad = case
    rng = np.random.default_rng(500 + sum(case))
    xt, xh = _bf16(torch, _vol(rng, nz, ny, nx, ci, ci + pad))
    gyt, gyh = _bf16(torch, _vol(rng, nz, ny, nx, co))
    gw = torch.full((co, 27, ci), float("nan"), device="cuda")
    gb = torch.full((co,), float("nan"), device="cuda")
    st = rsv.rsv_conv3d_wgrad(None, nx, ny, nz, 27, ci, co, _p(xt), ci + pad, _p(gyt), co, _p(gw), _p(gb))
    assert st == rsv.RSV_OK, rsv.status_string(st)
    x = xh[..., :ci]
    ref, absref = U.conv3_wgrad(gyh, x), U.conv3_wgrad(np.abs(gyh), np.abs(x))
    nvox = nx * ny * nz
    # one FP32 rounding per product and addition of at most nvox terms
    assert np.all(np.abs(gw.cpu().double().numpy() - ref) <= 2 * nvox * U32 * absref + 1e-30)
    flat = gyh.reshape(-1, co)
    assert np.all(np.abs(gb.cpu().double().numpy() - flat.sum(0)) <= 2 * nvox * U32 * np.abs(flat).sum(0) + 1e-30)


# The weight gradient's other forms at 27 taps, which the form by whole rows leaves to longer rows and unaligned leading
# dimensions.  (The 27-tap cases of WG_CASES all take the form by whole rows now; the labels beside them name what they
# took without it.)  Here: boxes of 64 voxels with either operand shifted, N = 192 and 256, several N tiles and channel blocks, ragged boxes; voxel-major copies with several blocks of
# 128 and of 32 channels.
OTHER_CASES = [
    # (nx, ny, nz, ci, co, extra ldx)
    (136, 5, 3, 192, 64, 8),
    (136, 2, 2, 384, 128, 0),
    (144, 3, 3, 128, 256, 8),
    (136, 1, 5, 96, 32, 0),
    (192, 3, 1, 32, 96, 0),
    (24, 5, 3, 256, 96, 4),
    (40, 3, 5, 160, 64, 4),
]


@pytest.mark.parametrize("case", OTHER_CASES, ids=["{}x{}x{}_ci{}_co{}_pad{}".format(*c) for c in OTHER_CASES])
def test_conv_wgrad_long_rows_and_unaligned(rsv, case):
    test_conv_wgrad_rows(rsv, case)


# The folded form with everything a layer's call can carry: rows that leave part of a tile invalid, one and two accumulator
# sets, resident and streamed weights, kept planes and one box at a time, a single pair and several per CTA.
FULL_CASES = [
    (24, 11, 3, 32, 32), (40, 7, 2, 64, 64), (128, 3, 3, 96, 32), (40, 21, 50, 32, 64), (32, 40, 40, 32, 32),
    (16, 66, 40, 64, 64), (128, 3, 90, 64, 32), (64, 5, 3, 192, 64),
]
FULL_IDS = [f"{c[0]}x{c[1]}x{c[2]}_ci{c[3]}_co{c[4]}" for c in FULL_CASES]


def _at(t, channel):
    return ctypes.c_void_p(t.data_ptr() + 2 * channel)


@pytest.mark.parametrize("relu,use_bias,masked", [(True, True, False), (False, False, True), (True, False, True)])
@pytest.mark.parametrize("case", FULL_CASES, ids=FULL_IDS)
def test_conv_narrow_layers_full_call(rsv, case, relu, use_bias, masked):
    """Padded input, a mask and a BF16 output at a channel offset of a wider tensor.  Same bound as above; the BF16 output is the
    round-to-nearest of the FP32 one, and the channels beside it stay as they were."""
    torch = pytest.importorskip("torch")
    nx, ny, nz, ci, co = case
    rng = np.random.default_rng(700 + sum(case))
    ldx, ldy, ldm = ci + 16, co + 48, co + 8
    xt, xh = _bf16(torch, rng.standard_normal((nz, ny, nx, ldx)))
    xh = xh[..., 8:8 + ci]
    wt, wh = _bf16(torch, rng.standard_normal((co, 27, ci)) * np.sqrt(2.0 / (27 * ci)))
    bias = rng.standard_normal(co).astype(np.float32) * 0.1
    bt = torch.tensor(bias).cuda()
    mt, mh = _bf16(torch, rng.standard_normal((nz, ny, nx, ldm)))
    y32 = torch.full((nz * ny * nx, co), float("nan"), device="cuda")
    yb = torch.full((nz * ny * nx, ldy), 3.0, dtype=torch.bfloat16, device="cuda")
    st = rsv.rsv_conv3d_fwd(None, nx, ny, nz, 27, ci, co, _at(xt, 8), ldx, _p(wt), _p(bt) if use_bias else None, int(relu),
                            _at(mt, 8) if masked else None, ldm if masked else 0, _at(yb, 32), ldy, _p(y32))
    assert st == rsv.RSV_OK, rsv.status_string(st)
    ref, absref = U.conv3(xh, wh), U.conv3(np.abs(xh), np.abs(wh))
    if use_bias:
        ref, absref = ref + bias, absref + np.abs(bias)
    if relu:
        ref = np.maximum(ref, 0)
    if masked:
        ref = ref * (mh[..., 8:8 + co] > 0)
    got = y32.cpu().double().numpy().reshape(ref.shape)
    assert np.all(np.abs(got - ref) <= 2 * (27 * ci + 1) * U32 * absref)
    gb = yb.float().cpu().double().numpy().reshape(nz, ny, nx, ldy)
    assert np.array_equal(gb[..., 32:32 + co], U.bf16_round(got))
    assert np.all(gb[..., :32] == 3) and np.all(gb[..., 32 + co:] == 3)


@pytest.mark.parametrize("case", FULL_CASES, ids=FULL_IDS)
def test_conv_narrow_layers_input_gradient(rsv, case):
    """The layer's output channels are the case's ci, its input channels (the gradient's) the case's co; masked by an
    activation inside a wider tensor, BF16 at a channel offset."""
    torch = pytest.importorskip("torch")
    nx, ny, nz, co, ci = case
    rng = np.random.default_rng(800 + sum(case))
    ldm, ldgx = ci + 24, ci + 16
    gyt, gyh = _bf16(torch, _vol(rng, nz, ny, nx, co, co + 8))
    wt, wh = _bf16(torch, rng.standard_normal((co, 27, ci)) * 0.1)
    mt, mh = _bf16(torch, rng.standard_normal((nz, ny, nx, ldm)))
    mh = mh[..., 16:16 + ci]
    gx32 = torch.full((nz * ny * nx, ci), float("nan"), device="cuda")
    gxb = torch.full((nz * ny * nx, ldgx), 3.0, dtype=torch.bfloat16, device="cuda")
    st = rsv.rsv_conv3d_dgrad(None, nx, ny, nz, ci, co, _p(gyt), co + 8, _p(wt), _at(mt, 16), ldm, _at(gxb, 8), ldgx, _p(gx32))
    assert st == rsv.RSV_OK, rsv.status_string(st)
    gyh = gyh[..., :co]
    ref, absref = U.conv3_dgrad(gyh, wh) * (mh > 0), U.conv3_dgrad(np.abs(gyh), np.abs(wh))
    got = gx32.cpu().double().numpy().reshape(ref.shape)
    assert np.all(np.abs(got - ref) <= 2 * 27 * co * U32 * absref + 1e-30)
    gb = gxb.float().cpu().double().numpy().reshape(nz, ny, nx, ldgx)
    assert np.array_equal(gb[..., 8:8 + ci], U.bf16_round(got))
    assert np.all(gb[..., :8] == 3) and np.all(gb[..., 8 + ci:] == 3)


@pytest.mark.parametrize("case", [(24, 21, 30, 384, 128), (40, 24, 20, 96, 32), (24, 20, 20, 256, 256), (40, 9, 12, 64, 64)],
                         ids=lambda c: "{}x{}x{}_ci{}_co{}".format(*c))
def test_conv_wgrad_forms_are_equally_accurate(rsv, case):
    """The form by whole rows and the one by voxel-major copies (a leading dimension that 16-byte loads cannot take) on the same
    values: both sum in FP32, whose error grows with the voxels that one accumulator takes.  The rows' form may take no
    more of them, so its error against 64 bits is no larger, but for a quarter of scatter."""
    torch = pytest.importorskip("torch")
    nx, ny, nz, ci, co = case
    rng = np.random.default_rng(900 + sum(case))
    x = np.maximum(_vol(rng, nz, ny, nx, ci, ci + 4), 0)
    gyt, gyh = _bf16(torch, _vol(rng, nz, ny, nx, co))
    ref = U.conv3_wgrad(gyh, _bf16(torch, x[..., :ci])[1])
    error = []
    for ld in (ci, ci + 4):
        xt, _ = _bf16(torch, x[..., :ld])
        gw = torch.full((co, 27, ci), float("nan"), device="cuda")
        st = rsv.rsv_conv3d_wgrad(None, nx, ny, nz, 27, ci, co, _p(xt), ld, _p(gyt), co, _p(gw), None)
        assert st == rsv.RSV_OK, rsv.status_string(st)
        error.append(np.linalg.norm(gw.cpu().double().numpy() - ref) / np.linalg.norm(ref))
    assert error[0] <= 1.25 * error[1], error
