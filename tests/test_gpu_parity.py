"""GPU parity: every step of the CUDA path against the CPU oracle, through the C ABI.

Integer results (codes, permutation, accumulators) must match bit for bit; fp32 outputs are a
single multiply of exactly converted integers and must match bit for bit too, and lie within
1e-6 relative of the double-precision value.
"""
import numpy as np
import pytest

from oracle import rmsmp_oracle as O
from paper_2111_00153_b200 import binding as R
from paper_2111_00153_b200 import synth
from tests import harness as Hn

pytestmark = pytest.mark.gpu

VARIANTS = [R.VARIANT_SIMPLE, R.VARIANT_SIMT, R.VARIANT_SHIFTADD, R.VARIANT_TENSOR, Hn.WORKSPACE]
VNAME = {R.VARIANT_SIMPLE: "simple", R.VARIANT_SIMT: "simt", R.VARIANT_SHIFTADD: "shiftadd",
         R.VARIANT_TENSOR: "tensor", R.VARIANT_AUTO: "auto", Hn.WORKSPACE: "workspace"}


def _mixed_map(M, seed, ratio=(60, 35, 5)):
    """A scheme map with the given ratio, rows shuffled (independent of weight values)."""
    nP, nF4, n8 = O.ratio_counts(M, ratio)
    kinds = np.array([0] * nP + [1] * nF4 + [2] * n8)
    np.random.default_rng(seed).shuffle(kinds)
    scheme = np.where(kinds == 0, 0, 1).astype(np.uint8)
    bits = np.where(kinds == 2, 8, 4).astype(np.uint8)
    return scheme, bits


def _check_layer_outputs(y, acc, acc_ref, ws, act_step, alpha, scheme, bits):
    assert np.array_equal(acc, acc_ref)
    y_ref = O.epilogue(acc_ref, ws, act_step)
    assert np.array_equal(y.view(np.uint32), y_ref.view(np.uint32))
    Qw = np.where(scheme == 0, 64.0, np.where(bits == 4, 7.0, 127.0))
    dbl = acc_ref.astype(np.float64) * (alpha.astype(np.float64) / Qw)[None, :] * float(act_step)
    nz = dbl != 0
    assert np.all(np.abs(y[nz] - dbl[nz]) <= 1e-6 * np.abs(dbl[nz]))


# ------------------------------------------------------------------ pack / unpack

@pytest.mark.parametrize("M,K,ratio", [(256, 512, (60, 35, 5)), (37, 200, (50, 40, 10)),
                                       (5, 3, (0, 100, 0)), (130, 1000, (100, 0, 0)),
                                       (64, 40000, (60, 35, 5)), (3, 7, (34, 33, 33))])
@pytest.mark.parametrize("mode", [R.POT_NEAREST, R.POT_LOG2])
def test_pack_codes_linear(M, K, ratio, mode):
    if mode == R.POT_LOG2 and K > 2000:
        pytest.skip("one large case per mode is enough")
    W = synth.weights_normal(synth.rng(70, M + K), (M, K))
    W[0, :min(K, 8)] = [0, 1e-9, -1e-9, 1, -1, 0.02, -0.02, 3e-4][:min(K, 8)]
    scheme, bits = O.assign_rows(W, ratio)
    alpha = synth.alpha_rows(W)
    layer, d_packed = Hn.pack_layer(W, scheme, bits, alpha, mode)
    vals, perm, ws = Hn.unpack(layer, d_packed)
    v_ref, ws_ref = O.quantize_rows(W, scheme, bits, alpha, mode)
    assert np.array_equal(vals, v_ref)
    assert np.array_equal(perm, O.group_rows(scheme, bits))
    assert np.array_equal(ws.view(np.uint32), ws_ref.view(np.uint32))


def test_pack_codes_on_rounding_ties_and_midpoints():
    # weights placed exactly on Fixed rounding ties and PoT decision points, alpha = 1
    ties4 = [np.float32((j + 0.5) / 7.0) for j in range(7)]
    ties8 = [np.float32((j + 0.5) / 127.0) for j in range(0, 127, 9)]
    mids = [2.0 ** -7] + [3 * 2.0 ** (k - 9) for k in range(2, 8)]
    geo = [2.0 ** -(j + 0.5) for j in range(7)]
    pts = []
    for v in ties4 + ties8 + mids + geo:
        f = np.float32(v)
        pts += [f, np.nextafter(f, np.float32(0)), np.nextafter(f, np.float32(2)), -f]
    K = len(pts)
    W = np.tile(np.array(pts, np.float32), (6, 1))
    scheme = np.array([0, 1, 1, 0, 1, 1], np.uint8)
    bits = np.array([4, 4, 8, 4, 4, 8], np.uint8)
    alpha = np.array([1, 1, 1, 0.5, 0.5, 0.5], np.float32)
    for mode in (R.POT_NEAREST, R.POT_LOG2):
        layer, d_packed = Hn.pack_layer(W, scheme, bits, alpha, mode)
        vals, _, _ = Hn.unpack(layer, d_packed)
        v_ref, _ = O.quantize_rows(W, scheme, bits, alpha, mode)
        assert np.array_equal(vals, v_ref)


@pytest.mark.parametrize("M,Cin,k", [(64, 64, 3), (20, 24, 3), (9, 5, 1), (12, 40, 5), (130, 16, 2)])
def test_pack_codes_conv(M, Cin, k):
    W = synth.weights_kaiming(synth.rng(71, M + Cin), M, Cin, k, k)
    scheme, bits = O.assign_rows(W, (60, 35, 5))
    alpha = synth.alpha_rows(W)
    layer, d_packed = Hn.pack_layer(W, scheme, bits, alpha)
    vals, perm, ws = Hn.unpack(layer, d_packed)
    v_ref, ws_ref = O.quantize_rows(W.reshape(M, -1), scheme, bits, alpha)
    assert np.array_equal(vals, v_ref)
    assert np.array_equal(perm, O.group_rows(scheme, bits))


# ------------------------------------------------------------------ activation quantizer

@pytest.mark.parametrize("count", [1, 15, 16, 1000, 4099, 1 << 20])
@pytest.mark.parametrize("kind", [R.ACT_U4, R.ACT_S4])
def test_quantize_act(count, kind):
    g = synth.rng(72, count)
    x = synth.act_halfnormal(g, count) if kind == R.ACT_U4 else synth.act_normal(g, count)
    x[: min(count, 6)] = [0.0, 0.1, 0.3, 3.0, 1.5, 2.9999][: min(count, 6)]
    codes, step = Hn.quantize_act(x, synth.ALPHA_ACT, kind)
    c_ref, s_ref = O.quantize_act(x, synth.ALPHA_ACT, kind)
    assert np.array_equal(codes, c_ref)
    assert step == s_ref


@pytest.mark.parametrize("alpha", [3.0, 2.9999998, 1.0, 1e-3, 7.3e5, 1e-35, 1e33])
@pytest.mark.parametrize("kind", [R.ACT_U4, R.ACT_S4])
def test_quantize_act_on_rounding_boundaries(alpha, kind):
    # Values on and a few ulps around every rounding boundary (k + 0.5) * alpha / Q and every level,
    # around the clip points, plus specials, repeated until the warp-wide vector path is used.
    # The code near a boundary depends on the single correctly rounded division x / alpha.
    Q = 15 if kind == R.ACT_U4 else 7
    a32 = np.float32(alpha)
    ks = np.arange(-2 * Q - 3, 2 * Q + 4, dtype=np.float64) / 2.0          # levels and half-levels, beyond the clips
    centre = (ks * np.float64(a32) / Q).astype(np.float32)
    pts = [centre]
    for d in range(1, 5):
        up, dn = centre.copy(), centre.copy()
        for _ in range(d):
            up = np.nextafter(up, np.float32(np.inf)); dn = np.nextafter(dn, np.float32(-np.inf))
        pts += [up, dn]
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.finfo(np.float32).tiny, 1e-45, -1e-45,
                        np.finfo(np.float32).max], dtype=np.float32)
    x = np.concatenate(pts + [special]).astype(np.float32)
    g = synth.rng(72, 991)
    x = np.concatenate([x, g.permutation(np.tile(x, 8))])                  # > 4096 values, mixed inside each warp step
    codes, step = Hn.quantize_act(x, float(a32), kind)
    c_ref, s_ref = O.quantize_act(x, float(a32), kind)
    assert np.array_equal(codes, c_ref)
    assert step == s_ref


# ------------------------------------------------------------------ linear layer

LIN_CASES = [
    # M, K, N, ratio        spans several 128-row blocks / 256-token tiles with ragged tails
    (256, 512, 64, (60, 35, 5)),        # config 1
    (128, 128, 256, (60, 35, 5)),
    (300, 200, 77, (50, 40, 10)),
    (130, 96, 513, (60, 35, 5)),
    (64, 576, 300, (65, 30, 5)),
    (1, 32, 1, (0, 100, 0)),
    (200, 48, 40, (0, 0, 100)),
    (150, 1000, 33, (100, 0, 0)),
    (257, 2304, 260, (60, 35, 5)),
    (500, 640, 300, (60, 35, 5)),       # four row blocks: two per tile in the workspace variant, ragged last block
]


@pytest.mark.parametrize("variant", VARIANTS, ids=lambda v: VNAME[v])
@pytest.mark.parametrize("M,K,N,ratio", LIN_CASES)
def test_linear_layer(M, K, N, ratio, variant):
    g = synth.rng(73, M * 7 + K + N)
    W = synth.weights_normal(g, (M, K))
    scheme, bits = _mixed_map(M, M + K, ratio)
    alpha = synth.alpha_rows(W)
    signed = (M % 2 == 0)
    act = g.integers(-7, 8, (N, K), dtype=np.int8) if signed else synth.act_codes_uniform(g, (N, K))
    act_step = np.float32(0.1)
    layer, d_packed = Hn.pack_layer(W, scheme, bits, alpha)
    try:
        y, acc = Hn.gemm(layer, d_packed, act, act_step, variant)
    except R.RmsmpError as e:
        if e.status == R.ERR_VARIANT and variant in (R.VARIANT_TENSOR, Hn.WORKSPACE) and K % 16 != 0:
            pytest.skip("tensor variant needs K % 16 == 0")
        raise
    v_ref, ws = O.quantize_rows(W, scheme, bits, alpha)
    acc_ref = O.matmul(v_ref, act)
    _check_layer_outputs(y, acc, acc_ref, ws, act_step, alpha, scheme, bits)


@pytest.mark.parametrize("variant", [R.VARIANT_SIMT, R.VARIANT_TENSOR, R.VARIANT_AUTO, Hn.WORKSPACE], ids=lambda v: VNAME[v])
def test_linear_layer_mn_layout_and_padded_ld(variant):
    M, K, N = 140, 160, 70
    g = synth.rng(74, variant if isinstance(variant, int) else 9)
    W = synth.weights_normal(g, (M, K))
    scheme, bits = O.assign_rows(W, (60, 35, 5))
    alpha = synth.alpha_rows(W)
    act = synth.act_codes_uniform(g, (N, K))
    layer, d_packed = Hn.pack_layer(W, scheme, bits, alpha)
    y, acc = Hn.gemm(layer, d_packed, act, 0.25, variant, out_layout=R.OUT_MN, ld_act=192)
    v_ref, ws = O.quantize_rows(W, scheme, bits, alpha)
    _check_layer_outputs(y, acc, O.matmul(v_ref, act), ws, np.float32(0.25), alpha, scheme, bits)
    y2, _ = Hn.gemm(layer, d_packed, act, 0.25, variant, want_acc=False)
    assert np.array_equal(y2, y)


def test_extreme_codes_do_not_overflow_or_lose_bits():
    # every weight at full scale, every activation at 15: |acc| = K*127*15 on Fixed-8 rows
    M, K, N = 130, 4608, 40
    W = np.ones((M, K), np.float32)
    W[::2] = -1
    scheme, bits = _mixed_map(M, 5, (40, 30, 30))
    alpha = np.ones(M, np.float32)
    act = np.full((N, K), 15, np.int8)
    layer, d_packed = Hn.pack_layer(W, scheme, bits, alpha)
    v_ref, ws = O.quantize_rows(W, scheme, bits, alpha)
    acc_ref = O.matmul(v_ref, act)
    assert np.array_equal(acc_ref.astype(np.int64), O.matmul_i64(v_ref, act))
    assert np.abs(acc_ref).max() == K * 127 * 15
    for variant in VARIANTS:
        y, acc = Hn.gemm(layer, d_packed, act, 1.0, variant)
        _check_layer_outputs(y, acc, acc_ref, ws, np.float32(1.0), alpha, scheme, bits)


# ------------------------------------------------------------------ convolution

CONV_CASES = [
    # M, Cin, k, stride, pad, B, H, W
    (64, 64, 3, 1, 1, 2, 14, 14),
    (40, 32, 3, 2, 1, 3, 14, 14),
    (130, 128, 3, 1, 1, 2, 7, 7),
    (24, 16, 1, 2, 0, 2, 8, 8),
    (16, 16, 1, 1, 0, 1, 5, 9),
    (32, 48, 3, 2, 1, 2, 9, 12),      # odd sizes, non-square
    (140, 256, 3, 1, 1, 5, 7, 7),     # several images per tile, ragged last tile
    (20, 20, 3, 1, 1, 1, 6, 6),       # Cin not a multiple of 16: CUDA-core variants only
    (64, 64, 3, 1, 1, 1, 56, 56),
    (200, 64, 2, 1, 0, 2, 9, 9),      # 64-byte pixels, even tap count, two row blocks (weights through the ring)
    (96, 64, 3, 2, 1, 3, 7, 7),       # 64-byte pixels, several images per tile, stride 2
    (64, 48, 1, 1, 0, 2, 12, 12),     # 64-byte pixels, one tap
    (48, 32, 3, 2, 0, 2, 9, 11),      # stride 2 without padding, odd sizes: the parity sub-grids differ in extent
    (32, 64, 5, 2, 2, 2, 10, 7),      # stride 2, 5x5: taps two rows / columns outside the image
    (24, 32, 2, 2, 0, 3, 8, 6),       # stride 2, even kernel
    (40, 32, 3, 3, 1, 2, 10, 13),     # stride 3: element-strided boxes (no parity split)
    (300, 128, 3, 2, 1, 2, 28, 28),   # stride 2, three row blocks, tiles of whole output rows
    (48, 64, 3, 1, 1, 3, 16, 8),      # resident weights, width a multiple of 8: one activation stage per kernel column
    (64, 32, 3, 1, 1, 2, 24, 24),     # the same with one 32-code step per tap, tiles of several output rows
    (100, 64, 3, 1, 1, 2, 40, 56),    # the same, ragged last row block, non-square image
    (64, 16, 7, 2, 3, 2, 32, 32),     # first-layer shape: 7x7 stride 2 pad 3 (3 input channels stored as 16, the rest zero)
    (256, 64, 1, 1, 0, 2, 14, 14),    # bottleneck 1x1 expansions and reductions (ResNet-50 style)
    (64, 256, 1, 1, 0, 2, 14, 14),
    (32, 32, 3, 1, 1, 2, 16, 16),     # depthwise-separable networks' pointwise/3x3 sizes with few channels
]


@pytest.mark.parametrize("variant", VARIANTS, ids=lambda v: VNAME[v])
@pytest.mark.parametrize("M,Cin,k,stride,pad,B,H,W", CONV_CASES)
def test_conv_layer(M, Cin, k, stride, pad, B, H, W, variant):
    g = synth.rng(75, M + Cin + H)
    Wt = synth.weights_kaiming(g, M, Cin, k, k)
    scheme, bits = O.assign_rows(Wt, (60, 35, 5))
    alpha = synth.alpha_rows(Wt)
    x = synth.act_halfnormal(g, (B, H, W, Cin))
    codes, act_step = O.quantize_act(x, synth.ALPHA_ACT, O.ACT_U4)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    try:
        y, acc = Hn.conv(layer, d_packed, codes, stride, pad, act_step, variant)
    except R.RmsmpError as e:
        if e.status == R.ERR_VARIANT and variant in (R.VARIANT_TENSOR, Hn.WORKSPACE) and Cin % 16 != 0:
            pytest.skip("tensor variant needs Cin % 16 == 0")
        raise
    v_ref, ws, acc_ref, y_ref = O.layer_conv(Wt, scheme, bits, alpha, codes, act_step, stride, pad)
    acc_ref = acc_ref.reshape(-1, M)
    _check_layer_outputs(y, acc, acc_ref, ws, act_step, alpha, scheme, bits)


def test_conv_mn_layout_auto():
    M, Cin, B, H = 72, 32, 2, 10
    g = synth.rng(76)
    Wt = synth.weights_kaiming(g, M, Cin, 3, 3)
    scheme, bits = O.assign_rows(Wt, (60, 35, 5))
    alpha = synth.alpha_rows(Wt)
    codes = synth.act_codes_uniform(g, (B, H, H, Cin))
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    y, acc = Hn.conv(layer, d_packed, codes, 1, 1, 0.2, R.VARIANT_AUTO, out_layout=R.OUT_MN)
    _, ws, acc_ref, _ = O.layer_conv(Wt, scheme, bits, alpha, codes, np.float32(0.2), 1, 1)
    _check_layer_outputs(y, acc, acc_ref.reshape(-1, M), ws, np.float32(0.2), alpha, scheme, bits)


# ------------------------------------------------------------------ the whole path, one call after the other

def test_full_path_fp32_in_fp32_out():
    """quantize_pack -> quantize_act -> conv, from fp32 tensors, as the benchmark runs it."""
    import torch
    L = synth.ConvShape("t", 96, 64, 3, 1, 1, 14)
    g = synth.rng(77)
    Wt = synth.weights_kaiming(g, L.M, L.Cin, 3, 3)
    x = synth.act_halfnormal(g, (4, 14, 14, 64))
    scheme, bits = R.rmsmp_assign_rows(Wt, synth.RATIO_RMSMP1)
    s2, b2 = O.assign_rows(Wt, synth.RATIO_RMSMP1)
    assert np.array_equal(scheme, s2) and np.array_equal(bits, b2)
    alpha = synth.alpha_rows(Wt)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    dx = torch.from_numpy(x).cuda()
    dc = torch.empty(x.shape, dtype=torch.int8, device="cuda")
    step = R.rmsmp_quantize_act(dx, dx.numel(), synth.ALPHA_ACT, R.ACT_U4, dc)
    N = 4 * 14 * 14
    y = torch.empty((N, L.M), dtype=torch.float32, device="cuda")
    R.rmsmp_conv_implicit(layer, d_packed, dc, 4, 14, 14, 1, 1, step, y)
    torch.cuda.synchronize()
    codes, st_ref = O.quantize_act(x, synth.ALPHA_ACT, O.ACT_U4)
    assert np.float32(step) == st_ref
    _, _, _, y_ref = O.layer_conv(Wt, scheme, bits, alpha, codes, st_ref, 1, 1)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), y_ref.reshape(N, L.M).view(np.uint32))


# ------------------------------------------------------------------ re-quantizing epilogue (layer chaining)
# The fused epilogue must give the codes of (this layer's fp32 output -> the activation quantizer),
# i.e. the oracle's layer followed by the oracle's quantizer, byte for byte.

def _next_alpha(y_ref):
    return float(np.float32(3.0 * float(np.std(y_ref))))


@pytest.mark.parametrize("kind", [R.ACT_U4, R.ACT_S4])
@pytest.mark.parametrize("M,K,N,ld_extra", [
    (256, 512, 300, 0),      # bulk stores, ragged last tile
    (200, 128, 77, 0),       # ld_codes = 200: not a multiple of 16 -> direct byte stores
    (130, 96, 513, 14),      # padded leading dimension (144), two row blocks, ragged rows
    (64, 576, 260, 0),       # duplicated rows, resident weights
])
def test_linear_requant_epilogue(M, K, N, ld_extra, kind):
    import torch
    g = synth.rng(81, M + K + N)
    Wt = synth.weights_normal(g, (M, K))
    codes = synth.act_codes_uniform(g, (N, K))
    act_step = np.float32(0.125)
    scheme, bits = O.assign_rows(Wt, (60, 35, 5))
    alpha = synth.alpha_rows(Wt)
    _, _, _, y_ref = O.layer_linear(Wt, scheme, bits, alpha, codes, act_step)
    na = _next_alpha(y_ref)
    want, want_step = O.quantize_act(y_ref.reshape(N, M), na, kind)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    ws = torch.empty(R.rmsmp_workspace_bytes(layer), dtype=torch.int8, device="cuda")
    R.rmsmp_expand_weights(layer, d_packed, ws)
    ld = M + ld_extra
    out = torch.full((N, ld), 99, dtype=torch.int8, device="cuda")
    step = R.rmsmp_gemm_workspace_requant(layer, d_packed, ws, torch.from_numpy(codes).cuda(), N, K, float(act_step),
                                          na, kind, out, ld)
    torch.cuda.synchronize()
    assert R.rmsmp_last_device_status(d_packed) == R.OK
    got = out.cpu().numpy()
    assert np.float32(step) == want_step
    assert np.array_equal(got[:, :M], want)
    assert (got[:, M:] == 99).all()                      # padding columns untouched


@pytest.mark.parametrize("kind", [R.ACT_U4, R.ACT_S4])
@pytest.mark.parametrize("M,Cin,k,stride,pad,B,H,W", [
    (64, 64, 3, 1, 1, 2, 14, 14),
    (140, 256, 3, 1, 1, 5, 7, 7),      # several images per tile, ragged last tile, two row blocks
    (32, 48, 3, 2, 1, 2, 9, 12),
    (128, 64, 1, 2, 0, 2, 8, 8),
])
def test_conv_requant_epilogue(M, Cin, k, stride, pad, B, H, W, kind):
    import torch
    g = synth.rng(82, M + Cin + H)
    Wt = synth.weights_kaiming(g, M, Cin, k, k)
    scheme, bits = O.assign_rows(Wt, (60, 35, 5))
    alpha = synth.alpha_rows(Wt)
    x = synth.act_halfnormal(g, (B, H, W, Cin))
    codes, act_step = O.quantize_act(x, synth.ALPHA_ACT, O.ACT_U4)
    _, _, _, y_ref = O.layer_conv(Wt, scheme, bits, alpha, codes, act_step, stride, pad)
    y_ref = y_ref.reshape(-1, M)
    na = _next_alpha(y_ref)
    want, want_step = O.quantize_act(y_ref, na, kind)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    ws = torch.empty(R.rmsmp_workspace_bytes(layer), dtype=torch.int8, device="cuda")
    R.rmsmp_expand_weights(layer, d_packed, ws)
    out = torch.full(y_ref.shape, 99, dtype=torch.int8, device="cuda")
    step = R.rmsmp_conv_implicit_workspace_requant(layer, d_packed, ws, torch.from_numpy(codes).cuda(), B, H, W,
                                                   stride, pad, float(act_step), na, kind, out)
    torch.cuda.synchronize()
    assert R.rmsmp_last_device_status(d_packed) == R.OK
    assert np.float32(step) == want_step
    assert np.array_equal(out.cpu().numpy(), want)


def _ulps(x, n):
    """fp32 value n units in the last place away from x."""
    v = np.float32(x)
    for _ in range(abs(n)):
        v = np.nextafter(v, np.float32(np.inf if n > 0 else -np.inf), dtype=np.float32)
    return v


@pytest.mark.parametrize("kind", [R.ACT_U4, R.ACT_S4])
@pytest.mark.parametrize("M,ld_extra", [(128, 0), (130, 14), (64, 0)], ids=["bulk", "direct", "dup"])
@pytest.mark.parametrize("step_ulps", [0, 1, -1, 4, -4])
def test_requant_epilogue_on_rounding_boundaries(M, ld_extra, step_ulps, kind):
    """The fused quantizer exactly ON, and a few units in the last place either side of, its
    rounding boundaries.  All rows are Fixed-8 with alpha = 127, so wstep = 1 and the weights are
    the integers they are given as; with act_step = 1 the layer output y equals the integer sum.
    next_alpha is chosen so that y / next_alpha * Q = y / 2: every odd sum lies exactly on a
    half-level (the tie goes to the even code), and an act_step a few ulps off 1 moves every value
    just off its level or half-level.  Expected codes: the oracle's epilogue followed by the
    oracle's quantizer, so its chain of fp32 roundings decides."""
    import torch
    K, N = 64, 700
    g = synth.rng(83, M + step_ulps + 10 * kind)
    lo = 0 if kind == R.ACT_U4 else -1
    Wt = g.integers(lo, 2, size=(M, K)).astype(np.float32)          # values in {0, 1} (U4) or {-1, 0, 1} (S4)
    Wt[g.random((M, K)) < (0.93 if kind == R.ACT_U4 else 0.8)] = 0.0  # sums of a few codes: mostly inside the clip range
    Wt[:, 0] = 127.0                                                  # one full-scale entry per row keeps the values exact ...
    scheme = np.ones(M, np.uint8)
    bits = np.full(M, 8, np.uint8)
    alpha = np.full(M, 127.0, np.float32)
    codes = synth.act_codes_uniform(g, (N, K))
    codes[:, 0] = 0                                                   # ... and never contributes to a sum
    if kind == R.ACT_S4:
        codes = (codes % 15 - 7).astype(np.int8)
        codes[:, 0] = 0
    act_step = _ulps(1.0, step_ulps)
    na = 30.0 if kind == R.ACT_U4 else 14.0
    values, wstep, acc_ref, y_ref = O.layer_linear(Wt, scheme, bits, alpha, codes, act_step)
    assert np.all(wstep == np.float32(1.0)) and np.array_equal(values, Wt.astype(np.int8))
    odd = (np.abs(acc_ref) % 2 == 1) & (np.abs(acc_ref) < 30)
    assert odd.mean() > 0.25                                           # a large share of outputs sits on a half-level
    want, _ = O.quantize_act(y_ref, na, kind)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    ws = torch.empty(R.rmsmp_workspace_bytes(layer), dtype=torch.int8, device="cuda")
    R.rmsmp_expand_weights(layer, d_packed, ws)
    ld = M + ld_extra
    out = torch.full((N, ld), 99, dtype=torch.int8, device="cuda")
    R.rmsmp_gemm_workspace_requant(layer, d_packed, ws, torch.from_numpy(codes).cuda(), N, K, float(act_step),
                                   na, kind, out, ld)
    torch.cuda.synchronize()
    assert R.rmsmp_last_device_status(d_packed) == R.OK
    got = out.cpu().numpy()
    assert np.array_equal(got[:, :M], want)
    assert (got[:, M:] == 99).all()
    if step_ulps == 0:
        # with exact halves the expected code is the even neighbour, by the definition alone
        q = 15 if kind == R.ACT_U4 else 7
        t = np.clip(acc_ref.astype(np.float64) / na, 0.0 if kind == R.ACT_U4 else -1.0, 1.0) * q
        assert np.array_equal(want, np.rint(t).astype(np.int8))


def test_conv_requant_epilogue_on_rounding_boundaries():
    """The same construction through the convolution kernel's resident-weight form (3x3, 64 channels)."""
    import torch
    M, Cin, k, B, H = 64, 64, 3, 2, 12
    g = synth.rng(83, 999)
    Wt = g.integers(0, 2, size=(M, Cin, k, k)).astype(np.float32)
    Wt[g.random(Wt.shape) < 0.992] = 0.0
    Wt[:, 0, 0, 0] = 127.0
    scheme = np.ones(M, np.uint8)
    bits = np.full(M, 8, np.uint8)
    alpha = np.full(M, 127.0, np.float32)
    codes = synth.act_codes_uniform(g, (B, H, H, Cin))
    codes[..., 0] = 0
    for ulps in (0, 2, -2):
        act_step = _ulps(1.0, ulps)
        _, _, acc_ref, y_ref = O.layer_conv(Wt, scheme, bits, alpha, codes, act_step, 1, 1)
        assert ((acc_ref % 2 == 1) & (acc_ref < 30)).mean() > 0.2
        want, _ = O.quantize_act(y_ref.reshape(-1, M), 30.0, O.ACT_U4)
        layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
        ws = torch.empty(R.rmsmp_workspace_bytes(layer), dtype=torch.int8, device="cuda")
        R.rmsmp_expand_weights(layer, d_packed, ws)
        out = torch.full(want.shape, 99, dtype=torch.int8, device="cuda")
        R.rmsmp_conv_implicit_workspace_requant(layer, d_packed, ws, torch.from_numpy(codes).cuda(), B, H, H, 1, 1,
                                                float(act_step), 30.0, R.ACT_U4, out)
        torch.cuda.synchronize()
        assert R.rmsmp_last_device_status(d_packed) == R.OK
        assert np.array_equal(out.cpu().numpy(), want)


def test_requant_rejects_bad_arguments():
    import torch
    g = synth.rng(83)
    Wt = synth.weights_normal(g, (32, 64))
    scheme, bits = O.assign_rows(Wt, (60, 35, 5))
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, synth.alpha_rows(Wt))
    ws = torch.empty(R.rmsmp_workspace_bytes(layer), dtype=torch.int8, device="cuda")
    R.rmsmp_expand_weights(layer, d_packed, ws)
    act = torch.zeros((40, 64), dtype=torch.int8, device="cuda")
    out = torch.zeros((40, 32), dtype=torch.int8, device="cuda")
    for bad_alpha in (0.0, -1.0, float("inf"), float("nan")):
        with pytest.raises(R.RmsmpError) as e:
            R.rmsmp_gemm_workspace_requant(layer, d_packed, ws, act, 40, 64, 0.1, bad_alpha, R.ACT_U4, out, 32)
        assert e.value.status == R.ERR_SCALE
    with pytest.raises(R.RmsmpError) as e:
        R.rmsmp_gemm_workspace_requant(layer, d_packed, ws, act, 40, 64, 0.1, 1.0, 7, out, 32)
    assert e.value.status == R.ERR_SCHEME
    with pytest.raises(R.RmsmpError) as e:
        R.rmsmp_gemm_workspace_requant(layer, d_packed, ws, act, 40, 64, 0.1, 1.0, R.ACT_U4, out, 16)   # ld < M
    assert e.value.status == R.ERR_SHAPE


def test_padded_output_rows_leave_the_padding_untouched():
    """[N][ld_out] fp32 output with ld_out > M and M not a multiple of 4: bulk stores clip in
    16-byte granules, so this shape must not go through them."""
    import torch
    M, K, N, ld = 130, 128, 300, 136
    g = synth.rng(84)
    Wt = synth.weights_normal(g, (M, K))
    codes = synth.act_codes_uniform(g, (N, K))
    scheme, bits = O.assign_rows(Wt, (60, 35, 5))
    alpha = synth.alpha_rows(Wt)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    ws = torch.empty(R.rmsmp_workspace_bytes(layer), dtype=torch.int8, device="cuda")
    R.rmsmp_expand_weights(layer, d_packed, ws)
    d_codes = torch.from_numpy(codes).cuda()
    _, _, _, y_ref = O.layer_linear(Wt, scheme, bits, alpha, codes, np.float32(0.25))
    for fn in (lambda y: R.rmsmp_gemm_workspace(layer, d_packed, ws, d_codes, N, K, 0.25, y, ld),
               lambda y: R.rmsmp_gemm(layer, d_packed, d_codes, N, K, 0.25, y, ld)):
        y = torch.full((N, ld), -7.0, dtype=torch.float32, device="cuda")
        fn(y)
        torch.cuda.synchronize()
        got = y.cpu().numpy()
        assert np.array_equal(got[:, :M].view(np.uint32), y_ref.reshape(N, M).view(np.uint32))
        assert (got[:, M:] == -7.0).all()


def test_a_bounded_wait_that_runs_out_reports_timeout_and_leaves_the_context_usable():
    """The failure path, without a fault: one warp waits on a barrier nobody signals, with the
    kernels' own bounded wait and a limit of about a millisecond.  The status word must read
    ERR_TIMEOUT afterwards, and an ordinary layer on the same stream must still be bit-exact."""
    import torch
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    R.rmsmp_selftest_bounded_wait(2_000_000, status)
    torch.cuda.synchronize()
    assert int(status[0].item()) == R.ERR_TIMEOUT
    with pytest.raises(R.RmsmpError) as e:
        R.rmsmp_selftest_bounded_wait(10 ** 10, status)          # beyond the tenth of a second the call allows
    assert e.value.status == R.ERR_SHAPE
    g = synth.rng(84, 1)
    Wt = synth.weights_normal(g, (256, 512))
    scheme, bits = O.assign_rows(Wt, (60, 35, 5))
    alpha = synth.alpha_rows(Wt)
    act = synth.act_codes_uniform(g, (300, 512))
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    y, acc = Hn.gemm(layer, d_packed, act, 0.25, R.VARIANT_TENSOR)
    _, _, acc_ref, y_ref = O.layer_linear(Wt, scheme, bits, alpha, act, np.float32(0.25))
    assert np.array_equal(acc, acc_ref)
    assert np.array_equal(y.view(np.uint32), y_ref.view(np.uint32))


# ------------------------------------------------------------------ narrow tiles, the reduction shared by a cluster

@pytest.mark.parametrize("variant", [R.VARIANT_TENSOR, Hn.WORKSPACE], ids=lambda v: VNAME[v])
@pytest.mark.parametrize("M,K,N", [
    (128, 128, 16),          # one k-block, one tile, nothing to share
    (130, 272, 33),          # a second row block of two rows, a last step of 16 codes
    (64, 1040, 17),          # 64-byte k-blocks
    (512, 2304, 49),         # eight CTAs to a tile, k-blocks shared unevenly
    (300, 4096, 100),        # more k-blocks than stages
    (4096, 512, 40),         # many row blocks
    (256, 6144, 128),
])
def test_small_linear_layers_share_their_reduction(M, K, N, variant):
    """Sums are integers and the output is one multiply: exact, in both layouts, with and without the sums."""
    g = synth.rng(88, M + K + N)
    Wt = synth.weights_normal(g, (M, K))
    scheme, bits = _mixed_map(M, 5, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    act = g.integers(-16, 17, size=(N, K)).astype(np.int8)
    _, ws, acc_ref, _ = O.layer_linear(Wt, scheme, bits, alpha, act, np.float32(0.25))
    for layout in (R.OUT_NM, R.OUT_MN):
        for want_acc in (True, False):
            y, acc = Hn.gemm(layer, d_packed, act, 0.25, variant, out_layout=layout, want_acc=want_acc)
            if want_acc:
                _check_layer_outputs(y, acc, acc_ref, ws, np.float32(0.25), alpha, scheme, bits)
            assert np.array_equal(y.view(np.uint32), O.epilogue(acc_ref, ws, np.float32(0.25)).view(np.uint32))


@pytest.mark.parametrize("workspace", [False, True])
@pytest.mark.parametrize("M,K,N", [
    (33, 64, 1), (130, 192, 37), (1088, 64, 515),      # rows and pixels beyond the last group, rows of no multiple of 16 bytes
    (96, 2048, 67), (257, 1008, 129),                  # a reduction shared by a cluster
    (130, 1024, 9001), (40, 160, 38001),               # more tiles than SMs
])
def test_outputs_by_row_of_any_length(M, K, N, workspace):
    """[row][pixel] outputs, turned in shared memory: exact, with and without the sums, nothing beyond the matrix."""
    import torch
    g = synth.rng(95, M + K + N)
    Wt = synth.weights_normal(g, (M, K))
    scheme, bits = _mixed_map(M, 5, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    act = g.integers(-16, 17, size=(N, K)).astype(np.int8)
    _, ws, acc_ref, _ = O.layer_linear(Wt, scheme, bits, alpha, act, np.float32(0.25))
    y_ref = np.ascontiguousarray(O.epilogue(acc_ref, ws, np.float32(0.25)).T)
    ld = (K + 15) // 16 * 16
    a = torch.zeros((N, ld), dtype=torch.int8, device="cuda")
    a[:, :K] = torch.from_numpy(act).cuda()
    if workspace:
        d_ws = torch.empty(R.rmsmp_workspace_bytes(layer), dtype=torch.int8, device="cuda")
        R.rmsmp_expand_weights(layer, d_packed, d_ws)
    for want_acc in (True, False):
        y = torch.full((M * N + 64,), -7.0, dtype=torch.float32, device="cuda")
        acc = torch.full((M * N + 64,), -9, dtype=torch.int32, device="cuda") if want_acc else None
        if workspace:
            R.rmsmp_gemm_workspace(layer, d_packed, d_ws, a, N, ld, 0.25, y, N, R.OUT_MN, acc)
        else:
            R.rmsmp_gemm(layer, d_packed, a, N, ld, 0.25, y, N, R.OUT_MN, acc)
        out = y.cpu().numpy()
        assert np.array_equal(out[:M * N].view(np.uint32), y_ref.ravel().view(np.uint32)) and (out[M * N:] == -7.0).all()
        if want_acc:
            out = acc.cpu().numpy()
            assert np.array_equal(out[:M * N], acc_ref.T.ravel()) and (out[M * N:] == -9).all()


@pytest.mark.parametrize("N", [1, 2, 31, 33, 300])
@pytest.mark.parametrize("M,K", [(96, 1), (130, 17), (200, 127), (64, 200), (1000, 513), (20000, 72)])
def test_linear_layers_of_any_length_under_auto(M, K, N):
    """K that is no multiple of 16, from one token up, with other bytes behind every row: exact as always."""
    g = synth.rng(90, M + K + N)
    Wt = synth.weights_normal(g, (M, K))
    scheme, bits = _mixed_map(M, 7, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    act = g.integers(-128, 128, size=(N, K)).astype(np.int8)
    ld = (K + 15) // 16 * 16 + 16
    import torch
    a = torch.full((N, ld), 55, dtype=torch.int8, device="cuda")
    a[:, :K] = torch.from_numpy(act).cuda()
    y = torch.full((N, M), float("nan"), dtype=torch.float32, device="cuda")
    acc = torch.full((N, M), -9, dtype=torch.int32, device="cuda")
    R.rmsmp_gemm(layer, d_packed, a, N, ld, 0.25, y, M, R.OUT_NM, acc)
    _, ws, acc_ref, _ = O.layer_linear(Wt, scheme, bits, alpha, act, np.float32(0.25))
    _check_layer_outputs(y.cpu().numpy(), acc.cpu().numpy(), acc_ref, ws, np.float32(0.25), alpha, scheme, bits)
    assert R.rmsmp_last_device_status(d_packed) == R.OK


@pytest.mark.parametrize("variant", [R.VARIANT_TENSOR, Hn.WORKSPACE], ids=lambda v: VNAME[v])
@pytest.mark.parametrize("M,Cin,k,stride,pad,B,H,W", [
    (64, 64, 3, 1, 1, 1, 30, 28),        # tiles of a few rows, the last tile of an image shorter than the others
    (256, 256, 3, 1, 1, 1, 14, 14),
    (512, 512, 3, 1, 1, 1, 7, 7),        # a tile is an image
    (130, 96, 3, 2, 1, 3, 15, 13),       # stride 2, odd sizes, several images
    (96, 48, 5, 1, 2, 2, 9, 20),
    (160, 320, 1, 2, 0, 5, 9, 9),
    (32, 16, 3, 3, 1, 2, 11, 10),        # stride 3
])
def test_small_convolutions_share_their_reduction(M, Cin, k, stride, pad, B, H, W, variant):
    import torch
    g = synth.rng(89, M + Cin + H)
    Wt = synth.weights_kaiming(g, M, Cin, k, k)
    scheme, bits = _mixed_map(M, 6, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    act = g.integers(-16, 17, size=(B, H, W, Cin)).astype(np.int8)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    _, ws, acc_ref, y_ref = O.layer_conv(Wt, scheme, bits, alpha, act, np.float32(0.25), stride, pad)
    y, acc = Hn.conv(layer, d_packed, act, stride, pad, 0.25, variant)
    assert np.array_equal(acc.reshape(-1, M), acc_ref.reshape(-1, M))
    assert np.array_equal(y.reshape(-1, M).view(np.uint32), y_ref.reshape(-1, M).view(np.uint32))
    if variant == Hn.WORKSPACE:
        d_ws = Hn._workspace(layer, d_packed)
        d_act = torch.from_numpy(act).cuda()
        out = torch.full((acc_ref.size // M, M), 99, dtype=torch.int8, device="cuda")
        for kind in (R.ACT_U4, R.ACT_S4):
            R.rmsmp_conv_implicit_workspace_requant(layer, d_packed, d_ws, d_act, B, H, W, stride, pad, 0.25, 1.7, kind, out)
            c_ref, _ = O.quantize_act(y_ref.reshape(-1, M), 1.7, kind)
            assert np.array_equal(out.cpu().numpy(), c_ref)


@pytest.mark.parametrize("M,Cin,k,stride,pad,B,H,W", [
    (144, 24, 1, 1, 0, 3, 17, 19),       # 8-byte loads, more pixels than a tile, the last tile ragged
    (40, 20, 3, 1, 1, 2, 9, 7),          # 4-byte loads
    (33, 3, 7, 2, 3, 2, 21, 15),         # single bytes; 49 taps of one step
    (130, 5, 3, 2, 1, 1, 8, 300),        # rows wider than any copy box, two row blocks
    (16, 72, 3, 3, 0, 2, 11, 10),        # a last step of eight codes
    (64, 200, 5, 1, 2, 1, 6, 6),         # more k-blocks than stages
    (8, 1, 1, 1, 0, 1, 1, 1),            # one code
    (24, 9, 2, 1, 1, 5, 3, 3),
])
def test_convolutions_of_any_channel_count_under_auto(M, Cin, k, stride, pad, B, H, W):
    """Channel counts that the copy engine cannot address, any int8 code: exact, both layouts."""
    g = synth.rng(93, M + Cin + H)
    Wt = synth.weights_kaiming(g, M, Cin, k, k)
    scheme, bits = _mixed_map(M, 8, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    act = g.integers(-128, 128, size=(B, H, W, Cin)).astype(np.int8)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    _, ws, acc_ref, y_ref = O.layer_conv(Wt, scheme, bits, alpha, act, np.float32(0.25), stride, pad)
    for layout in (R.OUT_NM, R.OUT_MN):
        for want_acc in (True, False):
            y, acc = Hn.conv(layer, d_packed, act, stride, pad, 0.25, R.VARIANT_AUTO, layout, want_acc)
            if want_acc:
                assert np.array_equal(acc, acc_ref.reshape(-1, M))
            assert np.array_equal(np.ascontiguousarray(y).view(np.uint32), y_ref.reshape(-1, M).view(np.uint32))


# ------------------------------------------------------------------ choice of tiles and kernels: neighbours cost about the same

def _call_us(M, Cin, k, pad, B, H, W, layout):
    """GPU time of one call on a workspace (a linear layer where k is 0: B tokens), and its exact sums' check."""
    import torch
    g = synth.rng(91, M + Cin + B)
    kk = max(k, 1)
    Wt = synth.weights_kaiming(g, M, Cin, kk, kk)
    scheme, bits = _mixed_map(M, 9)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, synth.alpha_rows(Wt))
    ws = Hn._workspace(layer, d_packed)
    N = B if k == 0 else B * (H + 2 * pad - k + 1) * (W + 2 * pad - k + 1)
    act = torch.randint(0, 16, (B, H, W, Cin) if k else (N, Cin), dtype=torch.int8, device="cuda")
    y = torch.empty((N, M) if layout == R.OUT_NM else (M, N), dtype=torch.float32, device="cuda")

    def call():
        if k:
            R.rmsmp_conv_implicit_workspace(layer, d_packed, ws, act, B, H, W, 1, pad, 0.5, y, layout)
        else:
            R.rmsmp_gemm_workspace(layer, d_packed, ws, act, N, Cin, 0.5, y, y.shape[1], layout)

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        call()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for _ in range(10):
                call()
        runs = []
        for _ in range(8):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record(stream)
            graph.replay()
            end.record(stream)
            torch.cuda.synchronize()
            runs.append(100.0 * start.elapsed_time(end))
    assert R.rmsmp_last_device_status(d_packed) == R.OK
    # the call against the kernel that shares no code with it
    ref = torch.empty_like(y)
    if k:
        R.rmsmp_conv_implicit_variant(layer, d_packed, act, B, H, W, 1, pad, 0.5, ref, layout, None, R.VARIANT_SIMPLE)
    else:
        R.rmsmp_gemm_variant(layer, d_packed, act, N, Cin, 0.5, ref, ref.shape[1], layout, None, R.VARIANT_SIMPLE)
    assert torch.equal(y.view(torch.int32), ref.view(torch.int32))
    return min(runs)


def test_patch_matrix_of_wide_rows_in_proportion():
    """720 rows of 1280 pixels against 448 of 640 (three and a fifth times the work): 34 us and 11 for two images and
    one; 105 when rows that wide went to the other kernel."""
    import torch

    def us(H, W):
        Ho, Wo = (H - 1) // 2 + 1, (W - 1) // 2 + 1
        act = torch.randint(0, 16, (2, H, W, 3), dtype=torch.int8, device="cuda")
        cols = torch.empty((2 * Ho * Wo, 160), dtype=torch.int8, device="cuda")
        runs = []
        for _ in range(8):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            start.record()
            for _ in range(10):
                R.rmsmp_im2col_codes(act, 2, H, W, 3, 3, 7, 7, 2, 3, cols, 160)
            end.record()
            torch.cuda.synchronize()
            runs.append(100.0 * start.elapsed_time(end))
        return min(runs)

    assert us(720, 1280) <= 6.0 * us(448, 640)


@pytest.mark.parametrize("call,other,bound", [
    # 256 rows, 20,000 tokens as [M][N] against [N][M]: 7.6 us and 6.8; tiles no multiple of 32 tokens 16.5
    ((256, 64, 0, 0, 20000, 1, 1, R.OUT_MN), (256, 64, 0, 0, 20000, 1, 1, R.OUT_NM), 1.7),
    # ten rows against 64: 24 us and 17; 28 with narrow tiles
    ((10, 4096, 0, 0, 20000, 1, 1, R.OUT_NM), (64, 4096, 0, 0, 20000, 1, 1, R.OUT_NM), 1.56),
    # two images of 49 x 49 against eight: 6.0 us and 8.3; 8.3 with tiles of five rows
    ((64, 32, 3, 1, 2, 49, 49, R.OUT_NM), (64, 32, 3, 1, 8, 49, 49, R.OUT_NM), 0.87),
    # 192 rows against 256: 46 us and 53; 56 with resident weights
    ((192, 512, 0, 0, 200000, 1, 1, R.OUT_NM), (256, 512, 0, 0, 200000, 1, 1, R.OUT_NM), 0.97),
    # 4880 tokens against 4864 and 1872 rows against 1920: 11.7 us and 10.2; 14.4 with three rounds of tiles
    ((1872, 160, 0, 0, 4880, 1, 1, R.OUT_MN), (1920, 160, 0, 0, 4864, 1, 1, R.OUT_MN), 1.28),
    # 17 images against 16: 10.9 us and 10; 17.6 with more clusters than the chip places at once
    ((48, 368, 3, 1, 17, 15, 11, R.OUT_NM), (48, 368, 3, 1, 16, 15, 11, R.OUT_NM), 1.35),
    # eight tokens as [M][N] against [N][M]: 3.3 us and 3.9; 5.5 on the persistent kernel
    ((64, 64, 0, 0, 8, 1, 1, R.OUT_MN), (64, 64, 0, 0, 8, 1, 1, R.OUT_NM), 1.15),
])
def test_neighbouring_problems_cost_about_the_same(call, other, bound):
    """(M, Cin, k, pad, B, H, W, layout): a rule that picks tiles or a kernel badly for one of two like problems shows in their
    times.  Each bound lies halfway between what the rule gives and what it gave when it was wrong (in the comments)."""
    assert _call_us(*call) <= bound * _call_us(*other)


# ------------------------------------------------------------------ row assignment on the device

@pytest.mark.parametrize("ratio", [(60, 35, 5), (65, 30, 5), (0, 100, 0), (50, 40, 10)], ids=lambda r: "%d-%d-%d" % r)
@pytest.mark.parametrize("shape", [(256, 512), (130, 96), (1000, 2304), (64, 64, 3, 3), (160, 48, 3, 3)], ids=str)
def test_assignment_on_the_device_matches_oracle(shape, ratio):
    """Ratio in, packed layer out: the assignment (variance rank), the grouping, the per-row steps and every
    code must equal the oracle's assign_rows -> quantize_rows -> group_rows; then the layer runs."""
    import torch
    g = synth.rng(85, sum(shape) + ratio[0])
    conv = len(shape) == 4
    Wt = synth.weights_kaiming(g, *shape) if conv else synth.weights_normal(g, shape)
    if not conv:
        Wt[7] = Wt[3]                                   # two rows of equal variance: the row index decides
    M = shape[0]
    Cin, kh, kw = (shape[1], shape[2], shape[3]) if conv else (shape[1], 1, 1)
    layer = R.rmsmp_layer_init_ratio(M, Cin, kh, kw, ratio)
    d_W = torch.from_numpy(Wt).cuda()
    d_packed = torch.empty(layer.packed_bytes, dtype=torch.uint8, device="cuda")
    scratch = torch.empty(R.rmsmp_assign_scratch_bytes(M), dtype=torch.uint8, device="cuda")
    d_scheme = torch.empty(M, dtype=torch.uint8, device="cuda")
    d_bits = torch.empty(M, dtype=torch.uint8, device="cuda")
    R.rmsmp_assign_quantize_pack(d_W, R.W_CONV_OIHW if conv else R.W_LINEAR, layer, ratio, None, R.POT_NEAREST, d_packed,
                                 scratch, d_scheme, d_bits)
    torch.cuda.synchronize()
    scheme, bits = O.assign_rows(Wt, ratio)
    assert np.array_equal(d_scheme.cpu().numpy(), scheme) and np.array_equal(d_bits.cpu().numpy(), bits)
    alpha = synth.alpha_rows(Wt)
    v_ref, ws_ref = O.quantize_rows(Wt.reshape(M, -1), scheme, bits, alpha)
    vals, perm, ws = Hn.unpack(layer, d_packed)
    assert np.array_equal(perm, O.group_rows(scheme, bits))
    assert np.array_equal(ws.view(np.uint32), ws_ref.view(np.uint32))
    assert np.array_equal(vals, v_ref)
    # the same descriptor as the host route gives, and a layer run on top of it
    ref_layer = R.rmsmp_layer_init(M, Cin, kh, kw, scheme, bits)
    assert (layer.nP, layer.nF4, layer.n8, layer.packed_bytes) == (ref_layer.nP, ref_layer.nF4, ref_layer.n8, ref_layer.packed_bytes)
    if not conv:
        act = synth.act_codes_uniform(g, (77, shape[1]))
        for variant in (R.VARIANT_AUTO, R.VARIANT_TENSOR if shape[1] % 16 == 0 else R.VARIANT_SIMT, Hn.WORKSPACE if shape[1] % 16 == 0 else R.VARIANT_SIMT):
            y, acc = Hn.gemm(layer, d_packed, act, 0.05, variant)
            assert np.array_equal(acc, O.matmul(v_ref, act))


def _rows_at_the_cuts(name, g, M, K):
    """Weights whose ranking the parallel variances cannot decide by themselves, or only just."""
    W = synth.weights_normal(g, (M, K))
    if name == "copies":                                # four different rows, each many times: ties at both cuts
        W = W[g.integers(0, min(4, M), size=M)]
    elif name == "all_equal":
        W[:] = W[0]
    elif name == "constant":                            # true variance zero, the definition's is rounding noise
        W[:] = g.uniform(0.1, 0.9, size=(M, 1)).astype(np.float32)
    elif name == "zero_rows":                           # pruned rows, more than fit in front of the first cut
        W[g.permutation(M)[: M * 7 // 10]] = 0.0
    elif name == "offset":                              # mean 2^12 times the spread: the parallel sums cancel
        W += np.float32(80.0)
    elif name == "permuted":                            # the same weights in another order: sums differ in the last bits only
        for r in range(1, M):
            W[r] = W[0][g.permutation(K)]
    elif name == "huge":                                # squares far beyond fp32, rows of several magnitudes
        W *= np.exp2(g.integers(80, 120, size=(M, 1))).astype(np.float32)
    elif name == "tiny":                                # squares below fp32's smallest number
        W *= np.exp2(-g.integers(80, 110, size=(M, 1))).astype(np.float32)
    return np.ascontiguousarray(W)


@pytest.mark.parametrize("name", ["normal", "copies", "all_equal", "constant", "zero_rows", "offset", "permuted", "huge", "tiny"])
@pytest.mark.parametrize("M,K,ratio", [(1, 5, (60, 35, 5)), (33, 31, (60, 35, 5)), (257, 100, (50, 40, 10)),
                                       (1024, 36, (60, 35, 5)), (1100, 36, (60, 35, 5)), (2500, 64, (65, 30, 5)),
                                       (4100, 20, (60, 35, 5)), (300, 64, (95, 0, 5)), (128, 16, (0, 100, 0)),
                                       (2500, 27, (0, 40, 60)), (20000, 12, (60, 35, 5))])
def test_assignment_at_the_cuts_of_the_ranking(M, K, ratio, name):
    """Whole-number result (which row gets which scheme), so no tolerance: it is the oracle's for rows whose
    variances tie, or differ by less than the summation error, at a cut; fewer and more rows than threads, and more
    than the statistics in shared memory."""
    import torch
    Wt = _rows_at_the_cuts(name, synth.rng(86, M + K), M, K)
    layer = R.rmsmp_layer_init_ratio(M, K, 1, 1, ratio)
    d_packed = torch.empty(layer.packed_bytes, dtype=torch.uint8, device="cuda")
    scratch = torch.full((R.rmsmp_assign_scratch_bytes(M),), 0xA5, dtype=torch.uint8, device="cuda")
    d_scheme, d_bits = (torch.empty(M, dtype=torch.uint8, device="cuda") for _ in range(2))
    R.rmsmp_assign_quantize_pack(torch.from_numpy(Wt).cuda(), R.W_LINEAR, layer, ratio, None, R.POT_NEAREST, d_packed, scratch,
                                 d_scheme, d_bits)
    scheme, bits = O.assign_rows(Wt, ratio)
    assert np.array_equal(d_scheme.cpu().numpy(), scheme) and np.array_equal(d_bits.cpu().numpy(), bits)
    vals, perm, ws = Hn.unpack(layer, d_packed)
    assert np.array_equal(perm, O.group_rows(scheme, bits))
    # the metadata that the host route writes for this map: header, permutation, scales, kinds, block table
    ref_layer, ref = Hn.pack_layer(Wt, scheme, bits, synth.alpha_rows(Wt))
    for off, n in ((0, 68), (layer.off_perm, 4 * M), (layer.off_slot, 4 * M), (layer.off_wstep, 4 * M), (layer.off_alpha, 4 * M),
                   (layer.off_kind, M), (layer.off_blocks, 32 * layer.nblocks)):
        assert torch.equal(d_packed[off:off + n], ref[off:off + n])


@pytest.mark.parametrize("name", ["copies", "constant", "zero_rows"])
def test_assignment_of_many_tied_rows_takes_no_quadratic_time(name):
    """20,000 rows of which most tie at a cut: within fifteen times what rows take that do not (100 us against 15 to
    32 ms when every tied row was compared with every other)."""
    import torch
    M, K, ratio = 20000, 64, (60, 35, 5)
    layer = R.rmsmp_layer_init_ratio(M, K, 1, 1, ratio)
    d_packed = torch.empty(layer.packed_bytes, dtype=torch.uint8, device="cuda")
    scratch = torch.empty(R.rmsmp_assign_scratch_bytes(M), dtype=torch.uint8, device="cuda")
    times = {}
    for which in ("normal", name):
        d_W = torch.from_numpy(_rows_at_the_cuts(which, synth.rng(90, M), M, K)).cuda()
        runs = []
        for _ in range(4):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            R.rmsmp_assign_quantize_pack(d_W, R.W_LINEAR, layer, ratio, None, R.POT_NEAREST, d_packed, scratch)
            end.record()
            torch.cuda.synchronize()
            runs.append(start.elapsed_time(end))
        times[which] = min(runs)
    assert times[name] <= 15.0 * times["normal"], times


# ------------------------------------------------------------------ depthwise convolution

@pytest.mark.parametrize("C,k,stride,pad,B,H,W,kind", [
    (32, 3, 1, 1, 2, 14, 14, R.ACT_U4),
    (96, 3, 2, 1, 3, 15, 13, R.ACT_U4),        # MobileNet-v2 style stride-2 block, odd sizes
    (144, 3, 1, 1, 1, 28, 28, R.ACT_S4),
    (960, 3, 1, 1, 2, 7, 7, R.ACT_U4),         # the widest depthwise layer of MobileNet-v2
    (8, 5, 1, 2, 2, 6, 9, R.ACT_S4),
    (1280, 3, 1, 1, 1, 5, 6, R.ACT_S4),        # more channel quads than threads of a block
    (16, 3, 3, 0, 2, 11, 10, R.ACT_U4),        # a stride the run kernel does not take
])
def test_depthwise_conv_matches_oracle(C, k, stride, pad, B, H, W, kind):
    import torch
    g = synth.rng(86, C + k + H)
    Wt = synth.weights_kaiming(g, C, 1, k, k)
    scheme, bits = O.assign_rows(Wt, (60, 35, 5))
    alpha = synth.alpha_rows(Wt)
    x = synth.act_halfnormal(g, (B, H, W, C)) if kind == R.ACT_U4 else synth.act_normal(g, (B, H, W, C))
    codes, act_step = O.quantize_act(x, synth.ALPHA_ACT, kind)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    v_ref, wstep = O.quantize_rows(Wt.reshape(C, -1), scheme, bits, alpha)
    acc_ref = O.conv_depthwise(v_ref.reshape(C, k, k), codes, stride, pad)
    y_ref = O.epilogue(acc_ref, wstep, act_step)
    Ho, Wo = O.conv_out_hw(H, W, k, k, stride, pad)
    y = torch.full((B, Ho, Wo, C), float("nan"), dtype=torch.float32, device="cuda")
    acc = torch.full((B, Ho, Wo, C), -5, dtype=torch.int32, device="cuda")
    R.rmsmp_conv_depthwise(layer, d_packed, torch.from_numpy(codes).cuda(), B, H, W, stride, pad, float(act_step), y, acc)
    torch.cuda.synchronize()
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), y_ref.view(np.uint32))


@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("C,pad,B,H,W", [
    (4, 0, 1, 3, 3),                           # one output
    (4, 1, 1, 1, 1), (8, 2, 1, 1, 4),          # images smaller than the filter, outputs made of padding only
    (12, 1, 3, 19, 5), (20, 1, 1, 8, 10),      # columns left over in the last group of four
    (1028, 1, 1, 9, 6),                        # more channel quads than threads of a block
    (96, 1, 40, 9, 9),                         # strips of several heights
])
def test_depthwise_strips_on_the_whole_code_range(C, pad, B, H, W, stride):
    """Integer sums of any int8 activation code (not only the 4-bit ones), exact: no tolerance."""
    import torch
    g = synth.rng(87, C + H + W)
    Wt = synth.weights_kaiming(g, C, 1, 3, 3)
    scheme, bits = O.assign_rows(Wt, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    codes = g.integers(-128, 128, size=(B, H, W, C), dtype=np.int8)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    v_ref, wstep = O.quantize_rows(Wt.reshape(C, -1), scheme, bits, alpha)
    acc_ref = O.conv_depthwise(v_ref.reshape(C, 3, 3), codes, stride, pad)
    for with_acc in (True, False):
        y = torch.full(acc_ref.shape, float("nan"), dtype=torch.float32, device="cuda")
        acc = torch.full(acc_ref.shape, -5, dtype=torch.int32, device="cuda")
        R.rmsmp_conv_depthwise(layer, d_packed, torch.from_numpy(codes).cuda(), B, H, W, stride, pad, 0.5, y, acc if with_acc else None)
        torch.cuda.synchronize()
        if with_acc:
            assert np.array_equal(acc.cpu().numpy(), acc_ref)
        assert np.array_equal(y.cpu().numpy().view(np.uint32), O.epilogue(acc_ref, wstep, np.float32(0.5)).view(np.uint32))


@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("C,pad,B,H,W", [
    (32, 4, 1, 8, 8), (32, 4, 2, 8, 8),        # strips of one output row, the first of them above every input row
    (32, 5, 1, 14, 14), (64, 8, 2, 14, 14),
    (192, 6, 4, 28, 28),                       # strips of two rows
    (8, 16, 3, 1, 5), (4, 16, 2, 6, 1),        # the widest padding
])
def test_depthwise_strips_that_lie_in_the_padding(C, pad, B, H, W, stride):
    """Outputs without an input row under them are zero.  The activations are the middle of a buffer of non-zero codes,
    so that a row read from outside the image stays inside the buffer and shows in the sums."""
    import torch
    g = synth.rng(89, C + H + W + pad)
    Wt = synth.weights_kaiming(g, C, 1, 3, 3)
    scheme, bits = O.assign_rows(Wt, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    codes = g.integers(0, 16, size=(B, H, W, C), dtype=np.int8)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    v_ref, wstep = O.quantize_rows(Wt.reshape(C, -1), scheme, bits, alpha)
    acc_ref = O.conv_depthwise(v_ref.reshape(C, 3, 3), codes, stride, pad)
    margin = (pad + 4) * (W + 2 * pad) * C // 16 * 16
    buf = torch.full((margin + codes.size + margin,), 15, dtype=torch.int8, device="cuda")
    act = buf[margin:margin + codes.size]
    act.copy_(torch.from_numpy(codes).cuda().view(-1))
    for with_acc in (True, False):
        y = torch.full(acc_ref.shape, float("nan"), dtype=torch.float32, device="cuda")
        acc = torch.full(acc_ref.shape, -5, dtype=torch.int32, device="cuda")
        R.rmsmp_conv_depthwise(layer, d_packed, act, B, H, W, stride, pad, 0.5, y, acc if with_acc else None)
        torch.cuda.synchronize()
        if with_acc:
            assert np.array_equal(acc.cpu().numpy(), acc_ref)
        assert np.array_equal(y.cpu().numpy().view(np.uint32), O.epilogue(acc_ref, wstep, np.float32(0.5)).view(np.uint32))


def test_depthwise_conv_rejects_what_it_cannot_run():
    import torch
    g = synth.rng(86, 1)
    Wt = synth.weights_kaiming(g, 6, 1, 3, 3)            # 6 channels: not a multiple of 4
    scheme, bits = O.assign_rows(Wt, (60, 35, 5))
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, synth.alpha_rows(Wt))
    a = torch.zeros((1, 4, 4, 8), dtype=torch.int8, device="cuda")
    y = torch.zeros((1, 4, 4, 8), dtype=torch.float32, device="cuda")
    with pytest.raises(R.RmsmpError) as e:
        R.rmsmp_conv_depthwise(layer, d_packed, a, 1, 4, 4, 1, 1, 0.1, y)
    assert e.value.status == R.ERR_VARIANT
    Wd = synth.weights_kaiming(g, 8, 2, 3, 3)            # an ordinary layer is not a depthwise one
    scheme, bits = O.assign_rows(Wd, (60, 35, 5))
    layer, d_packed = Hn.pack_layer(Wd, scheme, bits, synth.alpha_rows(Wd))
    with pytest.raises(R.RmsmpError) as e:
        R.rmsmp_conv_depthwise(layer, d_packed, a, 1, 4, 4, 1, 1, 0.1, y)
    assert e.value.status == R.ERR_SHAPE


# ---------------------------------------------------------------- first layer (few channels) as a patch matrix
@pytest.mark.gpu
@pytest.mark.parametrize("M,Cin,k,stride,pad,B,H,W,pitch", [
    (64, 3, 7, 2, 3, 2, 30, 26, 3),        # the networks' first layer (Section 4.1): 3 channels, 7 x 7, stride 2
    (24, 3, 3, 1, 1, 1, 9, 7, 4),          # a padded pixel pitch
    (40, 1, 5, 1, 0, 2, 8, 8, 1),
    (16, 64, 3, 1, 1, 1, 4, 262, 64),      # input rows too wide for shared memory: the direct-gather form
])
def test_first_layer_patch_matrix_and_gemm_match_oracle_conv(M, Cin, k, stride, pad, B, H, W, pitch):
    import torch
    g = synth.rng(91, M + Cin + H)
    Wt = synth.weights_normal(g, (M, Cin, k, k))
    scheme, bits = O.assign_rows(Wt.reshape(M, -1), (60, 35, 5))
    alpha = synth.alpha_rows(Wt.reshape(M, -1))
    act = synth.act_codes_uniform(g, (B, H, W, Cin))
    K = k * k * Cin
    ld = (K + 15) // 16 * 16
    # patch matrix on the device against the oracle's
    a = torch.zeros((B, H, W, pitch), dtype=torch.int8, device="cuda")
    a[..., :Cin] = torch.from_numpy(act).cuda()
    Ho, Wo = O.conv_out_hw(H, W, k, k, stride, pad)
    N = B * Ho * Wo
    cols = torch.full((N, ld), 99, dtype=torch.int8, device="cuda")
    R.rmsmp_im2col_codes(a, B, H, W, Cin, pitch, k, k, stride, pad, cols, ld)
    torch.cuda.synchronize()
    assert np.array_equal(cols.cpu().numpy(), O.im2col(act, k, k, stride, pad, ld))
    # the layer as a linear layer over the patches, filters flattened tap-major with zero columns appended
    Wl = np.zeros((M, ld), np.float32)
    Wl[:, :K] = Wt.transpose(0, 2, 3, 1).reshape(M, K)
    layer, d_packed = Hn.pack_layer(Wl, scheme, bits, alpha)
    step = np.float32(0.05)
    y = torch.full((N, M), float("nan"), dtype=torch.float32, device="cuda")
    acc = torch.zeros((N, M), dtype=torch.int32, device="cuda")
    R.rmsmp_gemm_variant(layer, d_packed, cols, N, ld, float(step), y, M, R.OUT_NM, acc, R.VARIANT_AUTO)
    torch.cuda.synchronize()
    assert R.rmsmp_last_device_status(d_packed) == R.OK
    _, _, acc_ref, y_ref = O.layer_conv(Wt, scheme, bits, alpha, act, step, stride, pad)
    assert np.array_equal(acc.cpu().numpy(), acc_ref.reshape(N, M))
    assert np.array_equal(y.cpu().numpy().view(np.uint32), y_ref.reshape(N, M).view(np.uint32))


@pytest.mark.gpu
@pytest.mark.parametrize("C,kh,kw,stride,pad,B,H,W,ld,offset", [
    (3, 7, 7, 2, 3, 1, 21, 70, 160, 0),        # more than one group of 32 pixels, the last one ragged
    (3, 7, 7, 2, 3, 2, 9, 11, 160, 5),         # input that does not start on a 16-byte boundary
    (1, 3, 3, 1, 1, 1, 6, 5, 16, 3),           # six runs of three bytes in a row's sixteen columns
    (1, 2, 1, 1, 0, 1, 4, 4, 48, 0),           # runs of one byte, zero columns beyond a whole unit
    (5, 3, 3, 3, 4, 1, 8, 300, 4096, 1),       # a tile of five pixels, padding wider than the image needs
    (2, 16, 16, 8, 16, 1, 3, 3, 512, 0),       # the largest filter: mostly padding
    (64, 3, 3, 1, 1, 1, 3, 33, 576, 0),        # runs longer than a unit
])
def test_patch_matrix_pieces(C, kh, kw, stride, pad, B, H, W, ld, offset):
    """Bytes are copied, so they must be the oracle's; the bytes around the matrix stay as they were."""
    import torch
    g = synth.rng(92, C + H + W)
    act = g.integers(-128, 128, size=(B, H, W, C), dtype=np.int8)
    raw = torch.full((offset + act.size + 64,), 77, dtype=torch.int8, device="cuda")
    raw[offset:offset + act.size] = torch.from_numpy(act.reshape(-1)).cuda()
    ref = O.im2col(act, kh, kw, stride, pad, ld)
    out = torch.full((ref.size + 256,), 99, dtype=torch.int8, device="cuda")
    R.rmsmp_im2col_codes(raw.data_ptr() + offset, B, H, W, C, C, kh, kw, stride, pad, out[128:], ld)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.array_equal(got[128:-128].reshape(ref.shape), ref)
    assert (got[:128] == 99).all() and (got[-128:] == 99).all()


@pytest.mark.gpu
@pytest.mark.parametrize("C,pitch,k,stride,pad,B,H,W,offset", [
    (3, 4, 7, 2, 3, 2, 9, 77, 0), (4, 16, 3, 1, 1, 2, 6, 40, 0), (1, 4, 5, 1, 2, 1, 5, 9, 4),      # a word a pixel
    (3, 4, 3, 1, 1, 1, 5, 6, 1), (24, 25, 3, 1, 1, 2, 5, 8, 0), (5, 7, 5, 3, 4, 2, 6, 11, 3),      # byte by byte
    (24, 32, 3, 1, 1, 2, 6, 9, 0), (12, 20, 3, 2, 0, 1, 7, 9, 8),                                   # four bytes at a time
    (32, 48, 3, 1, 1, 2, 5, 9, 0), (16, 64, 5, 1, 2, 1, 6, 7, 16),                                  # sixteen
    (3, 3, 7, 2, 3, 1, 320, 1100, 0), (3, 4, 7, 2, 3, 1, 320, 1100, 0),                             # rows that need more shared memory
    (16, 16, 5, 1, 2, 1, 160, 300, 0), (8, 12, 5, 1, 2, 1, 160, 500, 4),
    (3, 4, 7, 2, 3, 1, 20, 1100, 0),                                                                # ... and too few of them for that
])
def test_patch_matrix_of_padded_and_wide_pixels(C, pitch, k, stride, pad, B, H, W, offset):
    """The bytes between pixels are not zero and must not show; the tensor ends with the last pixel's channels."""
    import torch
    g = synth.rng(94, C + pitch + W)
    act = g.integers(-128, 128, size=(B, H, W, C), dtype=np.int8)
    pixels = np.full((B * H * W, pitch), 55, np.int8)
    pixels[:, :C] = act.reshape(-1, C)
    flat = pixels.reshape(-1)[:(B * H * W - 1) * pitch + C]
    a = torch.full((offset + flat.size,), 55, dtype=torch.int8, device="cuda")
    a[offset:] = torch.from_numpy(flat).cuda()
    Ho, Wo = O.conv_out_hw(H, W, k, k, stride, pad)
    ld = (k * k * C + 15) // 16 * 16
    N = B * Ho * Wo
    buf = torch.full((N * ld + 256,), 99, dtype=torch.int8, device="cuda")
    R.rmsmp_im2col_codes(a[offset:], B, H, W, C, pitch, k, k, stride, pad, buf[128:128 + N * ld], ld)
    torch.cuda.synchronize()
    assert np.array_equal(buf[128:128 + N * ld].cpu().numpy().reshape(N, ld), O.im2col(act, k, k, stride, pad, ld))
    assert (buf[:128] == 99).all() and (buf[128 + N * ld:] == 99).all()



@pytest.mark.gpu
def test_patch_matrix_rejects_bad_arguments():
    import torch
    a = torch.zeros((1, 4, 4, 3), dtype=torch.int8, device="cuda")
    cols = torch.zeros((16, 32), dtype=torch.int8, device="cuda")
    for args, status in [((a, 1, 4, 4, 3, 3, 3, 3, 1, 1, cols, 16), R.ERR_SHAPE),       # ld_cols below kh*kw*C
                         ((a, 1, 4, 4, 3, 3, 3, 3, 1, 1, cols, 40), R.ERR_ALIGN),       # not a multiple of 16
                         ((a, 1, 4, 4, 3, 2, 3, 3, 1, 1, cols, 32), R.ERR_SHAPE),       # pitch below the channel count
                         ((a, 1, 4, 4, 3, 3, 7, 7, 1, 0, cols, 160), R.ERR_SHAPE)]:     # filter larger than the image
        with pytest.raises(R.RmsmpError) as e:
            R.rmsmp_im2col_codes(*args)
        assert e.value.status == status


# ---------------------------------------------------------------- resident weights expanded by the CTA itself
@pytest.mark.gpu
@pytest.mark.parametrize("M,K,N,layout", [
    (48, 192, 300, R.OUT_MN),       # duplicated rows (M <= 64), 64-byte k-blocks, [M][N] output
    (100, 64, 515, R.OUT_NM),       # rows beyond M in the block, one short k-block
    (128, 576, 77, R.OUT_NM),       # the largest resident stripe (72 KB expanded)
    (64, 448, 1000, R.OUT_NM),      # 64-byte k-blocks with a last chunk of 64 codes
])
def test_linear_layer_without_workspace_on_resident_weights(M, K, N, layout):
    """A layer of one row block whose expanded weights stay in shared memory is expanded once per CTA from the
    packed codes (no workspace): every kind of row, both output layouts, with the raw sums."""
    g = synth.rng(93, M + K + N)
    W = synth.weights_normal(g, (M, K))
    scheme, bits = _mixed_map(M, M + K, (50, 30, 20))
    alpha = synth.alpha_rows(W)
    act = g.integers(-8, 16, (N, K), dtype=np.int8)
    layer, d_packed = Hn.pack_layer(W, scheme, bits, alpha)
    y, acc = Hn.gemm(layer, d_packed, act, 0.125, R.VARIANT_TENSOR, out_layout=layout)
    v_ref, ws = O.quantize_rows(W, scheme, bits, alpha)
    _check_layer_outputs(y, acc, O.matmul(v_ref, act), ws, np.float32(0.125), alpha, scheme, bits)


@pytest.mark.parametrize("variant", [R.VARIANT_AUTO, Hn.WORKSPACE], ids=["plain", "workspace"])
@pytest.mark.parametrize("M,Cin,k,B,H,W", [
    (130, 64, 1, 38001, 1, 1),      # two row blocks, the second of two rows; more than two tiles per SM
    (1930, 96, 1, 5121, 1, 1),      # sixteen row blocks: a grid of 144 CTAs, a last tile of one pixel
    (300, 160, 1, 27, 41, 37),      # 64-byte k-blocks with a half-used last chunk, tiles of whole image rows
    (200, 64, 3, 13, 56, 56),       # three taps per stage, shifted columns
    (140, 64, 3, 1, 9, 13),         # a tile per row block
])
def test_resident_weights_of_several_row_blocks(M, Cin, k, B, H, W, variant):
    """Every CTA keeps the weights of one of the layer's row blocks: exact sums and outputs for every block."""
    g = synth.rng(96, M + Cin + W)
    Wt = synth.weights_kaiming(g, M, Cin, k, k)
    scheme, bits = _mixed_map(M, M + k, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    act = g.integers(-8, 16, size=(B, H, W, Cin)).astype(np.int8)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    _, ws, acc_ref, y_ref = O.layer_conv(Wt, scheme, bits, alpha, act, np.float32(0.25), 1, k // 2)
    y, acc = Hn.conv(layer, d_packed, act, 1, k // 2, 0.25, variant)
    assert np.array_equal(acc, acc_ref.reshape(-1, M))
    assert np.array_equal(y.view(np.uint32), y_ref.reshape(-1, M).view(np.uint32))


@pytest.mark.parametrize("layout", [R.OUT_NM, R.OUT_MN], ids=["nm", "mn"])
@pytest.mark.parametrize("variant", [R.VARIANT_AUTO, Hn.WORKSPACE], ids=["plain", "workspace"])
@pytest.mark.parametrize("M,Cin,k,stride,B,H,W", [
    (130, 64, 3, 1, 40, 29, 31),     # four tiles of eight rows: three rows twice
    (96, 160, 3, 1, 60, 23, 32),     # tiles of 256 pixels that start at no multiple of the tile
    (256, 128, 3, 1, 45, 17, 19),    # halves of six rows for pairs of CTAs, pixels of no multiple of 32
    (64, 16, 5, 2, 40, 74, 41),      # a stride of two
    (72, 32, 1, 1, 90, 29, 23),      # a 1x1 layer: tiles across images
])
def test_images_whose_rows_no_tile_divides(M, Cin, k, stride, B, H, W, variant, layout):
    """The last tile of an image repeats rows of the one before it: exact everywhere, nothing beyond."""
    g = synth.rng(97, M + Cin + W)
    Wt = synth.weights_kaiming(g, M, Cin, k, k)
    scheme, bits = _mixed_map(M, M + k, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    act = g.integers(-8, 16, size=(B, H, W, Cin)).astype(np.int8)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    _, ws, acc_ref, y_ref = O.layer_conv(Wt, scheme, bits, alpha, act, np.float32(0.25), stride, k // 2)
    for want_acc in (True, False):
        y, acc = Hn.conv(layer, d_packed, act, stride, k // 2, 0.25, variant, layout, want_acc)
        if want_acc:
            assert np.array_equal(acc, acc_ref.reshape(-1, M))
        assert np.array_equal(np.ascontiguousarray(y).view(np.uint32), y_ref.reshape(-1, M).view(np.uint32))


@pytest.mark.parametrize("mix", [(50, 30, 20), (100, 0, 0), (0, 0, 100), (0, 100, 0)], ids=lambda m: "%d-%d-%d" % m)
@pytest.mark.parametrize("M,Cin,k,B,H,W", [
    (2500, 96, 1, 7401, 1, 1),       # twenty row blocks that change from tile to tile, one k-block a tile, a step unused
    (2500, 192, 1, 7401, 1, 1),      # two k-blocks: a group's next tile is one or two ahead
    (300, 1024, 1, 16001, 1, 1),     # a row block per CTA, three of them
    (16, 304, 5, 11, 43, 37),        # few rows; a last chunk of 48 channels
    (200, 48, 5, 30, 31, 33),        # 64-byte k-blocks, one and a half steps
])
def test_weights_expanded_for_every_tile(M, Cin, k, B, H, W, mix):
    """Neither a workspace nor room for a row block's weights: every kind of row, alone and mixed, exact."""
    g = synth.rng(98, M + Cin + W)
    Wt = synth.weights_kaiming(g, M, Cin, k, k)
    scheme, bits = _mixed_map(M, M + k, mix)
    alpha = synth.alpha_rows(Wt)
    act = g.integers(-8, 16, size=(B, H, W, Cin)).astype(np.int8)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    _, ws, acc_ref, y_ref = O.layer_conv(Wt, scheme, bits, alpha, act, np.float32(0.25), 1, k // 2)
    y, acc = Hn.conv(layer, d_packed, act, 1, k // 2, 0.25, R.VARIANT_TENSOR)
    assert np.array_equal(acc, acc_ref.reshape(-1, M))
    assert np.array_equal(y.view(np.uint32), y_ref.reshape(-1, M).view(np.uint32))


@pytest.mark.parametrize("M", [129, 144, 192, 193, 336])
@pytest.mark.parametrize("variant", [R.VARIANT_AUTO, Hn.WORKSPACE], ids=["plain", "workspace"])
def test_resident_weights_whose_last_row_block_is_short(M, variant):
    """The last block's rows lie twice in tensor memory and its tiles go to fewer CTAs: exact, and the codes of the
    re-quantizing call are the quantizer's."""
    import torch
    Cin, B, H, W = 64, 61, 31, 29
    g = synth.rng(99, M)
    Wt = synth.weights_kaiming(g, M, Cin, 1, 1)
    scheme, bits = _mixed_map(M, M, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    act = g.integers(0, 16, size=(B, H, W, Cin)).astype(np.int8)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    _, ws, acc_ref, y_ref = O.layer_conv(Wt, scheme, bits, alpha, act, np.float32(0.25), 1, 0)
    y, acc = Hn.conv(layer, d_packed, act, 1, 0, 0.25, variant)
    assert np.array_equal(acc, acc_ref.reshape(-1, M))
    assert np.array_equal(y.view(np.uint32), y_ref.reshape(-1, M).view(np.uint32))
    if variant == Hn.WORKSPACE:
        want, _ = O.quantize_act(y_ref.reshape(-1, M), 4.0, R.ACT_U4)
        codes = torch.full((B * H * W, M), 99, dtype=torch.int8, device="cuda")
        d_ws = torch.empty(R.rmsmp_workspace_bytes(layer), dtype=torch.int8, device="cuda")
        R.rmsmp_expand_weights(layer, d_packed, d_ws)
        R.rmsmp_conv_implicit_workspace_requant(layer, d_packed, d_ws, torch.from_numpy(act).cuda(), B, H, W, 1, 0, 0.25, 4.0, R.ACT_U4, codes)
        assert np.array_equal(codes.cpu().numpy(), want)


# ------------------------------------------------------------------ column-shift stages

def _check_some_images(Wt, scheme, bits, alpha, act, stride, pad, y, acc, images):
    """Sums and outputs of those images against the oracle's convolution of them alone."""
    M, B = Wt.shape[0], act.shape[0]
    _, _, acc_ref, y_ref = O.layer_conv(Wt, scheme, bits, alpha, np.ascontiguousarray(act[images]), np.float32(0.25), stride, pad)
    assert np.array_equal(y.reshape(B, -1, M)[images].view(np.uint32), y_ref.reshape(len(images), -1, M).view(np.uint32))
    if acc is not None:
        assert np.array_equal(acc.reshape(B, -1, M)[images], acc_ref.reshape(len(images), -1, M))


@pytest.mark.parametrize("M,Cin,B,H,W", [
    (48, 64, 300, 13, 11),         # rows of 11 pixels: a tap's rows start anywhere in the swizzle pattern
    (100, 32, 35, 37, 35),        # tiles of seven rows, the last one repeats rows; one 32-code step a tap
    (64, 48, 16, 51, 51),
    (128, 80, 150, 29, 9),        # two chunks a tap (the second of one step), weights of 144 KB resident
    (20, 128, 150, 29, 9),        # the same with duplicated rows
    (72, 96, 300, 15, 17),        # one image of 255 pixels a tile
])
def test_column_shift_stages_of_any_width(M, Cin, B, H, W):
    g = synth.rng(140, M + Cin + W)
    Wt = synth.weights_kaiming(g, M, Cin, 3, 3)
    scheme, bits = _mixed_map(M, 11, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    act = g.integers(-16, 17, size=(B, H, W, Cin)).astype(np.int8)
    images = sorted({0, 1, B // 2, B - 1})
    for want_acc in (True, False):
        y, acc = Hn.conv(layer, d_packed, act, 1, 1, 0.25, Hn.WORKSPACE, want_acc=want_acc)
        _check_some_images(Wt, scheme, bits, alpha, act, 1, 1, y, acc, images)


@pytest.mark.parametrize("want_acc", [True, False])
@pytest.mark.parametrize("M,Cin,B,H,W", [
    (128, 80, 150, 29, 9),        # the output turned in shared memory
    (20, 128, 150, 29, 9),
    (128, 128, 300, 16, 16),      # by bulk stores
])
def test_wide_column_shift_stages_into_rows_of_pixels(M, Cin, B, H, W, want_acc):
    g = synth.rng(148, M + Cin + W)
    Wt = synth.weights_kaiming(g, M, Cin, 3, 3)
    scheme, bits = _mixed_map(M, 13, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    act = g.integers(-16, 17, size=(B, H, W, Cin)).astype(np.int8)
    y, acc = Hn.conv(layer, d_packed, act, 1, 1, 0.25, Hn.WORKSPACE, R.OUT_MN, want_acc=want_acc)
    _check_some_images(Wt, scheme, bits, alpha, act, 1, 1, y, acc, sorted({0, 1, B // 2, B - 1}))


@pytest.mark.parametrize("Cin,B,H,W", [
    (256, 387, 7, 7),             # two images a half with staged rows between them, the last half has one
    (256, 200, 11, 13),           # halves of six rows, the last of an image repeats one
    (256, 100, 14, 14),
    (384, 230, 9, 9),             # three channel chunks, an image a half
    (256, 40, 5, 100),            # halves of a row: no column shift
    (256, 35, 20, 28),            # stages so large that two of them make the ring
])
def test_column_shift_stages_of_cta_pairs(Cin, B, H, W):
    M = 256
    g = synth.rng(141, Cin + W)
    Wt = synth.weights_kaiming(g, M, Cin, 3, 3)
    scheme, bits = _mixed_map(M, 12, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    act = g.integers(-16, 17, size=(B, H, W, Cin)).astype(np.int8)
    y, _ = Hn.conv(layer, d_packed, act, 1, 1, 0.25, Hn.WORKSPACE, want_acc=False)
    _check_some_images(Wt, scheme, bits, alpha, act, 1, 1, y, None, sorted({0, 1, B // 2, B - 2, B - 1}))


@pytest.mark.parametrize("kind", [R.ACT_U4, R.ACT_S4])
@pytest.mark.parametrize("M,Cin,k,B,H,W,ld_extra", [
    (144, 32, 1, 40, 31, 33, 16),       # a second row block of one 16-byte piece, ragged tiles, padding columns
    (48, 64, 3, 100, 21, 19, 0),        # duplicated rows, 48 of 64; column shift
    (128, 128, 3, 150, 29, 9, 0),       # resident weights of two chunks a tap
])
def test_requantized_codes_leave_in_sixteen_byte_pieces(M, Cin, k, B, H, W, ld_extra, kind):
    import torch
    g = synth.rng(142, M + Cin)
    Wt = synth.weights_kaiming(g, M, Cin, k, k)
    scheme, bits = O.assign_rows(Wt, (60, 35, 5))
    alpha = synth.alpha_rows(Wt)
    act = synth.act_codes_uniform(g, (B, H, W, Cin))
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    ws = torch.empty(R.rmsmp_workspace_bytes(layer), dtype=torch.int8, device="cuda")
    R.rmsmp_expand_weights(layer, d_packed, ws)
    N, pad = B * H * W, k // 2
    images = [0, B // 2, B - 1]
    _, _, _, y_ref = O.layer_conv(Wt, scheme, bits, alpha, np.ascontiguousarray(act[images]), np.float32(0.125), 1, pad)
    na = _next_alpha(y_ref)
    want, _ = O.quantize_act(y_ref.reshape(len(images), H * W, M), na, kind)
    a = torch.from_numpy(act).cuda()
    out = torch.full((N, M + ld_extra), 99, dtype=torch.int8, device="cuda")
    if ld_extra:
        R.rmsmp_gemm_workspace_requant(layer, d_packed, ws, a, N, Cin, 0.125, na, kind, out, M + ld_extra)
    else:
        R.rmsmp_conv_implicit_workspace_requant(layer, d_packed, ws, a, B, H, W, 1, pad, 0.125, na, kind, out)
    torch.cuda.synchronize()
    assert R.rmsmp_last_device_status(d_packed) == R.OK
    got = out.cpu().numpy()
    assert np.array_equal(got[:, :M].reshape(B, H * W, M)[images], want)
    assert (got[:, M:] == 99).all()


@pytest.mark.parametrize("k,stride,pad,B,H,W,offset", [
    (7, 2, 3, 3, 37, 64, 0),       # eight output rows a pass, the last one of an image has three
    (7, 2, 3, 1, 9, 223, 1),       # two rows a pass; rows that start at any byte
    (7, 3, 0, 2, 40, 65, 3),
    (3, 2, 1, 2, 31, 31, 0),       # more rows a pass than pixels would need
    (3, 1, 4, 1, 5, 6, 2),         # padding wider than the filter
    (3, 2, 1, 1, 200, 500, 0),
    (5, 2, 2, 2, 33, 47, 7),       # rows of five units
    (5, 4, 2, 1, 17, 300, 0),
    (7, 2, 3, 1, 3, 1, 5),         # a row of one pixel
])
def test_patch_matrix_of_three_channels(k, stride, pad, B, H, W, offset):
    """Bytes are copied: the oracle's, and nothing around them."""
    import torch
    g = synth.rng(143, k + H + W)
    act = g.integers(-128, 128, size=(B, H, W, 3), dtype=np.int8)
    raw = torch.full((offset + act.size,), 77, dtype=torch.int8, device="cuda")
    raw[offset:] = torch.from_numpy(act.reshape(-1)).cuda()
    ld = (3 * k * k + 15) // 16 * 16
    ref = O.im2col(act, k, k, stride, pad, ld)
    out = torch.full((ref.size + 256,), 99, dtype=torch.int8, device="cuda")
    R.rmsmp_im2col_codes(raw[offset:], B, H, W, 3, 3, k, k, stride, pad, out[128:], ld)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.array_equal(got[128:-128].reshape(ref.shape), ref)
    assert (got[:128] == 99).all() and (got[-128:] == 99).all()


@pytest.mark.parametrize("stride,B", [(1, 2048), (2, 4096)])
def test_depthwise_threads_that_take_several_strips(stride, B):
    """A thread's copies for one strip are over before those for the next begin."""
    import torch
    C, H = 96, 7
    g = synth.rng(144, B)
    Wt = synth.weights_kaiming(g, C, 1, 3, 3)
    scheme, bits = O.assign_rows(Wt, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    codes = g.integers(-128, 128, size=(B, H, H, C), dtype=np.int8)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    v_ref, wstep = O.quantize_rows(Wt.reshape(C, -1), scheme, bits, alpha)
    acc_ref = O.conv_depthwise(v_ref.reshape(C, 3, 3), codes, stride, 1)
    y = torch.full(acc_ref.shape, float("nan"), dtype=torch.float32, device="cuda")
    R.rmsmp_conv_depthwise(layer, d_packed, torch.from_numpy(codes).cuda(), B, H, H, stride, 1, 0.5, y)
    torch.cuda.synchronize()
    assert np.array_equal(y.cpu().numpy().view(np.uint32), O.epilogue(acc_ref, wstep, np.float32(0.5)).view(np.uint32))


@pytest.mark.parametrize("C,H,W,B,stride,with_acc", [
    (96, 32, 1, 1528, 1, False),        # strips of eleven rows through the ring, two for some threads
    (28, 32, 5, 2697, 1, False),
    (1028, 11, 1, 446, 1, False),       # several channel quads a thread
    (100, 29, 6, 64, 1, False),         # strips of fewer rows, in registers
    (20000, 11, 1, 100, 1, False),      # the ring beside a filter table of 180 KB
    (22752, 11, 1, 100, 1, False),      # no room for it beside the widest table
    (22260, 11, 1, 100, 1, False), (22300, 11, 1, 100, 1, False), (22340, 11, 1, 100, 1, False), (22416, 11, 1, 100, 1, False),      # the last tables with room, and the next
    (528, 14, 1, 464, 2, False),        # of stride two, two strips for some threads
    (516, 13, 4, 488, 2, False),
    (576, 30, 30, 43, 2, False),        # five rows twice, and six once
    (516, 43, 43, 9, 2, False),
    (20604, 13, 1, 40, 2, False), (18000, 13, 1, 100, 2, False),      # most threads have an item: registers
    (22752, 5, 3, 1, 1, True), (22752, 5, 4, 2, 2, False), (20604, 5, 3, 2, 2, False), (22752, 5, 3, 1, 2, True),
])
def test_depthwise_strips_with_and_without_a_ring(C, H, W, B, stride, with_acc):
    import torch
    g = synth.rng(145, C + H + B)
    Wt = synth.weights_kaiming(g, C, 1, 3, 3)
    scheme, bits = O.assign_rows(Wt, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    codes = g.integers(-128, 128, size=(B, H, W, C), dtype=np.int8)
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    v_ref, wstep = O.quantize_rows(Wt.reshape(C, -1), scheme, bits, alpha)
    acc_ref = O.conv_depthwise(v_ref.reshape(C, 3, 3), codes, stride, 1)
    y = torch.full(acc_ref.shape, float("nan"), dtype=torch.float32, device="cuda")
    acc = torch.full(acc_ref.shape, -5, dtype=torch.int32, device="cuda")
    R.rmsmp_conv_depthwise(layer, d_packed, torch.from_numpy(codes).cuda(), B, H, W, stride, 1, 0.5, y, acc if with_acc else None)
    torch.cuda.synchronize()
    if with_acc:
        assert np.array_equal(acc.cpu().numpy(), acc_ref)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), O.epilogue(acc_ref, wstep, np.float32(0.5)).view(np.uint32))


@pytest.mark.parametrize("k,stride,pad,B,H,W,offset", [
    (7, 2, 3, 64, 37, 64, 0),      # eight output rows a pass, the last one of an image has three
    (7, 2, 3, 40, 9, 223, 1),      # a pass of two rows, or one
    (3, 2, 1, 200, 31, 31, 0),     # more rows a pass than pixels would need
    (3, 1, 4, 100, 5, 6, 2),       # padding wider than the filter
    (5, 2, 2, 30, 33, 47, 7),      # three rows a pass: as many as leave every SM a pass
    (5, 4, 2, 300, 17, 40, 3),     # a step of four: passes enough
    (5, 4, 2, 100, 17, 40, 3),     # too few
])
def test_patch_matrix_of_three_channels_and_many_rows(k, stride, pad, B, H, W, offset):
    import torch
    g = synth.rng(146, k + H + W)
    act = g.integers(-128, 128, size=(B, H, W, 3), dtype=np.int8)
    raw = torch.full((offset + act.size,), 77, dtype=torch.int8, device="cuda")
    raw[offset:] = torch.from_numpy(act.reshape(-1)).cuda()
    ld = (3 * k * k + 15) // 16 * 16
    ref = O.im2col(act, k, k, stride, pad, ld)
    out = torch.full((ref.size + 256,), 99, dtype=torch.int8, device="cuda")
    R.rmsmp_im2col_codes(raw[offset:], B, H, W, 3, 3, k, k, stride, pad, out[128:], ld)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.array_equal(got[128:-128].reshape(ref.shape), ref)
    assert (got[:128] == 99).all() and (got[-128:] == 99).all()


@pytest.mark.parametrize("M,Cin,k,stride,B,H", [
    (32, 32, 7, 2, 145, 11),       # through the rings, sixteen codes a store
    (144, 80, 5, 1, 9, 17),        # two row blocks, the second of sixteen rows
    (256, 1040, 1, 1, 40, 13),     # 1x1 with a last chunk of sixteen channels
    (68, 96, 5, 1, 9, 17),         # codes one by one
    (20, 144, 3, 1, 30, 15),       # the same with duplicated rows
    (332, 384, 3, 1, 70, 7),
    (288, 288, 1, 2, 21, 50),      # resident weights of five k-blocks
    (144, 32, 1, 1, 75, 32),       # of one, and four rounds of tiles
    (148, 32, 1, 1, 75, 32),       # the same one by one
])
def test_requantized_codes_of_long_and_of_short_tiles(M, Cin, k, stride, B, H):
    import torch
    g = synth.rng(147, M + Cin)
    Wt = synth.weights_kaiming(g, M, Cin, k, k)
    scheme, bits = _mixed_map(M, M, (50, 30, 20))
    alpha = synth.alpha_rows(Wt)
    act = synth.act_codes_uniform(g, (B, H, H, Cin))
    layer, d_packed = Hn.pack_layer(Wt, scheme, bits, alpha)
    ws = torch.empty(R.rmsmp_workspace_bytes(layer), dtype=torch.int8, device="cuda")
    R.rmsmp_expand_weights(layer, d_packed, ws)
    images = sorted({0, B // 2, B - 1})
    _, _, _, y_ref = O.layer_conv(Wt, scheme, bits, alpha, np.ascontiguousarray(act[images]), np.float32(0.125), stride, k // 2)
    na = _next_alpha(y_ref)
    Ho = (H + 2 * (k // 2) - k) // stride + 1
    for kind in (R.ACT_U4, R.ACT_S4):
        want, _ = O.quantize_act(y_ref.reshape(len(images), Ho * Ho, M), na, kind)
        out = torch.full((B * Ho * Ho, M), 99, dtype=torch.int8, device="cuda")
        R.rmsmp_conv_implicit_workspace_requant(layer, d_packed, ws, torch.from_numpy(act).cuda(), B, H, H, stride, k // 2, 0.125, na, kind, out)
        torch.cuda.synchronize()
        assert R.rmsmp_last_device_status(d_packed) == R.OK
        assert np.array_equal(out.cpu().numpy().reshape(B, Ho * Ho, M)[images], want)
