"""The tcgen05 BF16 GEMM (the learned depth prior's contraction) against an
FP64 product of the same BF16 values.  FP32 accumulation over K terms is held to
|C - ref| <= 2e-6 * sum_k |a_k b_k| (K * 2^-24 with margin); BF16 outputs to one
BF16 rounding (2^-8 relative) on top."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2409_09295_gb300 import _abi, raster  # noqa: E402


def bf16_round(x):
    """Round float32 values to bfloat16 (nearest even); returns (values, bits)."""
    u = np.ascontiguousarray(x, np.float32).view(np.uint32)
    b = ((u + 0x7FFF + ((u >> 16) & 1)) >> 16).astype(np.uint16)
    return (b.astype(np.uint32) << 16).view(np.float32), b


def to_dev_bf16(bits):
    return torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)


@pytest.mark.parametrize("M,N,K", [(128, 16, 64), (1000, 48, 200), (300, 256, 1728),
                                   (77, 300, 96), (4096, 128, 576), (130, 32, 8)])
def test_gemm_bf16_fp32_out(M, N, K):
    rs = np.random.default_rng(M + N + K)
    a, abits = bf16_round(rs.normal(size=(M, K)).astype(np.float32))
    b, bbits = bf16_round(rs.normal(size=(N, K)).astype(np.float32))
    bias = rs.normal(size=N).astype(np.float32)
    ws = torch.zeros(1024, dtype=torch.uint8, device="cuda")
    C = torch.zeros(M, N, dtype=torch.float32, device="cuda")
    tb = torch.from_numpy(bias).cuda()
    _abi.gevo_gemm_bf16(M, N, K, to_dev_bf16(abits), K, to_dev_bf16(bbits), K, C, N, False, tb,
                        False, 0.0, ws)
    torch.cuda.synchronize()
    assert _abi.gevo_last_error(ws) == 0
    ref = a.astype(np.float64) @ b.astype(np.float64).T + bias
    scale = np.abs(a).astype(np.float64) @ np.abs(b).astype(np.float64).T + np.abs(bias)
    err = np.abs(C.cpu().numpy() - ref)
    assert (err <= 2e-6 * scale + 1e-30).all(), (err / scale).max()


def test_gemm_bf16_relu_bf16_out_and_accumulate():
    M, N, K = 513, 64, 144
    rs = np.random.default_rng(7)
    a, abits = bf16_round(rs.normal(size=(M, K)).astype(np.float32))
    b, bbits = bf16_round(rs.normal(size=(N, K)).astype(np.float32))
    ws = torch.zeros(1024, dtype=torch.uint8, device="cuda")
    C = torch.zeros(M, N, dtype=torch.bfloat16, device="cuda")
    _abi.gevo_gemm_bf16(M, N, K, to_dev_bf16(abits), K, to_dev_bf16(bbits), K, C, N, True, None,
                        True, 0.0, ws)
    ref = np.maximum(a.astype(np.float64) @ b.astype(np.float64).T, 0)
    got = C.float().cpu().numpy()
    scale = np.abs(a).astype(np.float64) @ np.abs(b).astype(np.float64).T
    assert (np.abs(got - ref) <= 2 ** -8 * np.abs(ref) + 2e-6 * scale + 1e-30).all()
    # accumulate: C = A B^T + 1.0 * C (FP32 output)
    C2 = torch.full((M, N), 0.5, dtype=torch.float32, device="cuda")
    _abi.gevo_gemm_bf16(M, N, K, to_dev_bf16(abits), K, to_dev_bf16(bbits), K, C2, N, False,
                        None, False, 1.0, ws)
    ref2 = a.astype(np.float64) @ b.astype(np.float64).T + 0.5
    assert (np.abs(C2.cpu().numpy() - ref2) <= 2e-6 * scale + 1e-6).all()
    assert _abi.gevo_last_error(ws) == 0


@pytest.mark.parametrize("nb,H,W,Cin,Cout", [(2, 6, 10, 24, 8), (1, 12, 20, 8, 40), (3, 5, 8, 16, 16)])
def test_conv_and_weight_gradient_ragged_sizes(nb, H, W, Cin, Cout):
    """The implicit-GEMM convolution and weight gradient (gathered A operands) on
    sizes that leave partial row tiles, partial column tiles and a partial last
    K slice (P = nb H W not a multiple of 64, 9 Cin not of 128), against the
    FP64 oracle convolution on the same BF16 values."""
    from oracle import unet as ounet
    rs = np.random.default_rng(nb * 1000 + H * 10 + Cin)
    P = nb * H * W
    x, xb = bf16_round(rs.normal(size=(nb, H, W, Cin)).astype(np.float32))
    w, wb = bf16_round(rs.normal(size=(Cout, 9, Cin)).astype(np.float32) * 0.2)
    dz, dzb = bf16_round(rs.normal(size=(nb, H, W, Cout)).astype(np.float32))
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    X = to_dev_bf16(xb.reshape(-1))
    Wt = to_dev_bf16(wb.reshape(-1))
    Y = torch.zeros(P * Cout, dtype=torch.float32, device="cuda")
    _abi.prior_call("gevo_conv3x3", nb, H, W, Cin, X, Cout, Wt, None, Y, Cout, 0, 0, 0.0, ws)
    dZt = to_dev_bf16(np.ascontiguousarray(dzb.reshape(P, Cout).T).reshape(-1))
    dW = torch.zeros(Cout * 9 * Cin, dtype=torch.float32, device="cuda")
    _abi.prior_call("gevo_conv3x3_wgrad", nb, H, W, Cin, X, Cout, dZt, dW, ws)
    torch.cuda.synchronize()
    assert _abi.gevo_last_error(ws) == 0
    x64, w64, dz64 = (a.astype(np.float64) for a in (x, w, dz))
    ref = ounet.conv3x3(x64, w64, np.zeros(Cout))
    mag = ounet.conv3x3(np.abs(x64), np.abs(w64), np.zeros(Cout))
    got = Y.cpu().numpy().reshape(nb, H, W, Cout)
    assert (np.abs(got - ref) <= 2e-6 * mag + 1e-30).all()
    _, dw_ref, _ = ounet.conv3x3_bwd(x64, w64, dz64)
    _, dw_mag, _ = ounet.conv3x3_bwd(np.abs(x64), w64, np.abs(dz64))
    got_dw = dW.cpu().numpy().reshape(Cout, 9, Cin)
    assert (np.abs(got_dw - dw_ref) <= 2e-6 * np.abs(dw_mag) + 1e-30).all()


def _conv_fp64(x, w):
    """3x3 zero-padded convolution in FP64 on the device: x NHWC, w [Cout, 9, Cin]."""
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    H, W = x.shape[1:3]
    return sum(xp[:, i:i + H, j:j + W] @ w[:, 3 * i + j].T for i in range(3) for j in range(3))


@pytest.mark.parametrize("nb,H,W,Cin,Cout", [
    (1, 16, 32, 16, 16),     # whole tiles
    (1, 1, 1, 16, 16),       # one pixel: every tap but the centre outside
    (2, 17, 33, 16, 24),     # one row and one column past a tile, partial column group
    (1, 15, 7, 8, 16),       # Cin = 8: two taps an instruction
    (1, 33, 18, 8, 250),
    (3, 16, 9, 40, 8),       # odd count of channel groups: a padding plane
    (1, 20, 24, 192, 64),    # column splits
    (1, 18, 10, 224, 16),    # near the most channels two tiles hold
    (1, 18, 10, 512, 32),    # beyond: the gathered GEMM
    (40, 30, 40, 32, 48),    # more tiles than CTAs: buffers reused
])
def test_convolution_tile_edges(nb, H, W, Cin, Cout):
    """The convolution at the edges of its tiles (8 mx columns x 16 rows, 16
    channels a step) against an FP64 convolution of the same BF16 values; FP32
    accumulation over 9 Cin terms within 2e-6 of the sum of magnitudes."""
    gen = torch.Generator("cuda").manual_seed(nb * 100 + H + Cin)
    P = nb * H * W
    x = torch.randn(nb, H, W, Cin, generator=gen, device="cuda").bfloat16()
    w = (0.2 * torch.randn(Cout, 9, Cin, generator=gen, device="cuda")).bfloat16()
    b = torch.randn(Cout, generator=gen, device="cuda")
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    ldy = Cout + 5                              # rows that keep no vector alignment
    Y = torch.full((P, ldy), 7.0, device="cuda")
    _abi.prior_call("gevo_conv3x3", nb, H, W, Cin, x, Cout, w, b, Y, ldy, 0, 0, 0.0, ws)
    Z = torch.full((P, Cout), 0.25, device="cuda").bfloat16()
    _abi.prior_call("gevo_conv3x3", nb, H, W, Cin, x, Cout, w, b, Z, Cout, 1, 1, 0.5, ws)
    torch.cuda.synchronize()
    assert _abi.gevo_last_error(ws) == 0
    ref = _conv_fp64(x.double(), w.double()).view(P, Cout) + b.double()
    mag = _conv_fp64(x.double().abs(), w.double().abs()).view(P, Cout) + b.double().abs()
    assert ((Y[:, :Cout].double() - ref).abs() <= 2e-6 * mag).all()
    assert (Y[:, Cout:] == 7.0).all()           # nothing past the row's columns
    want = (ref + 0.125).clamp_min(0)
    assert ((Z.double() - want).abs() <= 2 ** -8 * want.abs() + 2e-6 * (mag + 1)).all()


def test_convolution_keeps_infinities_local():
    """An infinite and a NaN activation reach only the 3x3 outputs around them,
    also where channel groups or taps are padded."""
    for Cin in (8, 16, 24):
        x = torch.rand(1, 20, 21, Cin, device="cuda").bfloat16()
        x[0, 4, 5, 1] = float("inf")
        x[0, 15, 20, Cin - 1] = float("nan")
        w = torch.rand(16, 9 * Cin, device="cuda").bfloat16()
        Y = torch.zeros(20 * 21, 16, device="cuda")
        ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
        _abi.prior_call("gevo_conv3x3", 1, 20, 21, Cin, x, 16, w, None, Y, 16, 0, 0, 0.0, ws)
        fin = torch.isfinite(Y.view(20, 21, 16)).all(-1)
        want = torch.ones(20, 21, dtype=torch.bool, device="cuda")
        want[3:6, 4:7] = False
        want[14:17, 19:21] = False
        assert torch.equal(fin, want)
        assert torch.isinf(Y.view(20, 21, 16)[3:6, 4:7]).all()


@pytest.mark.parametrize("nb,H,W,Cin,Cout", [
    (1, 1, 8, 8, 8),         # one row of eight pixels
    (2, 17, 24, 16, 16),     # partial tiles both ways, 48 of 64 rows
    (1, 33, 40, 48, 16),     # shifted operand: dZ (fewer channels)
    (2, 9, 32, 16, 200),     # wide: the vertical shifts in CTAs of their own
    (1, 18, 48, 96, 24),     # tap by tap, one row tile
    (1, 5, 16, 200, 64),     # tap by tap, two row tiles
    (3, 19, 40, 40, 128),    # many channels, width no multiple of 16
    (40, 24, 32, 32, 32),    # more tiles than CTAs: buffers reused
    (1, 13, 24, 136, 48),    # with dZt: the gathered GEMM
])
def test_weight_gradient_tile_edges(nb, H, W, Cin, Cout):
    """Both weight-gradient calls (dZ transposed and as it is) at the edges of their
    tiles against an FP64 sum over the same BF16 values; FP32 accumulation within
    2e-6 of the sum of magnitudes; the first call adds to what dW held, the second
    overwrites it."""
    gen = torch.Generator("cuda").manual_seed(nb * 100 + H + Cin)
    P = nb * H * W
    x = torch.randn(nb, H, W, Cin, generator=gen, device="cuda").bfloat16()
    dz = torch.randn(P, Cout, generator=gen, device="cuda").bfloat16()

    def ref(a, d):
        ap = torch.nn.functional.pad(a.double(), (0, 0, 1, 1, 1, 1))
        return torch.stack([d.double().T @ ap[:, i:i + H, j:j + W].reshape(P, Cin)
                            for i in range(3) for j in range(3)], 1).view(Cout, 9 * Cin)
    want, mag = ref(x, dz), ref(x.abs(), dz.abs())
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    dw = torch.full((Cout, 9 * Cin), 7.0, device="cuda")
    _abi.prior_call("gevo_conv3x3_wgrad_nhwc", nb, H, W, Cin, x, Cout, dz, dw, ws)
    assert ((dw.double() - 7.0 - want).abs() <= 2e-6 * (mag + 7.0)).all()
    if P % 8 == 0:
        dw.fill_(7.0)
        _abi.prior_call("gevo_conv3x3_wgrad", nb, H, W, Cin, x, Cout, dz.T.contiguous(), dw, ws)
        assert ((dw.double() - want).abs() <= 2e-6 * mag + 1e-30).all()
    assert _abi.gevo_last_error(ws) == 0


def test_weight_gradient_refusals():
    x = torch.zeros(64, 16, device="cuda").bfloat16()
    dw = torch.zeros(16 * 9 * 16 + 1, device="cuda")
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    for Cin, Cout, out in ((12, 16, dw), (16, 12, dw), (264, 16, dw), (16, 264, dw), (16, 16, dw[1:])):
        with pytest.raises(_abi.GevoError):
            _abi.prior_call("gevo_conv3x3_wgrad_nhwc", 1, 8, 8, Cin, x, Cout, x, out, ws)
