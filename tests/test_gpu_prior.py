"""The BF16 tensor-core U-Net (learned depth prior) against the FP64 oracle on
the same BF16 weights and inputs, the oracle storing activations and masked
gradients in BF16 at the same points (each layer computed in double).  What
remains is binary32 accumulation (K * 2^-24) and the rare BF16 rounding that
binary32 and double decide differently (one BF16 ulp, 2^-8), which then
propagates down the backward chain (up to 14 layers to the first one).
A rounding decides differently where the binary32 accumulation error, about
K 2^-24 ~ 7e-5 relative at K = 1152, straddles a BF16 rounding boundary: for
a fraction of about 7e-5 / 2^-8 ~ 2% of a layer's activations, each then off
by one BF16 ulp; over 14 layers that is a relative L2 error of about
2^-8 sqrt(14 x 0.02) ~ 2e-3 to be expected.  Bound: forward within twice that, 4e-3.
Gradients: how much BF16 storage moves a weight gradient depends on how much
its sum cancels (the first layer's, over centred inputs of both signs, moves
by about 17% between storing and not storing activations in BF16, the last
layers' by under 1%).  The two sides store at the same points and differ only
in the ~2% of roundings decided differently, so each gradient tensor must lie
within half of the oracle's own storage effect on it (the relative L2 error
and 1 - cosine between the oracle storing and not storing in BF16), plus 5e-3
relative L2 and 5e-4 in cosine."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import unet as ounet  # noqa: E402
from paper_2409_09295_gb300 import _abi  # noqa: E402
from paper_2409_09295_gb300.prior import DepthUNet  # noqa: E402


def _bf(x):
    return torch.from_numpy(np.ascontiguousarray(x, np.float32)).bfloat16().float().numpy().astype(np.float64)


def _case(nb, H, W, chans, seed):
    net = DepthUNet(nb, H, W, chans, seed=seed)
    rs = np.random.default_rng(seed + 1)
    rgb = rs.uniform(size=(nb, 3, H, W)).astype(np.float32)
    target = rs.normal(1.0, 0.3, size=nb * H * W).astype(np.float32)
    weight = (rs.uniform(size=nb * H * W) > 0.1).astype(np.float32)
    # oracle parameters: the GPU's BF16 weights, FP32 biases / head
    params = {}
    for name, lay in net.layers.items():
        w = lay["W16"].float().cpu().numpy().astype(np.float64).reshape(lay["cout"], 9, lay["cin"])
        params[name] = (w, lay["b32"].cpu().numpy().astype(np.float64))
    params["head"] = (net.head_w.cpu().numpy().astype(np.float64), net.head_b.cpu().numpy().astype(np.float64))
    x = np.zeros((nb, H, W, 8))
    x[..., :3] = _bf(rgb.transpose(0, 2, 3, 1) - 0.5)   # the network input: centred RGB
    return net, rgb, target, weight, params, x


@pytest.mark.parametrize("nb,H,W,chans", [(2, 16, 16, (8, 16)), (2, 48, 64, (16, 32, 64, 128))])
def test_prior_forward_and_gradients_match_oracle(nb, H, W, chans):
    net, rgb, target, weight, params, x = _case(nb, H, W, chans, seed=11)
    t_rgb = torch.from_numpy(rgb).cuda()
    pred = net.forward(t_rgb).cpu().numpy().astype(np.float64)
    ref, cache = ounet.forward(params, x, chans, store_bf16=True)
    rel = np.linalg.norm(pred - ref) / np.linalg.norm(ref)
    assert rel <= 4e-3, rel
    # pixels whose prediction lies within 0.05 of the target could take the L1
    # sign either way on the two sides: weight 0 there on both sides (decided
    # from the oracle's prediction), then each side uses its own loss gradient
    weight = (weight * (np.abs(ref.reshape(-1) - target) > 0.05)).astype(np.float32)
    assert weight.mean() > 0.8
    net.depth_loss(torch.from_numpy(target).cuda(), torch.from_numpy(weight).cuda())
    net.backward()
    torch.cuda.synchronize()
    _, dpred = ounet.loss_l1(ref.reshape(-1), target.astype(np.float64), weight.astype(np.float64))
    np.testing.assert_array_equal(np.sign(net.dpred.cpu().numpy()), np.sign(dpred))
    g = ounet.backward(params, cache, dpred.reshape(ref.shape), chans, store_bf16=True)
    # the oracle's own storage effect: the same pass without BF16 storage
    _, cache_d = ounet.forward(params, x, chans, store_bf16=False)
    g_d = ounet.backward(params, cache_d, dpred.reshape(ref.shape), chans, store_bf16=False)

    def rel_cos(a, b):
        return (np.linalg.norm(a - b) / (np.linalg.norm(b) + 1e-300),
                a @ b / (np.linalg.norm(a) * np.linalg.norm(b) + 1e-300))
    for name, lay in net.layers.items():
        for i, (got, what) in enumerate(((lay["dW"].cpu().numpy(), "W"), (lay["db"].cpu().numpy(), "b"))):
            got = got.astype(np.float64).reshape(-1)
            want = g[name][i].reshape(-1)
            rel, cos = rel_cos(got, want)
            rel_s, cos_s = rel_cos(want, g_d[name][i].reshape(-1))
            assert rel <= 0.5 * rel_s + 5e-3, (name, what, rel, rel_s)
            assert 1 - cos <= 0.5 * (1 - cos_s) + 5e-4, (name, what, cos, cos_s)
    gw = net.head_state[0].cpu().numpy()
    assert np.dot(gw, g["head"][0]) / (np.linalg.norm(gw) * np.linalg.norm(g["head"][0])) >= 0.9995
    assert _abi.gevo_last_error(net.ws) == 0


def test_prior_training_reduces_loss():
    nb, H, W = 4, 32, 32
    net = DepthUNet(nb, H, W, (16, 32, 64), seed=3)
    rs = np.random.default_rng(5)
    # a learnable synthetic mapping: log-depth = 1 + brightness of the image
    rgb = rs.uniform(size=(nb, 3, H, W)).astype(np.float32)
    target = (1.0 + rgb.mean(axis=1)).reshape(-1).astype(np.float32)
    t_rgb = torch.from_numpy(rgb).cuda()
    t_tar = torch.from_numpy(target).cuda()
    t_w = torch.ones_like(t_tar)
    losses = [float(net.train_step(t_rgb, t_tar, t_w, lr=3e-3).item()) for _ in range(60)]
    assert losses[-1] < 0.5 * losses[0], losses[::10]


# ---- a ReLU's gradient applied by the pass that makes its dY -----------------------
# Each fused call against the two it stands for: the same FP32 dY, mask and rounding,
# so dZ is equal bit for bit; db sums the same FP32 values in another order, held to
# P 2^-24 (the worst growth of an FP32 sum) times the sum of magnitudes.
def _masked(P, C, dY, lddy, Y, ldy):
    dZ = torch.zeros(P, C, dtype=torch.bfloat16, device="cuda")
    db = torch.zeros(C, device="cuda")
    _abi.prior_call("gevo_relu_bwd", P, C, dY, lddy, Y, ldy, dZ, None, db)
    return dZ, dZ.float().abs().sum(0)


def _db_exact(dY, Y):
    z = torch.where(Y.float() > 0, dY.double(), torch.zeros((), dtype=torch.float64, device="cuda"))
    return z.sum(0), z.abs().sum(0)


def _check(P, dZ, want, db, ref, mag):
    assert torch.equal(dZ.view(torch.int16), want.view(torch.int16))
    assert ((db.double() - 3.0 - ref).abs() <= (P * 2.0 ** -24) * mag + 1e-5).all()


@pytest.mark.parametrize("nb,H,W,Cin,Cout,pad", [(1, 16, 32, 16, 16, 0), (2, 17, 33, 32, 48, 8),
                                                 (1, 9, 9, 128, 128, 0), (3, 31, 8, 8, 24, 0),
                                                 (24, 48, 40, 16, 16, 32), (1, 20, 20, 192, 64, 0)])
def test_data_gradient_with_relu(nb, H, W, Cin, Cout, pad):
    g = torch.Generator("cuda").manual_seed(H * W + Cin)
    P, ldy = nb * H * W, Cout + pad
    X = torch.randn(P, Cin, generator=g, device="cuda").bfloat16()
    Wt = (0.2 * torch.randn(Cout, 9 * Cin, generator=g, device="cuda")).bfloat16()
    Y = torch.randn(P, ldy, generator=g, device="cuda").bfloat16()
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    dY = torch.zeros(P, Cout, device="cuda")
    _abi.prior_call("gevo_conv3x3", nb, H, W, Cin, X, Cout, Wt, None, dY, Cout, 0, 0, 0.0, ws)
    want, _ = _masked(P, Cout, dY, Cout, Y, ldy)
    dZ = torch.zeros(P, Cout, dtype=torch.bfloat16, device="cuda")
    db = torch.full((Cout,), 3.0, device="cuda")
    _abi.prior_call("gevo_conv3x3_relu_bwd", nb, H, W, Cin, X, Cout, Wt, Y, ldy, dZ, db, ws)
    assert _abi.gevo_last_error(ws) == 0
    _check(P, dZ, want, db, *_db_exact(dY, Y[:, :Cout]))


@pytest.mark.parametrize("nb,H,W,C,ldx,ldds", [(1, 2, 2, 8, 8, 8), (2, 16, 24, 16, 48, 48),
                                               (3, 10, 14, 40, 40, 44), (2, 30, 40, 128, 128, 128)])
def test_pool_gradient_with_relu(nb, H, W, C, ldx, ldds):
    g = torch.Generator("cuda").manual_seed(H * W + C)
    P = nb * H * W
    X = torch.relu(torch.randn(P, ldx, generator=g, device="cuda")).bfloat16()   # ties at 0
    dY = torch.randn(P // 4, C, generator=g, device="cuda")
    dS = torch.randn(P, ldds, generator=g, device="cuda")
    both = dS.clone()
    _abi.prior_call("gevo_maxpool2_bwd", nb, H, W, C, X, ldx, dY, both, ldds, 1.0)
    want, _ = _masked(P, C, both, ldds, X, ldx)
    dZ = torch.zeros(P, C, dtype=torch.bfloat16, device="cuda")
    db = torch.full((C,), 3.0, device="cuda")
    _abi.prior_call("gevo_maxpool2_relu_bwd", nb, H, W, C, X, ldx, dY, dS, ldds, dZ, db)
    _check(P, dZ, want, db, *_db_exact(both[:, :C], X[:, :C]))
    # and the pool itself, 8 channels a step, against torch
    Yp = torch.zeros(P // 4, C, dtype=torch.bfloat16, device="cuda")
    _abi.prior_call("gevo_maxpool2", nb, H, W, C, X, ldx, Yp)
    ref = torch.nn.functional.max_pool2d(X[:, :C].float().view(nb, H, W, C).permute(0, 3, 1, 2), 2)
    assert torch.equal(Yp.float().view(nb, H // 2, W // 2, C), ref.permute(0, 2, 3, 1))


@pytest.mark.parametrize("nb,h,w,C,lddu", [(1, 1, 1, 8, 8), (2, 9, 11, 32, 48), (1, 15, 20, 56, 60)])
def test_upsample_gradient_with_relu(nb, h, w, C, lddu):
    g = torch.Generator("cuda").manual_seed(h * w + C)
    P = nb * h * w
    dU = torch.randn(4 * P, lddu, generator=g, device="cuda")
    Y = torch.randn(P, C, generator=g, device="cuda").bfloat16()
    dY = torch.zeros(P, C, device="cuda")
    _abi.prior_call("gevo_upsample2_bwd", nb, h, w, C, dU, lddu, dY)
    want, _ = _masked(P, C, dY, C, Y, C)
    dZ = torch.zeros(P, C, dtype=torch.bfloat16, device="cuda")
    db = torch.full((C,), 3.0, device="cuda")
    _abi.prior_call("gevo_upsample2_relu_bwd", nb, h, w, C, dU, lddu, Y, dZ, db)
    _check(P, dZ, want, db, *_db_exact(dY, Y))


@pytest.mark.parametrize("P,C", [(1, 8), (777, 16), (100_000, 16)])
def test_head_gradient_with_relu(P, C):
    g = torch.Generator("cuda").manual_seed(P + C)
    X = torch.randn(P, C, generator=g, device="cuda").bfloat16()
    w = torch.randn(C, generator=g, device="cuda")
    dp = torch.randn(P, generator=g, device="cuda")
    dX, dw, db1 = torch.zeros(P, C, device="cuda"), torch.zeros(C, device="cuda"), torch.zeros(1, device="cuda")
    _abi.prior_call("gevo_head_bwd", P, C, X, w, dp, dX, dw, db1)
    want, _ = _masked(P, C, dX, C, X, C)
    dZ = torch.zeros(P, C, dtype=torch.bfloat16, device="cuda")
    db, dw2, db2 = torch.full((C,), 3.0, device="cuda"), torch.full((C,), 9.0, device="cuda"), torch.ones(1, device="cuda")
    _abi.prior_call("gevo_head_relu_bwd", P, C, X, w, dp, dZ, db, dw2, db2)
    _check(P, dZ, want, db, *_db_exact(dX, X))
    tol = P * 2.0 ** -24
    assert ((dw2 - dw).abs() <= 2 * tol * (dp.abs()[:, None] * X.float().abs()).sum(0) + 1e-6).all()
    assert (db2 - db1).abs() <= 2 * tol * dp.abs().sum() + 1e-6
    # the head itself: FP32 products summed in channel order, C 2^-24 of the magnitudes
    pred = torch.zeros(P, device="cuda")
    _abi.prior_call("gevo_head_fwd", P, C, X, w, db1, pred)
    ref = X.double() @ w.double() + db1.double()
    mag = X.double().abs() @ w.double().abs() + db1.double().abs()
    assert ((pred.double() - ref).abs() <= (C + 1) * 2.0 ** -23 * mag).all()


def test_batched_adam_and_flip_match_the_single_calls():
    g = torch.Generator("cuda").manual_seed(9)
    shapes = [(16, 8), (1, 24), (40, 16), (128, 64)]
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    one = [dict(p=r(co, 9 * ci), g=r(co, 9 * ci), m=r(co, 9 * ci), v=r(co, 9 * ci).abs(),
                h=torch.zeros(co, 9 * ci, dtype=torch.bfloat16, device="cuda"),
                f=torch.zeros(ci, 9 * co, dtype=torch.bfloat16, device="cuda")) for co, ci in shapes]
    many = [{k: t.clone() for k, t in d.items()} for d in one]
    for d, (co, ci) in zip(one, shapes):
        _abi.prior_call("gevo_adam", d["p"].numel(), d["p"], d["g"], d["m"], d["v"], d["h"], 1e-2, 0.9,
                        0.999, 1e-8, 3)
        _abi.prior_call("gevo_flip3x3", co, ci, d["h"], d["f"])
    import ctypes
    n = len(many)
    arr = lambda k: _abi.pointer_array([d[k] for d in many])  # noqa: E731
    _abi.prior_call("gevo_adam_batch", n, (ctypes.c_int64 * n)(*[d["p"].numel() for d in many]), arr("p"),
                    arr("g"), arr("m"), arr("v"), arr("h"), 1e-2, 0.9, 0.999, 1e-8, 3)
    _abi.prior_call("gevo_flip3x3_batch", n, (ctypes.c_int32 * n)(*[s[0] for s in shapes]),
                    (ctypes.c_int32 * n)(*[s[1] for s in shapes]), arr("h"), arr("f"))
    for a, b in zip(one, many):
        for k in a:
            assert torch.equal(a[k], b[k]), k
