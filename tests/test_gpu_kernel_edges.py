"""Kernels and launch rules at the sizes where they change path: remainders of tiles,
vector widths, view counts and unit sizes, against the FP64 oracle, the bit-exact sort
reference or the general path of the same call."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from gpu_helpers import upload_records  # noqa: E402
from oracle import costvol  # noqa: E402
from paper_2409_09295_gb300 import _abi, raster, scenes  # noqa: E402
from paper_2409_09295_gb300.mapping import DEFAULT_ADAM  # noqa: E402


# ---- default launch shapes ----------------------------------------------------------
@pytest.mark.parametrize("sizes", [[(65, 33)], [(640, 480)], [(640, 480)] * 2,
                                   [(640, 480), (1200, 680)], [(1200, 680)] * 3])
def test_default_launch_shapes_give_the_same_results(sizes):
    n = 3000
    scene = scenes.room_scene(n, 5, sh_degree=1)
    cams = [scenes.camera(*p, 0.8 * w, 0.8 * w, w / 2, h / 2, w, h)
            for p, (w, h) in zip(scenes.circle_poses(len(sizes), 2.0, seed=3), sizes)]
    g, camt = raster.gaussians_to_device(scene), raster.camera_tensor(cams, "cuda")
    res = []
    for tuning in (None, dict(raster.DEFAULT_TUNING)):
        p = raster.Pipeline(n, sizes, 1 << 20, colour="sh", sh_degree=1, tuning=tuning)
        p.forward(g, camt)
        gen = torch.Generator().manual_seed(1)
        up = [torch.randn(t.shape, generator=gen).cuda() for t in (p.rgb, p.depth, p.T_final)]
        grads = []
        for dT in (None, up[2]):
            p.render_bwd(up[0], up[1], dT)
            grads += [t.clone() for t in p.grad2d.values()]
        torch.cuda.synchronize()
        res.append(([p.rgb, p.depth, p.T_final, p.n_contrib], grads))
    for a, b in zip(res[0][0], res[1][0]):
        assert torch.equal(a, b)
    for a, b in zip(res[0][1], res[1][1]):
        # the walks add the same terms in another order: a few hundred binary32 terms a row
        assert float((a - b).norm()) <= 2e-5 * float(b.norm())


# ---- plain initialisation -------------------------------------------------------------
def _keyframes(nk, H, W, seed):
    r = np.random.default_rng(seed)
    cams = np.zeros((nk, 16))
    cams[:, [0, 4, 8]] = 1.0
    cams[:, 9] = -0.05 * (np.arange(nk) - nk / 2)
    cams[:, 12:16] = [0.8 * W, 0.8 * W, W / 2, H / 2]
    return r.uniform(size=(nk, 3, H, W)).astype(np.float32), cams.astype(np.float32)


@pytest.mark.parametrize("H,W,nk,nd", [(36, 44, 3, 37), (8, 8, 2, 2), (20, 132, 4, 64),
                                       (12, 16, 66, 33)])
def test_cost_volume_and_winner_at_odd_sizes(H, W, nk, nd):
    rgb, cams = _keyframes(nk, H, W, nd)
    h, w, ref, d0, d1 = H // 4, W // 4, nk // 2, 0.5, 8.0
    grey = torch.zeros(nk, h, w, device="cuda")
    vol = torch.zeros(h * w * nd, device="cuda")
    dep = torch.zeros(H, W, device="cuda")
    rg = torch.from_numpy(rgb).cuda()
    call = lambda: _abi.prior_call("gevo_cost_volume", nk, ref, H, W, rg,  # noqa: E731
                                   torch.from_numpy(cams).cuda(), nd, d0, d1, grey, vol, dep)

    def winner(V):   # the first of the lowest; nothing is lower than a NaN in first place
        best = np.zeros(V.shape[:2], int)
        for k in range(1, nd):
            best = np.where(V[..., k] < np.take_along_axis(V, best[..., None], -1)[..., 0], k, best)
        return d0 + (d1 - d0) * best / (nd - 1)

    call()
    V, frag = costvol.cost_volume(rgb.astype(np.float64), cams.astype(np.float64), ref, nd, d0, d1)
    Vg = vol.cpu().numpy().reshape(h, w, nd)
    # a random image's slope is up to 1 a pixel: positions of binary32 rays are good to
    # some 1e-6 of the width
    np.testing.assert_allclose(Vg[~frag], V[~frag], atol=1e-6 * (20 + W), rtol=0)
    np.testing.assert_allclose(dep.cpu().numpy()[::4, ::4], winner(Vg), rtol=1e-6)
    rg[ref, :, : H // 2, : W // 2] = float("nan")     # a source pixel without a value
    rg[(ref + 1) % nk, :, H // 2:, W // 2:] = float("nan")
    call()
    Vg = vol.cpu().numpy().reshape(h, w, nd)
    np.testing.assert_allclose(dep.cpu().numpy(), np.kron(winner(Vg), np.ones((4, 4))), rtol=1e-6)
