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


# ---- mapping update ---------------------------------------------------------------------
@pytest.mark.parametrize("K,listed", [(1, False), (4, True), (9, False), (9, True), (16, False)])
def test_map_step_on_buffers_off_the_vector_alignment(K, listed):
    n = 1003
    gen = torch.Generator().manual_seed(K)
    shapes = dict(means=(n, 3), log_scales=(n, 3), quats=(n, 4), logit_opacities=(n,),
                  colours=(n, K, 3))
    raw = {k: torch.randn(s, generator=gen) for k, s in shapes.items()}
    gr = {k: torch.randn(s, generator=gen) for k, s in
          dict(means=(n, 3), scales=(n, 3), quats=(n, 4), opacities=(n,)).items()}
    gr["rgb" if K == 1 else "sh"] = torch.randn((n, 3) if K == 1 else (n, K, 3), generator=gen)
    rows = cnt = None
    if listed:
        rows = torch.arange(0, n, 3, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(_abi.active_count_words(n), dtype=torch.int32, device="cuda")
        cnt[0] = rows.numel()
    got = []
    for off in (0, 1):
        def put(t, z=False):
            b = torch.zeros(t.numel() + off, device="cuda")[off:].view(t.shape)
            return b if z else b.copy_(t)
        dev = {k: put(t) for k, t in raw.items()}
        m, v = ({k: put(t, True) for k, t in raw.items()} for _ in range(2))
        sc, op, iso = put(raw["means"], True), put(raw["logit_opacities"], True), torch.zeros(1, device="cuda")
        for step in (1, 2):
            _abi.gevo_map_step(n, K, dev, {k: put(t) for k, t in gr.items()}, m, v,
                               dict(DEFAULT_ADAM, lambda_iso=2.0), step, rows, cnt, sc, op, iso)
        torch.cuda.synchronize()
        got.append([*dev.values(), *m.values(), *v.values(), sc, op])
    for a, b in zip(*got):
        assert torch.equal(a, b)


# ---- sort: unit and segment sizes --------------------------------------------------------
@pytest.mark.parametrize("sizes,n,sigma", [([(16, 16)], 5000, 3.0),          # one tile
                                           ([(320, 240)], 140000, 2.0),      # 273 segments
                                           ([(640, 480)], 20000, 40.0),      # units of 2048
                                           ([(64, 48), (640, 480)] * 9, 3000, 12.0)])
@pytest.mark.parametrize("slack", [0, 100000])
def test_bin_sort_unit_and_segment_sizes(sizes, n, sigma, slack):
    rec = scenes.random_records(sizes, n, seed=len(sizes) + n, sigma_px=(0.5, sigma))
    ref = oracle.bin_f32(sizes, rec["xy"], rec["radius"], rec["depth"])
    D = ref["n_dup"]
    pipe = raster.Pipeline(n, sizes, D + slack, keep_keys=True)
    upload_records(pipe, rec)
    pipe.bin_sort()
    torch.cuda.synchronize()
    assert pipe.last_error() == 0 and int(pipe.n_dup.item()) == D
    np.testing.assert_array_equal(pipe.ranges.cpu().numpy().view(np.uint32), ref["ranges"])
    np.testing.assert_array_equal(pipe.keys[:D].cpu().numpy().view(np.uint64), ref["keys"])
    np.testing.assert_array_equal(pipe.vals[:D].cpu().numpy().view(np.uint32), ref["vals"])


# ---- projection backward: view counts of the pose sums and of the coefficient reads -------
@pytest.mark.parametrize("deg", [None, 0, 1, 2, 3])
@pytest.mark.parametrize("V,n", [(2, 1000), (3, 129), (5, 700), (17, 333)])
def test_projection_backward_of_views_is_the_sum_of_its_views(deg, V, n):
    scene = scenes.room_scene(n, 7, sh_degree=deg)
    cams = [scenes.camera(*p, 200.0, 200.0, 100.0, 75.0, 200, 150)
            for p in scenes.circle_poses(V, 2.0, seed=9)]
    g = raster.gaussians_to_device(scene)
    kw = dict(colour="rgb" if deg is None else "sh", sh_degree=deg or 0)
    gen = torch.Generator().manual_seed(V)

    def run(cs, rows):
        p = raster.Pipeline(n, [(200, 150)] * len(cs), 1 << 16, **kw)
        camt = raster.camera_tensor(cs, "cuda")
        p.project(g, camt)
        for k, t in p.grad2d.items():
            t.copy_(rows[k])
        p.project_bwd(g, camt)
        torch.cuda.synchronize()
        return {k: t.double() for k, t in p.grads.items()}, p.dxi.double()

    widths = dict(xy=2, conic_opacity=4, rgb_depth=4)
    rows = {k: 1e-2 * torch.randn(V * n, w, generator=gen) for k, w in widths.items()}
    joint, dxi = run(cams, rows)
    parts = [run([c], {k: t[v * n:(v + 1) * n] for k, t in rows.items()}) for v, c in enumerate(cams)]
    for k, t in joint.items():
        want = sum(p[0][k] for p in parts)
        # up to V binary32 terms a value, of either sign
        assert float((t - want).norm()) <= 1e-5 * float(want.norm()), k
    for v, p in enumerate(parts):
        # up to n terms of either sign a sum
        assert float((dxi[v] - p[1][0]).norm()) <= 3e-5 * float(p[1].norm())
