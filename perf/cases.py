"""The work a program has this framework do, as measured cases.

Each case goes through a public entry point: `batch.BatchedReplay` (a captured
forward + L1 + backward step), `batch.HostStep` (the same from host memory),
`raster.Pipeline` (single stages), `raster.rasterize` (autograd), the map
optimisation step, the depth prior (training, inference, one layer) and the plain
initialisation (cost volume + belief propagation).  Scenes follow
`scenes.py`'s distributions, drawn on the GPU; targets are smooth random images
with noise, as a camera's differ from a render everywhere.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2409_09295_gb300 import _abi, batch, prior, raster, scenes

DEV = "cuda"
CHANS = (16, 32, 64, 128)      # the prior's levels
ADAM = dict(lr_means=1.6e-4, lr_log_scales=5e-3, lr_quats=1e-3, lr_logit_opacities=5e-2,
            lr_colour_dc=2.5e-3, lr_colour_rest=1.25e-4, beta1=0.9, beta2=0.999, eps=1e-15,
            lambda_iso=10.0)
ADAM_STEP = 50                 # moments as after this many steps
BP = dict(s=0.01, tau=0.1, iters=10, d0=0.25, d1=25.0)
# list entries a pixel examines, and blends, on average (counted with
# BatchedReplay.eval_counts on these scenes at 20k in the box, 500k in the room)
EVALS = {"box": (258.0, 41.0), "room": (205.0, 75.0)}


def listed():
    return [
        # tracking one frame against a small local map: plain RGB colours (the
        # paper switches SH off), pose gradient, a quarter-VGA image
        dict(name="track_20k_rgb_320x240", kind="replay", scene="box", n=20_000, sh=-1, views=1,
             small=0, W=320, H=240, f=300.0, depth=False),
        # the largest map and image: one Replica-sized frame, SH 3, pose gradient
        dict(name="track_1m_sh3_1200x680", kind="replay", scene="room", n=1_000_000, sh=3,
             views=1, small=0, W=1200, H=680, f=600.0, depth=False),
        # the benchmark: batched keyframe replay of uneven resolutions with
        # colour and depth terms (the window and the rendered past keyframes)
        dict(name="keyframes_500k_sh3_16view", kind="replay", scene="room", n=500_000, sh=3,
             views=16, small=4, W=640, H=480, f=525.0, depth=True),
        # rendering past keyframes instead of storing them (forward only, eager),
        # image sizes that leave partial tiles
        dict(name="render_300k_sh2_2view_613x467", kind="render", scene="room", n=300_001, sh=2,
             views=2, small=0, W=613, H=467, f=510.0),
        # a torch program differentiating through four small views (E_pc): odd
        # sizes, SH 1, upstream gradients on colour, depth and transmittance
        dict(name="autograd_60k_sh1_4view_325x243", kind="autograd", scene="room", n=60_003, sh=1,
             views=4, small=0, W=325, H=243, f=270.0),
        # one frame end to end for a caller whose map and images live in host
        # memory (VGA, SH 3, colour and depth targets)
        dict(name="host_200k_sh3_640x480", kind="host", scene="room", n=200_000, sh=3, views=1,
             small=0, W=640, H=480, f=525.0, depth=True),
        # an iteration of the global stage on its active set: the forward that
        # records the walk's start, L1, masked reverse walk and projection backward
        dict(name="active_250k_sh3_4view_640x480", kind="active", scene="room", n=250_000, sh=3,
             views=4, small=0, W=640, H=480, f=525.0, share=0.15),
        # the optimiser step of that stage: Adam and the isotropic loss over the
        # active rows of a map
        dict(name="map_step_500k_sh3_active", kind="map_step", n=500_000, sh=3, share=0.15),
        # training the depth prior: one batch of quarter-VGA renders
        dict(name="prior_train_32x320x240", kind="prior_train", nb=32, W=320, H=240),
        # proposing depths for one new keyframe
        dict(name="prior_infer_1x640x480", kind="prior_infer", nb=1, W=640, H=480),
        # one decoder layer of the prior, forward and backward
        dict(name="prior_layer_16x160x120_96to32", kind="prior_layer", nb=16, W=160, H=120,
             cin=96, cout=32),
        # plain initialisation of a new region: cost volume over eight VGA
        # keyframes, belief propagation
        dict(name="plain_init_8x640x480", kind="init", nk=8, W=640, H=480, nd=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["replay", "replay", "render", "autograd", "host", "active", "map_step",
                       "prior_train", "prior_infer", "prior_layer", "init"])
    if kind in ("replay", "render", "autograd", "host", "active"):
        views = {"replay": rng.choice([1, 1, 2, 4, 8, 12]), "render": rng.choice([1, 2, 4]),
                 "autograd": rng.choice([1, 2, 4]), "host": rng.choice([1, 2, 4]),
                 "active": rng.choice([2, 4, 8])}[kind]
        top = 1_000_000 if views == 1 else 400_000
        n = _log(rng, 10_000, top // 4 if kind == "autograd" else top)
        W = _log(rng, 300, 1200 if views == 1 else 640)
        H = int(W * rng.uniform(0.55, 0.8))
        room = n > 60_000 or rng.random() < 0.5
        c = dict(kind=kind, scene="room" if room else "box", n=n, sh=rng.choice([-1, 0, 1, 2, 3, 3]),
                 views=views, small=views // 4 if kind == "replay" else 0, W=W, H=H,
                 f=round(W * rng.uniform(0.5, 0.95), 1))
        if kind in ("replay", "host"):
            c["depth"] = rng.random() < 0.5
        if kind == "host":                     # its gradient read-back is laid out for SH maps
            c["sh"] = max(c["sh"], 0)
        if kind == "active":
            c["share"] = round(rng.uniform(0.02, 0.2), 3)
        return c
    if kind == "map_step":
        return dict(kind=kind, n=_log(rng, 10_000, 1_000_000), sh=rng.choice([-1, 0, 1, 2, 3, 3]),
                    share=rng.choice([1.0, round(rng.uniform(0.02, 0.2), 3)]))
    if kind in ("prior_train", "prior_infer"):
        W = 16 * _log(rng, 8, 20 if kind == "prior_train" else 75)
        return dict(kind=kind, nb=2 * _log(rng, 1, 16) if kind == "prior_train" else 1, W=W,
                    H=16 * int(W * rng.uniform(0.55, 0.8) / 16))
    if kind == "prior_layer":
        return dict(kind=kind, nb=_log(rng, 1, 16), W=8 * _log(rng, 5, 40), H=_log(rng, 30, 240),
                    cin=8 * _log(rng, 1, 24), cout=8 * _log(rng, 1, 16))
    W = 4 * _log(rng, 40, 200)
    return dict(kind="init", nk=rng.randint(2, 8), W=W, H=4 * int(W * rng.uniform(0.55, 0.8) / 4),
                nd=rng.choice([32, 48, 64]))


# ---- inputs ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(DEV)
    g.manual_seed(1000 + int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _gaussians(case, g):
    n, sh = case["n"], case["sh"]
    lo, hi = ((scenes.ROOM_LO, scenes.ROOM_HI) if case.get("scene", "room") == "room"
              else ((-2.0, -1.5, 2.0), (2.0, 1.5, 8.0)))
    lo = torch.tensor([float(x) for x in lo], device=DEV)
    hi = torch.tensor([float(x) for x in hi], device=DEV)
    q = _randn(g, n, 4)
    out = dict(means=lo + (hi - lo) * _rand(g, n, 3),
               scales=torch.exp(math.log(0.03) + 0.5 * _randn(g, n, 3)),
               quats=q / q.norm(dim=1, keepdim=True), opacities=torch.sigmoid(_randn(g, n)),
               sh_degree=max(sh, 0))
    if sh < 0:
        out["rgb"] = _rand(g, n, 3)
    else:
        out["sh"] = 0.05 * _randn(g, n, (sh + 1) ** 2, 3)
        out["sh"][:, 0] = _rand(g, n, 3)
    return out


def _cameras(case, seed):
    """Room: poses on a 2 m circle looking across the room; box: near identity."""
    V, W, H, f = case["views"], case["W"], case["H"], case["f"]
    cams = []
    if case["scene"] == "room":
        poses = scenes.circle_poses(V, 2.0, 2000 + seed)
    else:
        r = np.random.default_rng(2000 + seed)
        poses = [scenes.look_at(r.uniform(-0.2, 0.2, 3), (0.0, 0.0, 5.0)) for _ in range(V)]
    for k, (R, t) in enumerate(poses):
        h = 2 if k >= V - case["small"] else 1     # the last views at half size
        cams.append(scenes.camera(R, t, f / h, f / h, W / (2 * h), H / (2 * h), W // h, H // h))
    return cams


def _image(g, c, H, W, lo, hi, noise):
    """[c, H, W]: smooth random image in [lo, hi] plus noise."""
    low = _rand(g, 1, c, H // 32 + 2, W // 32 + 2)
    x = F.interpolate(low, size=(H, W), mode="bilinear", align_corners=True)[0]
    return lo + (hi - lo) * x + noise * _randn(g, c, H, W)


def _targets(cams, g):
    rgb = [_image(g, 3, c["H"], c["W"], 0.0, 1.0, 0.05).reshape(-1) for c in cams]
    dep = [_image(g, 1, c["H"], c["W"], 1.0, 5.0, 0.1).reshape(-1) for c in cams]
    return torch.cat(rgb).contiguous(), torch.cat(dep).contiguous()


def _raster_inputs(case, seed):
    g = _gen(seed)
    gs = _gaussians(case, g)
    cams = _cameras(case, seed)
    rgb, dep = _targets(cams, g)
    return gs, cams, rgb, dep, g


def _pixels(case):
    V, s = case["views"], case["small"]
    return (V - s) * case["W"] * case["H"] + s * (case["W"] // 2) * (case["H"] // 2)


def _active_mask(case, g):
    return _rand(g, case["n"]) < case["share"]


def _mask_words(mask):
    n = mask.numel()
    m = F.pad(mask.to(torch.int64), (0, (-n) % 32)).view(-1, 32)
    w = (m << torch.arange(32, device=DEV)).sum(1)
    return torch.where(w >= 1 << 31, w - (1 << 32), w).to(torch.int32)


def _rows(mask):
    """Row list and counts in gevo_active_set's layout."""
    n = mask.numel()
    lst = torch.zeros(max(n, 1), dtype=torch.int32, device=DEV)
    idx = mask.nonzero()[:, 0].to(torch.int32)
    lst[:idx.numel()] = idx
    cnt = torch.zeros(_abi.active_count_words(n), dtype=torch.int32, device=DEV)
    cnt[0] = idx.numel()
    return lst, cnt


def _map_inputs(case, seed):
    """Map parameters, gradients and Adam moments as in mid-optimisation."""
    g = _gen(seed)
    gs = _gaussians(case, g)
    col = gs["rgb"][:, None] if case["sh"] < 0 else gs["sh"]
    p = dict(means=gs["means"], log_scales=gs["scales"].log(), quats=gs["quats"],
             logit_opacities=torch.logit(gs["opacities"]), colours=col.contiguous())
    gr = {k: 1e-5 * _randn(g, *t.shape) for k, t in p.items()}
    m = {k: 1e-5 * _randn(g, *t.shape) for k, t in p.items()}
    v = {k: 1e-12 + 1e-10 * _rand(g, *t.shape) for k, t in p.items()}
    mask = _active_mask(case, g)
    return p, gr, m, v, mask


def _net_layers():
    L, c = len(CHANS), CHANS
    out = {}
    for i in range(L):
        out[f"enc{i}a"] = (8 if i == 0 else c[i - 1], c[i])
        out[f"enc{i}b"] = (c[i], c[i])
    for i in range(L - 2, -1, -1):
        out[f"dec{i}a"] = (c[i + 1] + c[i], c[i])
        out[f"dec{i}b"] = (c[i], c[i])
    return out


def _net_inputs(case, seed):
    """Weights (a checkpoint's), image batch, log-depth targets and their weights."""
    g = _gen(seed)
    w = {}
    for name, (cin, cout) in _net_layers().items():
        real = 3 if name == "enc0a" else cin
        W = _randn(g, cout, 9, cin) * math.sqrt(2.0 / (9 * real))
        W[:, :, real:] = 0.0
        w[name] = (W.reshape(cout, 9 * cin), 0.05 * _randn(g, cout))
    w["head"] = (_randn(g, CHANS[0]) / 4.0, torch.ones(1, device=DEV))
    nb, H, W = case["nb"], case["H"], case["W"]
    rgb = torch.stack([_image(g, 3, H, W, 0.0, 1.0, 0.05) for _ in range(nb)]).clamp(0, 1)
    target = torch.cat([_image(g, 1, H, W, 0.3, 1.7, 0.05).reshape(-1) for _ in range(nb)])
    weight = (_rand(g, nb * H * W) < 0.9).float()
    return w, rgb.contiguous(), target.contiguous(), weight


def _layer_inputs(case, seed):
    g = _gen(seed)
    nb, H, W, ci, co = (case[k] for k in ("nb", "H", "W", "cin", "cout"))
    P = nb * H * W
    return dict(X=F.relu(_randn(g, P, ci)).bfloat16(),
                Wt=(_randn(g, co, 9 * ci) * math.sqrt(2.0 / (9 * ci))).bfloat16(),
                b=0.05 * _randn(g, co), dY=1e-3 * _randn(g, P, co))


def _keyframes(case, seed):
    """nk keyframes 0.1 m apart and slightly rotated, looking at a textured plane."""
    g = _gen(seed)
    nk, H, W = case["nk"], case["H"], case["W"]
    r = np.random.default_rng(3000 + seed)
    f = 0.82 * W
    cams = np.zeros((nk, 16))
    for i in range(nk):
        a = r.normal(0, 0.02, size=3)
        th = np.linalg.norm(a)
        K = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
        cams[i, :9] = (np.eye(3) + np.sin(th) / th * K + (1 - np.cos(th)) / th ** 2 * K @ K).reshape(9)
        cams[i, 9:12] = [-0.1 * (i - nk / 2), 0.03 * np.sin(i), 0.0]
        cams[i, 12:16] = [f, f, W / 2, H / 2]
    tex = [[r.uniform(2.0, 12.0, 2), r.uniform(0, 6.28, 2)] for _ in range(9)]
    d = float(r.uniform(2.0, 5.0))
    ys, xs = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float64),
                            torch.arange(W, device=DEV, dtype=torch.float64), indexing="ij")
    ims = []
    for c in cams:
        R = torch.from_numpy(c[:9].reshape(3, 3)).to(DEV)
        o = -(R.T @ torch.from_numpy(c[9:12]).to(DEV))
        ray = torch.stack([(xs + 0.5 - c[14]) / c[12], (ys + 0.5 - c[15]) / c[13],
                           torch.ones_like(xs)], -1) @ R
        s = (d - o[2]) / ray[..., 2]
        px, py = o[0] + s * ray[..., 0], o[1] + s * ray[..., 1]
        ims.append(torch.stack([0.5 + sum(0.15 * torch.sin(tex[3 * k + j][0][0] * px + tex[3 * k + j][1][0])
                                          * torch.cos(tex[3 * k + j][0][1] * py + tex[3 * k + j][1][1])
                                          for j in range(3)) for k in range(3)]))
    rgb = torch.stack(ims).float() + 0.01 * _randn(g, nk, 3, H, W)
    return rgb.clamp(0, 1).contiguous(), torch.from_numpy(cams.astype(np.float32)).to(DEV)


# ---- what a program keeps -------------------------------------------------------------
def _pipeline(case, gs, cams):
    colour = "rgb" if "rgb" in gs else "sh"
    camt = raster.camera_tensor(cams)
    pipe = raster.Pipeline(case["n"], [(c["W"], c["H"]) for c in cams], 1 << 20, colour=colour,
                           sh_degree=gs["sh_degree"])
    D = pipe.ensure_capacity(gs, camt)
    if D * 1.3 > pipe.capacity:
        pipe.alloc_capacity(int(D * 1.3) + 1024)
    return pipe, camt


def prepare(case, seed):
    k = case["kind"]
    s = dict(case=case)
    if k in ("replay", "host"):
        gs, cams, rgb, dep, _ = _raster_inputs(case, seed)
        rep = batch.BatchedReplay(gs, cams, rgb, dep if case["depth"] else None,
                                  1.0 if case["depth"] else 0.0)
        if k == "replay":
            rep.capture()
            s["rep"] = rep
        else:
            s["host"] = batch.HostStep(rep)
            s["host"].capture()
    elif k in ("render", "autograd", "active"):
        gs, cams, rgb, dep, g = _raster_inputs(case, seed)
        s["pipe"], s["camt"] = _pipeline(case, gs, cams)
        s["g"] = gs
        if k == "autograd":
            s["leaves"] = [gs[x].requires_grad_() for x in
                           ("means", "scales", "quats", "opacities", "rgb" if "rgb" in gs else "sh")]
            s["leaves"].append(torch.zeros(case["views"], 6, device=DEV, requires_grad=True))
            P = rgb.numel() // 3
            s["up"] = [(rgb - 0.5) / (3 * P), (dep - 3.0) / P, _randn(g, P) / P]
        if k == "active":
            s["target"] = rgb
            mask = _active_mask(case, g)
            s["pipe"].alloc_active()
            s["pipe"].active.copy_(_mask_words(mask))
            lst, cnt = _rows(mask)
            s["pipe"].active_list.copy_(lst)
            s["pipe"].active_counts.copy_(cnt)
    elif k == "map_step":
        s["p"], gr, s["m"], s["v"], mask = _map_inputs(case, seed)
        s["grads"] = dict(means=gr["means"], scales=gr["log_scales"], quats=gr["quats"],
                          opacities=gr["logit_opacities"])
        s["grads"]["rgb" if case["sh"] < 0 else "sh"] = gr["colours"]
        s["rows"] = _rows(mask) if case["share"] < 1.0 else (None, None)
        s["scales"] = torch.exp(s["p"]["log_scales"])
        s["opac"] = torch.sigmoid(s["p"]["logit_opacities"])
        s["iso"] = torch.zeros(1, device=DEV)
    elif k in ("prior_train", "prior_infer"):
        w, s["rgb"], s["target"], s["weight"] = _net_inputs(case, seed)
        net = prior.DepthUNet(case["nb"], case["H"], case["W"], CHANS)
        for name, lay in net.layers.items():
            lay["W32"].copy_(w[name][0])
            lay["b32"].copy_(w[name][1])
            _abi.prior_call("gevo_to_bf16", lay["W32"].numel(), lay["W32"], lay["W16"])
            _abi.prior_call("gevo_flip3x3", lay["cout"], lay["cin"], lay["W16"], lay["Wf16"])
        net.head_w.copy_(w["head"][0])
        net.head_b.copy_(w["head"][1])
        s["net"] = net
    elif k == "prior_layer":
        s |= _layer_inputs(case, seed)
        P, ci, co = case["nb"] * case["H"] * case["W"], case["cin"], case["cout"]
        b16 = dict(dtype=torch.bfloat16, device=DEV)
        s |= dict(Wf=torch.zeros(ci, 9 * co, **b16), Y=torch.zeros(P, co, **b16),
                  dZ=torch.zeros(P, co, **b16), dZt=torch.zeros(co, P, **b16),
                  db=torch.zeros(co, device=DEV), dW=torch.zeros(co, 9 * ci, device=DEV),
                  dX=torch.zeros(P, ci, device=DEV),
                  ws=torch.zeros(256, dtype=torch.uint8, device=DEV))
        _abi.prior_call("gevo_flip3x3", co, ci, s["Wt"], s["Wf"])
    else:
        s["rgb"], s["cams"] = _keyframes(case, seed)
        nk, H, W, nd = (case[x] for x in ("nk", "H", "W", "nd"))
        h, w = H // 4, W // 4
        s |= dict(grey=torch.zeros(nk, h, w, device=DEV), vol=torch.zeros(h, w, nd, device=DEV),
                  wta=torch.zeros(H, W, device=DEV), msgs=torch.zeros(8, h, w, nd, device=DEV),
                  depth=torch.zeros(H, W, device=DEV), beliefs=torch.zeros(h, w, nd, device=DEV),
                  labels=torch.zeros(h, w, dtype=torch.int32, device=DEV))
    return s


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "replay":
        rep = s["rep"]
        rep.replay()
        p = rep.pipe
        return dict(image=p.rgb, depth=p.depth, T=p.T_final, loss=p.loss, dxi=p.dxi, **p.grads)
    if k == "host":
        s["host"].step()
        return dict(s["host"].host_out)
    if k == "render":
        p = s["pipe"]
        p.forward(s["g"], s["camt"])
        return dict(image=p.rgb, depth=p.depth, T=p.T_final, n_contrib=p.n_contrib)
    if k == "autograd":
        out = raster.rasterize(s["pipe"], *s["leaves"][:5], s["camt"], twist=s["leaves"][5])
        gr = torch.autograd.grad(out, s["leaves"], s["up"])
        return dict(out=[t.detach() for t in out], grads=list(gr))
    if k == "active":
        p, g, camt = s["pipe"], s["g"], s["camt"]
        p.project(g, camt)
        p.bin_sort()
        p.render_fwd_active()
        p.loss_l1(s["target"])
        p.render_bwd_active(p.dL_drgb, error=False, masked=True, from_state=True)
        p.project_bwd_active(g, camt)
        return dict(image=p.rgb, loss=p.loss, dxi=p.dxi, **p.grads)
    if k == "map_step":
        s["iso"].zero_()
        n, K = case["n"], s["p"]["colours"].shape[1]
        _abi.gevo_map_step(n, K, s["p"], s["grads"], s["m"], s["v"], ADAM, ADAM_STEP, *s["rows"],
                           s["scales"], s["opac"], s["iso"])
        return dict(p=s["p"], m=s["m"], v=s["v"], scales=s["scales"], opac=s["opac"], iso=s["iso"])
    if k == "prior_train":
        # a warm-up's first step (rate 0), so that every pass trains the same weights
        net = s["net"]
        net.train_step(s["rgb"], s["target"], s["weight"], lr=0.0)
        out = dict(pred=net.pred, loss=net.loss, dhead=net.head_state[0], dhead_b=net.head_state[3])
        for name, lay in net.layers.items():
            out["dW_" + name], out["db_" + name] = lay["dW"], lay["db"]
        return out
    if k == "prior_infer":
        return s["net"].forward(s["rgb"])
    if k == "prior_layer":
        nb, H, W, ci, co = (case[x] for x in ("nb", "H", "W", "cin", "cout"))
        call = _abi.prior_call
        call("gevo_conv3x3", nb, H, W, ci, s["X"], co, s["Wt"], s["b"], s["Y"], co, 1, 1, 0.0, s["ws"])
        s["db"].zero_()
        call("gevo_relu_bwd", nb * H * W, co, s["dY"], co, s["Y"], co, s["dZ"], s["dZt"], s["db"])
        call("gevo_conv3x3_wgrad", nb, H, W, ci, s["X"], co, s["dZt"], s["dW"], s["ws"])
        call("gevo_conv3x3", nb, H, W, co, s["dZ"], ci, s["Wf"], None, s["dX"], ci, 0, 0, 0.0, s["ws"])
        return dict(Y=s["Y"], db=s["db"], dW=s["dW"], dX=s["dX"])
    nk, H, W, nd = (case[x] for x in ("nk", "H", "W", "nd"))
    _abi.prior_call("gevo_cost_volume", nk, nk - 1, H, W, s["rgb"], s["cams"], nd, BP["d0"], BP["d1"],
                    s["grey"], s["vol"], s["wta"])
    _abi.prior_call("gevo_depth_bp", H // 4, W // 4, nd, s["vol"], BP["s"], BP["tau"], BP["iters"],
                    BP["d0"], BP["d1"], s["msgs"], s["depth"], s["labels"], s["beliefs"])
    return dict(volume=s["vol"], beliefs=s["beliefs"], wta=s["wta"], depth=s["depth"],
                labels=s["labels"])


# ---- the work of one pass -------------------------------------------------------------
def work(case):
    k = case["kind"]
    if k in ("replay", "render", "autograd", "host", "active"):
        n, P, V = case["n"], _pixels(case), case["views"]
        K = 1 if case["sh"] < 0 else (case["sh"] + 1) ** 2
        param = 4 * n * (11 + 3 * K)
        ev, bl = (x * P for x in EVALS[case["scene"]])
        # examined entries 12 FLOPs each way, blended ones 11 and 49; the
        # projection about 250 per view and 6 per SH coefficient
        fwd = 12 * ev + 11 * bl + n * V * 250.0
        bwd = 12 * ev + 49 * bl + n * V * 300.0
        img = 4 * P * 5                        # colour, depth, transmittance
        if k == "render":
            return dict(bytes=param + img, flops=fwd)
        share = case.get("share", 1.0)
        tgt = 4 * P * (4 if case.get("depth") else 3) if k != "autograd" else 4 * P * 5
        return dict(bytes=param * (1 + share) + img + tgt, flops=fwd + bwd)
    if k == "map_step":
        K = 1 if case["sh"] < 0 else (case["sh"] + 1) ** 2
        rows = case["n"] * case["share"]
        per = 11 + 3 * K                       # parameters of a row: p, m, v, gradient
        return dict(bytes=4 * rows * (7 * per + 4 + 1), flops=12 * rows * per)
    if k in ("prior_train", "prior_infer"):
        P = case["nb"] * case["H"] * case["W"]
        flops, nw = 0.0, 0
        for name, (cin, cout) in _net_layers().items():
            flops += 2.0 * 9 * (3 if name == "enc0a" else cin) * cout * P / 4 ** int(name[3])
            nw += 9 * cin * cout + cout
        if k == "prior_infer":
            return dict(bytes=P * (12 + 4) + 2 * nw, flops=flops)
        # every layer's output written and read again by the backward pass
        act = sum(2 * 2 * cout * P / 4 ** int(name[3]) for name, (_, cout) in _net_layers().items())
        return dict(bytes=P * (12 + 4 + 8) + act + 4 * 7 * nw, flops=3 * flops)
    if k == "prior_layer":
        P, ci, co = case["nb"] * case["H"] * case["W"], case["cin"], case["cout"]
        return dict(bytes=P * (2 * ci + 2 * co + 4 * co + 4 * ci) + 9 * ci * co * 8,
                    flops=3 * 2.0 * 9 * ci * co * P)
    nk, H, W, nd = (case[x] for x in ("nk", "H", "W", "nd"))
    q = H // 4 * (W // 4)
    return dict(bytes=12.0 * nk * H * W + 8 * H * W + 4 * q * (2 * nd + 1),
                flops=q * nd * ((nk - 1) * 30.0 + BP["iters"] * 4 * 12.0))


# ---- the same results in 64 bits -------------------------------------------------------
_SH = [0.5 * math.sqrt(1 / math.pi), math.sqrt(3 / (4 * math.pi)), 0.5 * math.sqrt(15 / math.pi),
       0.25 * math.sqrt(5 / math.pi), 0.25 * math.sqrt(15 / math.pi),
       0.25 * math.sqrt(35 / (2 * math.pi)), 0.5 * math.sqrt(105 / math.pi),
       0.25 * math.sqrt(21 / (2 * math.pi)), 0.25 * math.sqrt(7 / math.pi),
       0.25 * math.sqrt(105 / math.pi)]


def _sh_basis(d, deg):
    x, y, z = d.unbind(-1)
    Y = [torch.full_like(x, _SH[0])]
    if deg > 0:
        Y += [-_SH[1] * y, _SH[1] * z, -_SH[1] * x]
    if deg > 1:
        Y += [_SH[2] * x * y, -_SH[2] * y * z, _SH[3] * (2 * z * z - x * x - y * y), -_SH[2] * x * z,
              _SH[4] * (x * x - y * y)]
    if deg > 2:
        Y += [-_SH[5] * y * (3 * x * x - y * y), _SH[6] * x * y * z,
              -_SH[7] * y * (4 * z * z - x * x - y * y),
              _SH[8] * z * (2 * z * z - 3 * x * x - 3 * y * y),
              -_SH[7] * x * (4 * z * z - x * x - y * y), _SH[9] * z * (x * x - y * y),
              -_SH[5] * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


def _project64(p, cam, twist, W, H):
    """Records of the Gaussians visible in one view (ids, xy, conic, opacity,
    colour, depth, tile rectangle), differentiable."""
    c = cam.double()
    R0, t0 = c[:9].view(3, 3), c[9:12]
    fx, fy, cx, cy = c[12], c[13], c[14], c[15]
    a = twist[3:]
    z0 = torch.zeros_like(a[0])
    K = torch.stack([z0, -a[2], a[1], a[2], z0, -a[0], -a[1], a[0], z0]).view(3, 3)
    R, t = R0 + K @ R0, t0 + K @ t0 + twist[:3]
    with torch.no_grad():
        near = ((p["means"] @ R0.T + t0)[:, 2] > 0.2).nonzero()[:, 0]
    mu, s, q, o = (p[x][near] for x in ("means", "scales", "quats", "opacities"))
    pc = mu @ R.T + t
    z = pc[:, 2]
    lx, ly = 1.3 * 0.5 * W / fx, 1.3 * 0.5 * H / fy
    tx = torch.minimum(torch.maximum(pc[:, 0] / z, -lx), lx)
    ty = torch.minimum(torch.maximum(pc[:, 1] / z, -ly), ly)
    # a clamped ratio passes no gradient: J's third column with its camera point held
    inx, iny = (pc[:, 0] / z).abs() < lx, (pc[:, 1] / z).abs() < ly
    tx = torch.where(inx, pc[:, 0] / z, tx.detach())
    ty = torch.where(iny, pc[:, 1] / z, ty.detach())
    w, x, y, zz = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    Rq = torch.stack([1 - 2 * (y * y + zz * zz), 2 * (x * y - w * zz), 2 * (x * zz + w * y),
                      2 * (x * y + w * zz), 1 - 2 * (x * x + zz * zz), 2 * (y * zz - w * x),
                      2 * (x * zz - w * y), 2 * (y * zz + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    zero = torch.zeros_like(z)
    J = torch.stack([fx / z, zero, -fx * tx / z, zero, fy / z, -fy * ty / z], 1).view(-1, 2, 3)
    T = J @ R @ Rq * s[:, None, :]
    S = T @ T.transpose(1, 2)
    A, B, C = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    det = A * C - B * B
    xy = torch.stack([fx * pc[:, 0] / z + cx - 0.5, fy * pc[:, 1] / z + cy - 0.5], 1)
    with torch.no_grad():
        mid = 0.5 * (A + C)
        rad = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp_min(0.1))))
        nt = torch.tensor([(W + 15) // 16, (H + 15) // 16], device=DEV)
        m = xy.float().double()
        lo = torch.minimum(torch.floor((m - rad[:, None]) / 16).clamp_min(0), nt).long()
        hi = torch.minimum(torch.floor((m + rad[:, None] + 15) / 16).clamp_min(0), nt).long()
        vis = ((hi - lo).prod(1) > 0) & (det > 0)
    if "rgb" in p:
        col = p["rgb"][near[vis]]
    else:
        d = mu[vis] - (-(R.T @ t))
        Y = _sh_basis(d / d.norm(dim=1, keepdim=True), p["deg"])
        col = (torch.einsum("nk,nkc->nc", Y, p["sh"][near[vis]]) + 0.5).clamp_min(0.0)
    det = det[vis]
    conic = torch.stack([C[vis] / det, -B[vis] / det, A[vis] / det], 1)
    return near[vis], xy[vis], conic, o[vis], col, z[vis], lo[vis], hi[vis]


def _tile_lists(z, lo, hi, nx, ny):
    """Record indices in (tile, depth, id) order and each tile's start."""
    w, cnt = (hi - lo)[:, 0], (hi - lo).prod(1)
    rec = torch.repeat_interleave(torch.arange(len(cnt), device=DEV), cnt)
    k = torch.arange(len(rec), device=DEV) - torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt)
    tile = (lo[rec, 1] + k // w[rec]) * nx + lo[rec, 0] + k % w[rec]
    by_z = torch.argsort(z.float()[rec], stable=True)
    order = by_z[torch.argsort(tile[by_z], stable=True)]
    start = torch.searchsorted(tile[order], torch.arange(nx * ny + 1, device=DEV)).tolist()
    return rec[order], start


def _blend64(rec, W, H, grad_of=None):
    """Images of one view (3 + depth + T planes) and, given grad_of(planes) ->
    dL/dplanes [5, H, W], the record gradients."""
    ids, xy, conic, o, col, z, lo, hi = [t.detach() for t in rec]
    nx, ny = (W + 15) // 16, (H + 15) // 16
    order, start = _tile_lists(z, lo, hi, nx, ny)
    img = torch.zeros(5, H, W, dtype=torch.float64, device=DEV)
    img[4] = 1.0
    q4 = torch.cat([col, z[:, None]], 1)
    gxy, gcon, go, gq = (torch.zeros_like(t) for t in (xy, conic, o, q4))

    def tile(t):
        x0, y0 = t % nx * 16, t // nx * 16
        x1, y1 = min(x0 + 16, W), min(y0 + 16, H)
        L = order[start[t]:start[t + 1]]
        ys, xs = torch.meshgrid(torch.arange(y0, y1, device=DEV, dtype=torch.float64),
                                torch.arange(x0, x1, device=DEV, dtype=torch.float64), indexing="ij")
        dx = xy[L, 0] - xs.reshape(-1, 1)
        dy = xy[L, 1] - ys.reshape(-1, 1)
        a, b, c = conic[L].unbind(1)
        power = -0.5 * (a * dx * dx + c * dy * dy) - b * dx * dy
        G = torch.exp(power)
        raw = o[L] * G
        al = raw.clamp_max(0.99)
        al = torch.where((power > 0) | (al < 1 / 255), torch.zeros_like(al), al)
        after = torch.cumprod(1 - al, 1)
        al = torch.where(after < 1e-4, torch.zeros_like(al), al)   # stopped: nothing from here on
        after = torch.cumprod(1 - al, 1)
        before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
        return L, (x0, x1, y0, y1), dx, dy, G, raw, al, before, after

    todo = [t for t in range(nx * ny) if start[t + 1] > start[t]]
    for t in todo:
        L, (x0, x1, y0, y1), dx, dy, G, raw, al, before, after = tile(t)
        v = torch.cat([(al * before) @ q4[L], after[:, -1:]], 1)
        img[:, y0:y1, x0:x1] = v.T.reshape(5, y1 - y0, x1 - x0)
    if grad_of is None:
        return img, None
    g = grad_of(img)
    for t in todo:
        L, (x0, x1, y0, y1), dx, dy, G, raw, al, before, after = tile(t)
        gp = g[:, y0:y1, x0:x1].reshape(5, -1)
        wgt = al * before
        q = gp[:4].T @ q4[L].T
        wq = wgt * q
        behind = wq.sum(1, keepdim=True) - wq.cumsum(1) + (gp[4] * after[:, -1])[:, None]
        da = torch.where(al > 0, before * q - behind / (1 - al), torch.zeros_like(al))
        da = torch.where(raw > 0.99, torch.zeros_like(da), da)
        dp = da * raw
        a, b, c = conic[L].unbind(1)
        gq.index_add_(0, L, wgt.T @ gp[:4].T)
        go.index_add_(0, L, (da * G).sum(0))
        gxy.index_add_(0, L, torch.stack([-(dp * (a * dx + b * dy)).sum(0),
                                          -(dp * (c * dy + b * dx)).sum(0)], 1))
        gcon.index_add_(0, L, torch.stack([-0.5 * (dp * dx * dx).sum(0), -(dp * dx * dy).sum(0),
                                           -0.5 * (dp * dy * dy).sum(0)], 1))
    return img, (gxy, gcon, go, gq[:, :3].contiguous(), gq[:, 3].contiguous())


def _raster64(case, seed):
    k = case["kind"]
    gs, cams, rgb_t, dep_t, g = _raster_inputs(case, seed)
    if sum((-(-c["W"] // 16)) * (-(-c["H"] // 16)) for c in cams) > 3600:
        return None                            # the loop over tiles would take too long
    names = ["means", "scales", "quats", "opacities", "rgb" if "rgb" in gs else "sh"]
    p = {x: gs[x].double().requires_grad_() for x in names}
    p["deg"] = gs["sh_degree"]
    twist = torch.zeros(len(cams), 6, dtype=torch.float64, device=DEV, requires_grad=True)
    camt = torch.from_numpy(np.stack([np.concatenate(
        [np.asarray(c["R"], np.float32).reshape(9), np.asarray(c["t"], np.float32),
         np.float32([c["fx"], c["fy"], c["cx"], c["cy"]])]) for c in cams])).to(DEV)
    ups = None
    if k == "autograd":
        P = rgb_t.numel() // 3
        ups = [(rgb_t - 0.5) / (3 * P), (dep_t - 3.0) / P, _randn(g, P) / P]
    mask = _active_mask(case, g) if k == "active" else None
    imgs, losses, roots, gouts, base = [], [], [], [], 0
    for v, c in enumerate(cams):
        W, H = c["W"], c["H"]
        N = W * H
        rec = _project64(p, camt[v], twist[v], W, H)
        sl3, sl = slice(3 * base, 3 * (base + N)), slice(base, base + N)
        base += N

        def grad_of(img, sl3=sl3, sl=sl, W=W, H=H, N=N):
            out = torch.zeros_like(img)
            if ups is not None:
                out[:3] = ups[0][sl3].view(3, H, W)
                out[3], out[4] = ups[1][sl].view(H, W), ups[2][sl].view(H, W)
                return out
            e = img[:3] - rgb_t[sl3].view(3, H, W)
            loss = e.abs().mean()
            out[:3] = e.sign() / (3 * N)
            if case.get("depth"):
                e = img[3] - dep_t[sl].view(H, W)
                loss = loss + e.abs().mean()
                out[3] = e.sign() / N
            losses.append(loss)
            return out

        img, gr = _blend64(rec, W, H, None if k == "render" else grad_of)
        imgs.append(img)
        if gr is not None:
            keep = mask[rec[0]].double() if mask is not None else None
            for r, x in zip(rec[1:6], gr):
                roots.append(r)
                gouts.append(x if keep is None else x * keep.view(-1, *[1] * (x.dim() - 1)))
    rgb = torch.cat([i[:3].reshape(-1) for i in imgs])
    dep, T = (torch.cat([i[j].reshape(-1) for i in imgs]) for j in (3, 4))
    if k == "render":
        return dict(image=rgb, depth=dep, T=T, n_contrib=None)
    gr = torch.autograd.grad(roots, [p[x] for x in names] + [twist], gouts)
    if k == "autograd":
        return dict(out=[rgb, dep, T], grads=list(gr))
    out = dict(zip(names, gr[:5]), loss=torch.stack(losses), dxi=gr[5])
    if k == "active":
        return dict(out, image=rgb)
    return out if k == "host" else dict(out, image=rgb, depth=dep, T=T)


def _map64(case, seed):
    p, gr, m, v, mask = _map_inputs(case, seed)
    s0, o0 = torch.exp(p["log_scales"]), torch.sigmoid(p["logit_opacities"])
    p, gr, m, v = ({k: t.double() for k, t in d.items()} for d in (p, gr, m, v))
    rows = mask if case["share"] < 1.0 else torch.ones_like(mask)
    R = float(rows.sum())
    s, o = s0.double(), o0.double()
    d = s - s.mean(1, keepdim=True)
    iso = (ADAM["lambda_iso"] / R * d[rows].abs().sum()).reshape(1)
    gi = ADAM["lambda_iso"] / R * (d.sign() - d.sign().sum(1, keepdim=True) / 3)
    gr["log_scales"] = (gr["log_scales"] + gi) * s
    gr["logit_opacities"] = gr["logit_opacities"] * o * (1 - o)
    for k in p:
        lr = ADAM["lr_colour_dc" if k == "colours" else "lr_" + k]
        if k == "colours":
            lr = torch.full((1, p[k].shape[1], 1), ADAM["lr_colour_rest"], device=DEV, dtype=torch.float64)
            lr[:, 0] = ADAM["lr_colour_dc"]
        on = rows.view(-1, *[1] * (p[k].dim() - 1))
        m2 = ADAM["beta1"] * m[k] + (1 - ADAM["beta1"]) * gr[k]
        v2 = ADAM["beta2"] * v[k] + (1 - ADAM["beta2"]) * gr[k] ** 2
        st = lr * (m2 / (1 - ADAM["beta1"] ** ADAM_STEP)) / (
            torch.sqrt(v2 / (1 - ADAM["beta2"] ** ADAM_STEP)) + ADAM["eps"])
        p[k], m[k], v[k] = (torch.where(on, a, b) for a, b in ((p[k] - st, p[k]), (m2, m[k]), (v2, v[k])))
    return dict(p=p, m=m, v=v, iso=iso, scales=torch.where(rows[:, None], torch.exp(p["log_scales"]), s),
                opac=torch.where(rows, torch.sigmoid(p["logit_opacities"]), o))


class _Conv64(torch.autograd.Function):
    """bf16(ReLU(conv3x3 + b)) with the masked gradient in BF16 for the two
    convolutions of the backward pass (where the prior stores BF16), the sums in
    64 bits.  x NCHW, w [Cout, 9 Cin]."""

    @staticmethod
    def forward(ctx, x, w, b):
        w4 = w.view(w.shape[0], 3, 3, x.shape[1]).permute(0, 3, 1, 2).contiguous()
        y = F.relu(F.conv2d(x, w4, b, padding=1)).bfloat16().double()
        ctx.save_for_backward(x, w4, y)
        return y

    @staticmethod
    def backward(ctx, dy):
        x, w4, y = ctx.saved_tensors
        dz = torch.where(y > 0, dy, torch.zeros_like(dy))
        db = dz.sum((0, 2, 3))
        dz = dz.bfloat16().double()
        dx = F.conv_transpose2d(dz, w4, padding=1)
        xp = F.pad(x, (1, 1, 1, 1))
        H, W = y.shape[2:]
        dw = torch.stack([torch.einsum("bohw,bchw->oc", dz, xp[:, :, i:i + H, j:j + W])
                          for i in range(3) for j in range(3)], 1)
        return dx, dw.reshape(w4.shape[0], -1), db


def _net64(case, seed):
    w, rgb, target, weight = _net_inputs(case, seed)
    train, conv = case["kind"] == "prior_train", _Conv64.apply
    w16 = {k: (a.bfloat16().double() if k != "head" else a.double(), b.double()) for k, (a, b) in w.items()}
    out = None
    per = max(1, min(case["nb"], 1_000_000 // (case["H"] * case["W"])))
    preds, P = [], case["nb"] * case["H"] * case["W"]
    loss = 0.0
    for i in range(0, case["nb"], per):        # a few images at a time
        leaf = {k: [t.clone().requires_grad_(train) for t in ab] for k, ab in w16.items()}
        x = (rgb[i:i + per] - 0.5).bfloat16().double()
        x = F.pad(x, (0, 0, 0, 0, 0, 5))
        skips = []
        for lv in range(len(CHANS)):
            x = conv(conv(x, *leaf[f"enc{lv}a"]), *leaf[f"enc{lv}b"])
            if lv < len(CHANS) - 1:
                skips.append(x)
                x = F.max_pool2d(x, 2)
        for lv in range(len(CHANS) - 2, -1, -1):
            x = torch.cat([x.repeat_interleave(2, 2).repeat_interleave(2, 3), skips[lv]], 1)
            x = conv(conv(x, *leaf[f"dec{lv}a"]), *leaf[f"dec{lv}b"])
        pred = torch.einsum("bchw,c->bhw", x, leaf["head"][0]) + leaf["head"][1]
        preds.append(pred.detach().reshape(-1))
        if train:
            sl = slice(i * case["H"] * case["W"], i * case["H"] * case["W"] + pred.numel())
            l = (weight[sl].double() * (pred.reshape(-1) - target[sl].double()).abs()).sum() / P
            names = list(leaf)
            gr = torch.autograd.grad(l, [t for k in names for t in leaf[k]])
            out = list(gr) if out is None else [a + b for a, b in zip(out, gr)]
            loss = loss + l.detach()
    pred = torch.cat(preds)
    if not train:
        return pred
    res = dict(pred=pred, loss=loss.reshape(1))
    for j, k in enumerate(w16):
        if k == "head":
            res["dhead"], res["dhead_b"] = out[2 * j], out[2 * j + 1]
        else:
            res["dW_" + k], res["db_" + k] = out[2 * j], out[2 * j + 1]
    return res


def _layer64(case, seed):
    d = _layer_inputs(case, seed)
    nb, H, W, ci, co = (case[x] for x in ("nb", "H", "W", "cin", "cout"))
    x = d["X"].double().view(nb, H, W, ci).permute(0, 3, 1, 2).contiguous().requires_grad_()
    w = d["Wt"].double().requires_grad_()
    b = d["b"].double().requires_grad_()
    y = _Conv64.apply(x, w, b)
    dy = d["dY"].double().view(nb, H, W, co).permute(0, 3, 1, 2)
    dx, dw, db = torch.autograd.grad(y, [x, w, b], dy)
    flat = lambda t: t.detach().permute(0, 2, 3, 1).reshape(nb * H * W, -1)  # noqa: E731
    return dict(Y=flat(y), db=db, dW=dw, dX=flat(dx))


def _init64(case, seed):
    rgb, cams = _keyframes(case, seed)
    nk, H, W, nd = (case[x] for x in ("nk", "H", "W", "nd"))
    h, w, ref = H // 4, W // 4, nk - 1
    f64 = dict(dtype=torch.float64, device=DEV)
    grey = rgb.double().mean(1).view(nk, h, 4, w, 4).mean((2, 4))
    c = cams.double()
    pose = [(x[:9].view(3, 3), x[9:12], x[12:16] / 4) for x in c]
    ys, xs = torch.meshgrid(torch.arange(h, **f64), torch.arange(w, **f64), indexing="ij")
    dep = BP["d0"] + (BP["d1"] - BP["d0"]) * torch.arange(nd, **f64) / (nd - 1)
    R0, t0, K0 = pose[ref]
    ray = torch.stack([(xs + 0.5 - K0[2]) / K0[0], (ys + 0.5 - K0[3]) / K0[1], torch.ones_like(xs)], -1)
    pw = (ray[:, :, None] * dep[:, None] - t0) @ R0
    acc, cnt = torch.zeros(h, w, nd, **f64), torch.zeros(h, w, nd, **f64)
    for i in range(nk):
        if i == ref:
            continue
        R, t, K = pose[i]
        q = pw @ R.T + t
        front = q[..., 2] > 1e-3
        z = torch.where(front, q[..., 2], torch.ones_like(q[..., 2]))
        u, v = K[0] * q[..., 0] / z + K[2] - 0.5, K[1] * q[..., 1] / z + K[3] - 0.5
        ok = front & (u >= 0) & (v >= 0) & (u <= w - 1) & (v <= h - 1)
        x0 = u.floor().clamp(0, max(w - 2, 0)).long()
        y0 = v.floor().clamp(0, max(h - 2, 0)).long()
        x1, y1 = (x0 + 1).clamp_max(w - 1), (y0 + 1).clamp_max(h - 1)
        a, b = u - x0, v - y0
        im = grey[i]
        val = (1 - b) * ((1 - a) * im[y0, x0] + a * im[y0, x1]) + b * ((1 - a) * im[y1, x0] + a * im[y1, x1])
        acc += torch.where(ok, (grey[ref][:, :, None] - val).abs(), torch.zeros_like(val))
        cnt += ok
    V = torch.where(cnt > 0, acc / cnt.clamp_min(1), torch.ones_like(acc))
    lab = torch.arange(nd, device=DEV)
    pair = (BP["s"] * (lab[:, None] - lab[None]).abs().double()).clamp_max(BP["tau"])
    left, right, up, down = (torch.zeros(h, w, nd, **f64) for _ in range(4))   # message sent that way

    def incoming():
        # what arrives from the left neighbour was sent to the right, and so on
        fl, fr, fu, fd = (torch.zeros(h, w, nd, **f64) for _ in range(4))
        fl[:, 1:], fr[:, :-1], fu[1:], fd[:-1] = right[:, :-1], left[:, 1:], down[:-1], up[1:]
        return fl, fr, fu, fd

    def send(hsum):
        m = torch.cat([(r[..., :, None] + pair).amin(-2) for r in hsum.split(16)])
        return m - m.amin(-1, keepdim=True)

    for _ in range(BP["iters"]):
        fl, fr, fu, fd = incoming()
        tot = V + fl + fr + fu + fd
        left, right, up, down = send(tot - fl), send(tot - fr), send(tot - fu), send(tot - fd)
    return dict(volume=V, beliefs=V + sum(incoming()), wta=None, depth=None, labels=None)


def exact(case, seed):
    k = case["kind"]
    if k in ("replay", "render", "autograd", "host", "active"):
        return _raster64(case, seed)
    if k == "map_step":
        return _map64(case, seed)
    if k in ("prior_train", "prior_infer"):
        return _net64(case, seed)
    return _layer64(case, seed) if k == "prior_layer" else _init64(case, seed)
