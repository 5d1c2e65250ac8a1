"""Learned depth prior: a small U-Net trained on (RGB, depth) pairs rendered
from the map, proposing depths for the Gaussians of newly observed regions.

GEVO initialises those Gaussians from a photometric cost volume (Eq. 1) with
belief propagation and SPGF* (Section III-A); the prior replaces the depth
proposal with one network evaluation and is judged against that plain
initialisation after the same optimisation.

Architecture (levels l = 0..L-1, channels c_l, default 16/32/64/128): per level
two 3x3 conv + ReLU; 2x2 max pool between encoder levels; x2 nearest upsample,
concatenation with the encoder's skip, two 3x3 conv + ReLU per decoder level;
1x1 head to log-depth.  BF16 weights and activations, FP32 accumulation (in
tensor memory), FP32 master weights with Adam.  Every step runs in libgevo's
kernels (include/gevo_prior.h); torch only holds the buffers.
"""
from __future__ import annotations

import ctypes

import numpy as np
import torch

from . import _abi

BF16 = torch.bfloat16


def _ptr(t: torch.Tensor, offset_elems: int = 0):
    return ctypes.c_void_p(t.data_ptr() + offset_elems * t.element_size())


class DepthUNet:
    def __init__(self, nb: int, H: int, W: int, chans=(16, 32, 64, 128), device="cuda",
                 seed: int = 0):
        L = len(chans)
        assert H % (1 << (L - 1)) == 0 and W % (1 << (L - 1)) == 0
        assert all(c % 8 == 0 for c in chans) and chans[0] <= 16
        self.nb, self.H, self.W, self.L, self.chans = nb, H, W, L, tuple(chans)
        self.dev = torch.device(device)
        self.hw = [(H >> i, W >> i) for i in range(L)]
        self.P = [nb * h * w for h, w in self.hw]
        self.ccat = [chans[i + 1] + chans[i] for i in range(L - 1)]
        rs = np.random.default_rng(seed)
        self.layers = {}
        for i in range(L):
            self._layer(f"enc{i}a", 8 if i == 0 else chans[i - 1], chans[i], rs, 3 if i == 0 else None)
            self._layer(f"enc{i}b", chans[i], chans[i], rs)
        for i in range(L - 2, -1, -1):
            self._layer(f"dec{i}a", self.ccat[i], chans[i], rs)
            self._layer(f"dec{i}b", chans[i], chans[i], rs)
        f32 = torch.float32
        d = self.dev
        self.head_w = torch.from_numpy((rs.normal(size=chans[0]) * np.sqrt(1.0 / chans[0]))
                                       .astype(np.float32)).to(d)
        self.head_b = torch.full((1,), 1.0, dtype=f32, device=d)   # log(2.7 m): room-scale start
        self.head_state = [torch.zeros_like(self.head_w) for _ in range(3)] + \
            [torch.zeros_like(self.head_b) for _ in range(3)]       # dw, m, v, db, m, v
        # activations
        z16 = lambda p, c: torch.zeros(p, c, dtype=BF16, device=d)
        z32 = lambda p, c: torch.zeros(p, c, dtype=f32, device=d)
        self.X0 = z16(self.P[0], 8)
        self.A = [z16(self.P[i], chans[i]) for i in range(L)]
        self.CAT = [z16(self.P[i], self.ccat[i]) for i in range(L - 1)]
        self.BOT = z16(self.P[L - 1], chans[L - 1])
        self.POOL = [None] + [z16(self.P[i], chans[i - 1]) for i in range(1, L)]
        self.DA = [z16(self.P[i], chans[i]) for i in range(L - 1)]
        self.DB = [z16(self.P[i], chans[i]) for i in range(L - 1)]
        self.pred = torch.zeros(self.P[0], dtype=f32, device=d)
        self.dpred = torch.zeros_like(self.pred)
        self.loss = torch.zeros(1, dtype=f32, device=d)
        # gradients of activations: FP32 where two paths meet or a gradient is summed over
        # pixels before its ReLU, else only the masked BF16 dZ of two layers at a time
        self.dCAT = [z32(self.P[i], self.ccat[i]) for i in range(L - 1)]
        self.dPOOL = [None] + [z32(self.P[i], chans[i - 1]) for i in range(1, L)]
        zmax = max(self.P[i] * chans[i] for i in range(L))
        self.dZ = torch.zeros(zmax, dtype=BF16, device=d)
        self.dZ2 = torch.zeros(zmax, dtype=BF16, device=d)
        self.ws = torch.zeros(256, dtype=torch.uint8, device=d)
        self.step_count = 0

    # ---- parameters ----------------------------------------------------------------
    def _layer(self, name, cin, cout, rs, cin_real=None):
        fan_in = 9 * (cin_real if cin_real is not None else cin)
        w = (rs.normal(size=(cout, 9, cin)) * np.sqrt(2.0 / fan_in)).astype(np.float32)
        if cin_real is not None:
            w[:, :, cin_real:] = 0.0
        d = self.dev
        W32 = torch.from_numpy(w.reshape(cout, 9 * cin)).to(d)
        lay = dict(cin=cin, cout=cout, W32=W32, b32=torch.zeros(cout, device=d),
                   W16=torch.zeros(cout, 9 * cin, dtype=BF16, device=d),
                   Wf16=torch.zeros(cin, 9 * cout, dtype=BF16, device=d),
                   dW=torch.zeros_like(W32), db=torch.zeros(cout, device=d),
                   mW=torch.zeros_like(W32), vW=torch.zeros_like(W32),
                   mb=torch.zeros(cout, device=d), vb=torch.zeros(cout, device=d))
        self.layers[name] = lay
        _abi.prior_call("gevo_to_bf16", W32.numel(), W32, lay["W16"])
        _abi.prior_call("gevo_flip3x3", cout, cin, lay["W16"], lay["Wf16"])

    def parameters_numpy(self):
        """FP32 masters (for the oracle comparison)."""
        out = {k: (v["W32"].cpu().numpy().reshape(v["cout"], 9, v["cin"]), v["b32"].cpu().numpy())
               for k, v in self.layers.items()}
        out["head"] = (self.head_w.cpu().numpy(), self.head_b.cpu().numpy())
        return out

    # ---- forward -------------------------------------------------------------------
    def _conv(self, name, nb, h, w, X, Y, ldy, y_off=0, relu=True):
        lay = self.layers[name]
        _abi.prior_call("gevo_conv3x3", nb, h, w, lay["cin"], X, lay["cout"], lay["W16"],
                        lay["b32"], _ptr(Y, y_off), ldy, 1, int(relu), 0.0, self.ws)

    def forward(self, rgb_planar: torch.Tensor):
        """rgb_planar: FP32 [nb, 3, H, W] (contiguous).  Returns pred (log-depth, [nb*H*W])."""
        nb, L, c = self.nb, self.L, self.chans
        _abi.prior_call("gevo_rgb_pack", nb, self.H, self.W, rgb_planar, self.X0)
        for i in range(L):
            h, w = self.hw[i]
            Xin = self.X0 if i == 0 else self.POOL[i]
            self._conv(f"enc{i}a", nb, h, w, Xin, self.A[i], c[i])
            if i < L - 1:
                self._conv(f"enc{i}b", nb, h, w, self.A[i], self.CAT[i], self.ccat[i], c[i + 1])
                _abi.prior_call("gevo_maxpool2", nb, h, w, c[i], _ptr(self.CAT[i], c[i + 1]),
                                self.ccat[i], self.POOL[i + 1])
            else:
                self._conv(f"enc{i}b", nb, h, w, self.A[i], self.BOT, c[i])
        up = self.BOT
        for i in range(L - 2, -1, -1):
            h, w = self.hw[i]
            _abi.prior_call("gevo_upsample2", nb, h // 2, w // 2, c[i + 1], up, self.CAT[i],
                            self.ccat[i])
            self._conv(f"dec{i}a", nb, h, w, self.CAT[i], self.DA[i], c[i])
            self._conv(f"dec{i}b", nb, h, w, self.DA[i], self.DB[i], c[i])
            up = self.DB[i]
        last = self.DB[0] if L > 1 else self.BOT
        _abi.prior_call("gevo_head_fwd", self.P[0], c[0], last, self.head_w, self.head_b, self.pred)
        return self.pred

    # ---- backward ------------------------------------------------------------------
    def _wgrad(self, name, nb, h, w, Xin, dZ):
        lay = self.layers[name]
        _abi.prior_call("gevo_conv3x3_wgrad_nhwc", nb, h, w, lay["cin"], Xin, lay["cout"], dZ,
                        lay["dW"], self.ws)

    def _dgrad(self, name, nb, h, w, dZ, dX):
        """The FP32 gradient of a layer's input (one that has other uses than a ReLU)."""
        lay = self.layers[name]
        _abi.prior_call("gevo_conv3x3", nb, h, w, lay["cout"], dZ, lay["cin"], lay["Wf16"], None, dX,
                        lay["cin"], 0, 0, 0.0, self.ws)

    def _pair_bwd(self, lvl, kind, nb, h, w, Xin, mid, dZb):
        """Weight gradients of level lvl's two layers from the second one's dZ: the
        first one's (masked by its output `mid`) and its bias gradient come out of the
        second one's data gradient.  Returns the first one's dZ."""
        a, b = f"{kind}{lvl}a", f"{kind}{lvl}b"
        la, lb = self.layers[a], self.layers[b]
        self._wgrad(b, nb, h, w, mid, dZb)
        _abi.prior_call("gevo_conv3x3_relu_bwd", nb, h, w, lb["cout"], dZb, lb["cin"], lb["Wf16"], mid,
                        lb["cin"], self.dZ2, la["db"], self.ws)
        self._wgrad(a, nb, h, w, Xin, self.dZ2)
        return self.dZ2

    def backward(self):
        """Gradients of self.loss (after depth_loss) w.r.t. every parameter.  Every
        ReLU's gradient is applied by the pass that makes its dY (the head, a data
        gradient, the upsampling's or the pool's gradient), so dY is never stored."""
        nb, L, c = self.nb, self.L, self.chans
        # the weight gradients and the bias gradients are added to: clear them all at once
        torch._foreach_zero_([la[k] for la in self.layers.values() for k in ("dW", "db")])
        last, top = (self.DB[0], "dec0b") if L > 1 else (self.BOT, "enc0b")
        dw, _, _, db, _, _ = self.head_state
        _abi.prior_call("gevo_head_relu_bwd", self.P[0], c[0], last, self.head_w, self.dpred, self.dZ,
                        self.layers[top]["db"], dw, db)
        for i in range(L - 1):
            h, w = self.hw[i]
            dz = self._pair_bwd(i, "dec", nb, h, w, self.CAT[i], self.DA[i], self.dZ)
            self._dgrad(f"dec{i}a", nb, h, w, dz, self.dCAT[i])
            below, name = (self.BOT, f"enc{L - 1}b") if i + 1 == L - 1 else (self.DB[i + 1], f"dec{i + 1}b")
            _abi.prior_call("gevo_upsample2_relu_bwd", nb, h // 2, w // 2, c[i + 1], self.dCAT[i],
                            self.ccat[i], below, self.dZ, self.layers[name]["db"])
        for i in range(L - 1, -1, -1):
            h, w = self.hw[i]
            if i < L - 1:
                off = c[i + 1]
                _abi.prior_call("gevo_maxpool2_relu_bwd", nb, h, w, c[i], _ptr(self.CAT[i], off),
                                self.ccat[i], self.dPOOL[i + 1], _ptr(self.dCAT[i], off), self.ccat[i],
                                self.dZ, self.layers[f"enc{i}b"]["db"])
            Xin = self.X0 if i == 0 else self.POOL[i]
            dz = self._pair_bwd(i, "enc", nb, h, w, Xin, self.A[i], self.dZ)
            if i > 0:
                self._dgrad(f"enc{i}a", nb, h, w, dz, self.dPOOL[i])

    def depth_loss(self, target: torch.Tensor, weight: torch.Tensor):
        _abi.prior_call("gevo_depth_l1", self.P[0], self.pred, target, weight, self.loss, self.dpred)
        return self.loss

    def adam_step(self, lr=1e-3, b1=0.9, b2=0.999, eps=1e-8):
        self.step_count += 1
        lays = list(self.layers.values())
        dw, mw, vw, db, mb, vb = self.head_state
        # (parameter, gradient, moments, BF16 copy) of every tensor, one launch for all
        rows = [(la["W32"], la["dW"], la["mW"], la["vW"], la["W16"]) for la in lays] + \
            [(la["b32"], la["db"], la["mb"], la["vb"], None) for la in lays] + \
            [(self.head_w, dw, mw, vw, None), (self.head_b, db, mb, vb, None)]
        for i in range(0, len(rows), 64):
            part = rows[i:i + 64]
            size = (ctypes.c_int64 * len(part))(*[r[0].numel() for r in part])
            _abi.prior_call("gevo_adam_batch", len(part), size,
                            *[_abi.pointer_array([r[k] for r in part]) for k in range(5)],
                            lr, b1, b2, eps, self.step_count)
        for i in range(0, len(lays), 32):
            part = lays[i:i + 32]
            ints = [(ctypes.c_int32 * len(part))(*[la[k] for la in part]) for k in ("cout", "cin")]
            _abi.prior_call("gevo_flip3x3_batch", len(part), *ints,
                            _abi.pointer_array([la["W16"] for la in part]),
                            _abi.pointer_array([la["Wf16"] for la in part]))

    def train_step(self, rgb_planar, target, weight, lr=1e-3):
        self.forward(rgb_planar)
        self.depth_loss(target, weight)
        self.backward()
        self.adam_step(lr)
        return self.loss
