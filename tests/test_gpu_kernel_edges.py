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
