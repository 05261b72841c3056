"""The chain rule moves SH rows through shared memory a warp at a time: counts
around a warp and a block, every degree, gradient arrays on a 16-byte boundary
and 4 bytes off one, with culled and frozen Gaussians among the rows."""
import pytest
import torch

import numpy as np
import synth
from paper_2410_16978_gb300 import DeviceScene, Rasterizer

pytestmark = pytest.mark.gpu
FIELDS = ("means", "log_scales", "quats", "opacity_logit", "sh")


def _off(t):
    return torch.empty(t.numel() + 1, device="cuda")[1:].view(t.shape).copy_(t)


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 31, 33, 128, 161])
def test_unaligned_rows_equal_aligned(deg, n):
    rng = np.random.default_rng(10 * n + deg)
    sc = synth.uniform_scene(rng, n, n_layers=2, extent=1.5, log_scale_mu=-2.0, log_scale_sigma=0.3)
    K = (deg + 1) ** 2
    sh = rng.standard_normal((n, K, 3)).astype(np.float32) * 0.3
    cam = synth.look_at_camera((0.0, 0.0, 4.0), fov_x_deg=30.0, width=50, height=41)    # the outer ones are culled
    d = torch.randn((3, 41, 50), generator=torch.Generator("cuda").manual_seed(n), device="cuda")
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (sc.means, sc.log_scales, sc.quats, sc.opacity_logit, sh)]
    layer = torch.from_numpy(sc.layer.astype(np.uint8)).cuda()

    def run(move):
        ds = DeviceScene(*t, layer, deg)
        r = Rasterizer(n, 50, 41)
        r.render(ds, cam)
        out = {k: move(torch.full(p.shape, float("nan"), device="cuda")) for k, p in zip(FIELDS, ds.params())}
        return r.backward(ds, cam, (0.0, 0.0, 0.0), d, None, 0b10, grads=out)

    a, b = run(lambda x: x.clone()), run(_off)
    for k in FIELDS:
        assert bool(torch.isfinite(a[k]).all()), k                 # every row is written
        assert float((a[k] - b[k]).norm()) <= 1e-5 * float(a[k].norm()) + 1e-20, k     # (sums are atomic)
        assert bool((a[k][layer == 0] == 0).all()), k
