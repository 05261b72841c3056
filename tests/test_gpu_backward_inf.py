"""An infinite upstream gradient at one pixel reaches the splats blended there
and no others: the backward's lanes take every splat of their 8x8 block, also
those that do not touch their pixels."""
import pytest
import torch

import synth
from paper_2410_16978_gb300 import DeviceScene, Rasterizer

pytestmark = pytest.mark.gpu
FIELDS = ("means", "log_scales", "quats", "opacity_logit", "sh")


@pytest.mark.parametrize("x,y", [(40, 41), (0, 0), (88, 76)])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_stays_with_its_pixel(x, y, value):
    w = synth.scene_c4(scale=0.01, width=89, height=77)
    sc, cam, bg = DeviceScene.from_host(w["scene"]), w["cameras"][0], (0.1, 0.2, 0.3)
    r = Rasterizer(sc.n, cam.width, cam.height)
    r.render(sc, cam, w["layer_mask"], (), bg)
    g = torch.Generator("cuda").manual_seed(5)
    d = torch.randn((3, 77, 89), generator=g, device="cuda")
    d[:, y, x] = 0.0
    only = torch.zeros_like(d)
    only[:, y, x] = 1.0
    bad = d.clone()
    bad[1, y, x] = value
    ref, one, got = (r.backward(sc, cam, bg, t) for t in (d, only, bad))
    csum = torch.zeros(sc.n, device="cuda")
    r.backward(sc, cam, bg, only, contrib_sum=csum)
    touched = one["sh"].reshape(sc.n, -1).abs().amax(1) + one["opacity_logit"].abs() > 0
    for k in FIELDS:
        a, b = got[k][~touched], ref[k][~touched]
        assert bool(torch.isfinite(a).all()), k
        assert float((a - b).norm()) <= 1e-5 * float(b.norm()) + 1e-20, k
