"""An upstream gradient that is not finite at one pixel, of the colour or of alpha: it reaches splats that are blended
there, and no others."""
import pytest
import torch

import synth
from paper_2410_16978_gb300 import DeviceScene, Rasterizer

pytestmark = pytest.mark.gpu
FIELDS = ("means", "log_scales", "quats", "opacity_logit", "sh")


@pytest.mark.parametrize("of_alpha", [False, True])
@pytest.mark.parametrize("x,y,covered", [(44, 38, True), (51, 30, True), (0, 0, False), (88, 76, False)])
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
def test_reaches_the_splats_of_its_pixel_alone(x, y, covered, value, of_alpha):
    w = synth.scene_c4(scale=0.01, width=89, height=77)
    sc, cam, bg = DeviceScene.from_host(w["scene"]), w["cameras"][0], (0.1, 0.2, 0.3)
    r = Rasterizer(sc.n, cam.width, cam.height)
    r.render(sc, cam, 0xFFFFFFFF, (), bg)
    g = torch.Generator("cuda").manual_seed(5)
    d = torch.randn((3, 77, 89), generator=g, device="cuda")
    da = torch.randn((77, 89), generator=g, device="cuda")
    d[:, y, x] = 0.0
    da[y, x] = 0.0
    only, bad, bad_a = torch.zeros_like(d), d.clone(), da.clone()
    only[:, y, x] = 1.0
    if of_alpha:
        bad_a[y, x] = value
    else:
        bad[1, y, x] = value
    ref, one, got = r.backward(sc, cam, bg, d, da), r.backward(sc, cam, bg, only), r.backward(sc, cam, bg, bad, bad_a)
    touched = (one["sh"].reshape(sc.n, -1).abs().amax(1) > 0) | (one["opacity_logit"].abs() > 0)
    assert bool(touched.any()) or not covered
    for k in FIELDS:
        a, b = got[k][~touched], ref[k][~touched]
        assert bool(torch.isfinite(a).all()), k
        assert float((a - b).norm()) <= 1e-5 * float(b.norm()) + 1e-20, k
    if covered:
        assert not bool(torch.isfinite(got["opacity_logit"][touched]).all())
