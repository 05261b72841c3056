"""Views of one scene whose preprocess is taken together (2^19 Gaussians times
views or more) give the bits of single renders: different cameras, sizes, layer masks
and clip planes, a scene just below and just above the size, in 32 and 16 bits,
and a batch in which one view shows another scene."""
import numpy as np
import pytest
import torch

import synth
from paper_2410_16978_gb300 import DeviceScene, Rasterizer, _lib

pytestmark = pytest.mark.gpu


def _scene(n, dt, seed):
    rng = np.random.default_rng(seed)
    sc = synth.uniform_scene(rng, n, n_layers=3, extent=0.9, log_scale_mu=-4.5, log_scale_sigma=0.4, sh_degree=1,
                             sh_sigma=0.2)
    return DeviceScene.from_host(sc, sh_dtype=dt, sr_dtype=dt)


def _views(scenes):
    out = []
    for k, (eye, w, h, mask, planes) in enumerate([
            ((0.0, 0.0, 4.0), 96, 80, 0b111, []),
            ((2.0, 0.5, 1.0), 65, 97, 0b010, [((0.0, 1.0, 0.0), 0.1, 0b111)]),
            ((0.2, 0.1, 0.3), 40, 40, 0b101, [((1.0, 0.0, 0.0), 0.0, 0b100), ((0.0, 0.0, 1.0), 0.2, 0b001)])]):
        sc = scenes[min(k, len(scenes) - 1)]
        cam = synth.look_at_camera(eye, fov_x_deg=45.0, width=w, height=h)
        out.append((sc, cam, mask, planes, (0.1 * k, 0.2, 0.3), Rasterizer(sc.n, w, h, dup_capacity=4 << 20)))
    return out


@pytest.mark.parametrize("dt", ["f32", "f16"])
@pytest.mark.parametrize("sizes", [(174_762,), (174_763,), (190_001,), (190_001, 189_000)])
def test_batch_equals_single_renders(dt, sizes):
    views = _views([_scene(n, dt, n) for n in sizes])
    ref = [r.render(sc, cam, mask, planes, bg) for sc, cam, mask, planes, bg, r in views]
    status = [r.status() for *_, r in views]
    img = [torch.empty_like(i) for i, _ in ref]
    al = [torch.empty_like(a) for _, a in ref]
    _lib.gs_render_batch([dict(scene=sc.c_struct(), camera=_lib.make_camera(cam), layer_mask=mask, planes=planes, bg=bg,
                               workspace=r.workspace, ws_bytes=r.ws_bytes, image=img[k], alpha=al[k])
                          for k, (sc, cam, mask, planes, bg, r) in enumerate(views)],
                         int(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    for k, (*_, r) in enumerate(views):
        assert status[k].error == 0 and r.status().n_dup == status[k].n_dup > 0
        assert torch.equal(img[k], ref[k][0]) and torch.equal(al[k], ref[k][1]), k
