"""The forward's tile order and checkpoint bases, which the tile binning writes:
every tile once, heaviest bucket first, empty lists last and counted out of the
queue, disjoint checkpoint segments; also after a pair list that overflowed."""
import numpy as np
import pytest
import torch

import synth
from paper_2410_16978_gb300 import DeviceScene, Rasterizer, _lib
from tests.gpu_util import gpu_render, read_ws

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h,n", [(1, 1, 3), (16, 16, 40), (17, 33, 700), (4096, 31, 900), (50, 4096, 900), (640, 480, 9000)])
def test_images_of_every_grid(w, h, n):
    """Grids of one tile, one row and one column up to the 256 the binning takes: the image is the
    background where a tile has no list, and a second render (other tie orders) gives the same bits."""
    rng = np.random.default_rng(n)
    sc = synth.uniform_scene(rng, n, n_layers=1, extent=0.6, log_scale_mu=-3.0, log_scale_sigma=0.3)
    cam = synth.look_at_camera((0.0, 0.0, 4.0), fov_x_deg=40.0, width=w, height=h)
    ds, rast, img, al = gpu_render(sc, cam, bg=(0.2, 0.4, 0.6))
    ws = read_ws(rast)
    assert ws["status"].error == 0
    rg = ws["ranges"].reshape(-1, 2).astype(np.int64)
    ty, tx = (h + 15) // 16, (w + 15) // 16
    empty = np.repeat(np.repeat((rg[:, 0] == rg[:, 1]).reshape(ty, tx), 16, 0), 16, 1)[:h, :w]
    got = img.cpu().numpy()
    for c, v in enumerate((0.2, 0.4, 0.6)):
        assert (got[c][empty] == np.float32(v)).all()
    assert (al.cpu().numpy()[empty] == 0).all()
    img2, al2 = rast.render(ds, cam, bg=(0.2, 0.4, 0.6))
    assert torch.equal(img, img2) and torch.equal(al, al2)


def test_overflowed_list_renders_background():
    rng = np.random.default_rng(1)
    sc = synth.uniform_scene(rng, 5000, n_layers=1, extent=0.6, log_scale_mu=-2.0, log_scale_sigma=0.3)
    cam = synth.look_at_camera((0.0, 0.0, 4.0), fov_x_deg=40.0, width=300, height=200)
    ds = DeviceScene.from_host(sc)
    r = Rasterizer(sc.n, 300, 200, dup_capacity=1000)
    for _ in range(2):
        img, al = r.render(ds, cam, bg=(0.2, 0.4, 0.6), check=False)
        assert r.status().error == _lib.GS_ERR_WORKSPACE
        assert all(bool((img[c] == v).all()) for c, v in enumerate((0.2, 0.4, 0.6)))
        assert bool((al == 0).all())


@pytest.mark.parametrize("n", [65_536, 65_537])
def test_pair_counts_beyond_32_bits(n):
    """65,536 Gaussians that cover the 65,536 tiles of the largest image are 2^32 pairs: the total must not wrap
    into the capacity.  No list is written, and the status holds what the frame needs."""
    from tests.helpers import axis_camera, make_scene
    means = np.random.default_rng(n).uniform(-0.1, 0.1, (n, 3))
    sc = make_scene(means, 3.0, opacity_logit=-3.0)
    cam = axis_camera(width=4096, height=4096)
    r = Rasterizer(n, 4096, 4096, dup_capacity=1 << 20)
    img, al = r.render(DeviceScene.from_host(sc), cam, bg=(0.2, 0.4, 0.6), check=False)
    st = r.status()
    assert st.n_visible == n
    assert st.n_dup == n * 65_536
    assert st.error == _lib.GS_ERR_WORKSPACE
    assert all(bool((img[c] == v).all()) for c, v in enumerate((0.2, 0.4, 0.6)))
    assert bool((al == 0).all())
