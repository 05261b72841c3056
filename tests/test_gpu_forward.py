"""The forward compositor at the edges of its chunks (64 and 128 list entries),
checkpoint segments (256) and both pixel layouts (one pixel per lane, and two for
launches of many pixels): lists of exactly n splats over the same tiles, faint
ones (every walk reaches the end) and opaque ones (walks stop inside a chunk).
Every compared pixel is within 1e-5 of the FP64 compositor over the GPU's records
or of its alternative at a fragile threshold."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import compare_image, gpu_render, read_ws

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _stack(n, logit):
    rng = np.random.default_rng(n)
    sc = synth.uniform_scene(rng, n, n_layers=1, extent=0.25, log_scale_mu=-1.0, log_scale_sigma=0.2)
    sc.opacity_logit[:] = logit + 0.2 * rng.standard_normal(n).astype(np.float32)
    return sc


@pytest.mark.parametrize("n", [1, 2, 3, 63, 64, 65, 127, 128, 129, 255, 256, 257, 385, 513])
@pytest.mark.parametrize("logit", [-4.0, 1.0])
def test_chunk_and_segment_edges(n, logit):
    sc = _stack(n, logit)
    cam = synth.look_at_camera((0.0, 0.0, 4.0), fov_x_deg=40.0, width=45, height=37)
    bg = (0.2, 0.4, 0.6)
    ds, rast, img, al = gpu_render(sc, cam, bg=bg)
    pre = oracle.preprocess(sc, cam, 0xFFFFFFFF, [], "f32")
    ranges, lst = oracle.bin_tiles(pre)
    ws = read_ws(rast)
    st = compare_image(img.cpu().numpy(), al.cpu().numpy(), ws["n_contrib"].astype(np.int64),
                       oracle.composite(pre, ranges, lst, bg), TOL)
    assert st["n_bad"] == 0, st


@pytest.mark.parametrize("n,logit", [(1, -4.0), (65, -4.0), (128, 1.0), (257, -4.0), (600, -3.0)])
def test_two_pixels_per_lane(n, logit):
    W, H = 1637, 1003                      # ragged, above the size from which the forward takes two pixels per lane
    sc = _stack(n, logit)
    cam = synth.look_at_camera((0.0, 0.0, 4.0), fov_x_deg=60.0, width=W, height=H)
    bg = (0.2, 0.4, 0.6)
    ds, rast, img, al = gpu_render(sc, cam, bg=bg, cap=4 << 20)
    pre = oracle.preprocess(sc, cam, 0xFFFFFFFF, [], "f32")
    ranges, lst = oracle.bin_tiles(pre)
    ws = read_ws(rast)
    assert ws["status"].error == 0
    rng = np.random.default_rng(3)
    xs = np.concatenate([rng.integers(0, W, 3000), np.full(200, W - 1), rng.integers(0, W, 200)]).astype(np.int32)
    ys = np.concatenate([rng.integers(0, H, 3000), rng.integers(0, H, 200), np.full(200, H - 1)]).astype(np.int32)
    cp = oracle.composite_pixels(pre, ranges, lst, xs, ys, bg)
    rgb, a = img.cpu().numpy()[:, ys, xs].T.astype(np.float64), al.cpu().numpy()[ys, xs].astype(np.float64)
    nc = ws["n_contrib"][ys, xs].astype(np.int64)
    e1 = np.maximum(np.abs(rgb - cp["rgb"]).max(1), np.abs(a - cp["alpha"]))
    e2 = np.maximum(np.abs(rgb - cp["alt_rgb"]).max(1), np.abs(a - cp["alt_alpha"]))
    ok = ((e1 <= TOL) & (nc == cp["ncontrib"])) | ((e2 <= TOL) & (nc == cp["alt_ncontrib"]) & (cp["fragile"] > 0))
    assert np.all(ok | (cp["fragile"] > 1)), (np.flatnonzero(~ok)[:5], e1.max())
