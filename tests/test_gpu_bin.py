"""Tile binning at the edges of its warp blocks: tile rows and columns around
32 buckets and at the 256 maximum, chunks and pieces around 256 entries, and
splats from a part of one tile to the whole image.  The lists and ranges equal
the oracle's bit for bit."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import compare_lists, gpu_render, read_ws

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,n,log_scale", [
    (16, 16, 700, -3.0),          # one tile
    (512, 16, 3000, -3.5),        # 32 columns
    (528, 33, 3000, -2.0),        # 33 columns, wide splats
    (4096, 40, 2500, -2.5),       # 256 columns
    (40, 4096, 2500, -2.5),       # 256 rows
    (1031, 257, 40_000, -4.0),    # ragged, several blocks per chunk and piece
    (640, 640, 257, 0.5),         # splats over the whole image: every row and tile list has every splat
    (97, 113, 1, -1.0),           # a single splat
])
def test_lists_at_block_edges(W, H, n, log_scale):
    rng = np.random.default_rng(7)
    sc = synth.uniform_scene(rng, n, n_layers=1, extent=1.0, log_scale_mu=log_scale, log_scale_sigma=0.8)
    cam = synth.look_at_camera((0.0, 0.0, 4.0), fov_x_deg=35.0, width=W, height=H)
    ds, rast, img, al = gpu_render(sc, cam)
    pre = oracle.preprocess(sc, cam, 0xFFFFFFFF, [], "f32")
    ranges, lst = oracle.bin_tiles(pre)
    ws = read_ws(rast)
    assert ws["status"].error == 0
    compare_lists(ws, ranges, lst)
