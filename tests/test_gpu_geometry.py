"""The geometry that the compositors read, a copy of every visible Gaussian's record: bit for bit the record, which
the other tests compare with the oracle."""
import numpy as np
import pytest
import torch

import synth
from paper_2410_16978_gb300 import DeviceScene, Rasterizer, _lib
from tests.helpers import branch_scene

pytestmark = pytest.mark.gpu


def _check(r, n, cam):
    lay = _lib.gs_workspace_layout(n, cam.width, cam.height, r.ws_bytes)
    ws = r.workspace.cpu().numpy()
    rec = ws[lay["rec"]:lay["rec"] + 48 * n].view(np.uint32).reshape(n, 12)
    at = (lay["rec"] + 48 * n + 255) // 256 * 256
    geo = ws[at:at + 32 * n].view(np.uint32).reshape(n, 8)
    vis = ws[lay["tiles"]:lay["tiles"] + 4 * n].view(np.uint32) > 0
    assert vis.any()
    assert np.array_equal(geo[vis], rec[vis, :8])


@pytest.mark.parametrize("sh_dtype,sr_dtype", [("f32", "f32"), ("f16", "f16"), ("bf16", "bf16")])
def test_copy_equals_record(sh_dtype, sr_dtype):
    sc, cam, planes, _ = branch_scene()
    ds = DeviceScene.from_host(sc, sh_dtype=sh_dtype, sr_dtype=sr_dtype)
    r = Rasterizer(sc.n, cam.width, cam.height)
    r.workspace.fill_(0xFF)
    r.render(ds, cam, 0xFFFFFFFF, planes)
    _check(r, sc.n, cam)


def test_copy_equals_record_in_views_of_one_scene():
    w = synth.scene_c4(scale=0.1, width=512, height=480)     # enough Gaussians that a thread takes one through both views
    ds = DeviceScene.from_host(w["scene"])
    n = w["scene"].n
    assert 2 * n >= 1 << 19
    cams = w["cameras"]
    rs = [Rasterizer(n, c.width, c.height) for c in cams]
    views = []
    for r, c in zip(rs, cams):
        r.workspace.fill_(0xFF)
        views.append(dict(scene=ds.c_struct(), camera=_lib.make_camera(c), layer_mask=0xFFFFFFFF, planes=[],
                          bg=(0.0, 0.0, 0.0), workspace=r.workspace, ws_bytes=r.ws_bytes,
                          image=torch.empty((3, c.height, c.width), device="cuda"), alpha=None))
    _lib.gs_render_batch(views, int(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    for r, c in zip(rs, cams):
        assert r.status().error == _lib.GS_OK
        _check(r, n, c)
