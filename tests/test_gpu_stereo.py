"""Stereo rendering (Sec. 3.3: one render per eye; the paper's shared-eye
sort as an option).  Exact mode equals two gs_render calls bit for bit.
Shared mode: the left eye is still exact; the right eye's tile lists equal the
oracle's lists of the right eye ordered by the shared key (left-eye depth
where the left eye sees the Gaussian, else right-eye depth) bit for bit, and
its pixels match the oracle compositor over those lists within 1e-5."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2410_16978_gb300 import DeviceScene, Rasterizer, _lib
from tests.gpu_util import compare_image, compare_lists, dequantised, psnr, read_ws

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _stereo(scale=0.01, W=160, H=176):
    w = synth.scene_c4(scale=scale, width=W, height=H)
    return w["scene"], w["cameras"], w["layer_mask"], w["planes"]


def _run(sc, cams, mask, planes, bg, shared):
    ds = DeviceScene.from_host(sc)
    r = [Rasterizer(sc.n, c.width, c.height) for c in cams]
    for rr, c in zip(r, cams):      # size each eye's pair list (grows the workspace when needed)
        rr.render(ds, c, mask, planes, bg, check=True)
    if shared:                      # the shared order adds the Gaussians only the other eye sees
        for rr in r:
            rr._alloc(int(rr.dup_capacity * 1.1) + 4096)
    imgs = [torch.empty((3, c.height, c.width), device="cuda") for c in cams]
    als = [torch.empty((c.height, c.width), device="cuda") for c in cams]
    _lib.gs_render_stereo(ds.c_struct(), _lib.make_camera(cams[0]), _lib.make_camera(cams[1]), mask, list(planes), bg,
                          r[0].workspace, r[0].ws_bytes, r[1].workspace, r[1].ws_bytes, imgs[0], als[0], imgs[1],
                          als[1], shared, 0)
    torch.cuda.synchronize()
    assert r[0].status().error == 0 and r[1].status().error == 0
    return ds, r, imgs, als


def test_exact_stereo_equals_two_renders():
    sc, cams, mask, planes = _stereo()
    bg = (0.1, 0.2, 0.3)
    ds, r, imgs, als = _run(sc, cams, mask, planes, bg, False)
    for e in range(2):
        rr = Rasterizer(sc.n, cams[e].width, cams[e].height)
        img, al = rr.render(ds, cams[e], mask, planes, bg)
        torch.cuda.synchronize()
        assert torch.equal(img, imgs[e]) and torch.equal(al, als[e]), e


def test_shared_sort_matches_oracle():
    sc, cams, mask, planes = _stereo()
    bg = (0.0, 0.0, 0.0)
    ds, r, imgs, als = _run(sc, cams, mask, planes, bg, True)
    # left eye: exactly the mono render
    rl = Rasterizer(sc.n, cams[0].width, cams[0].height)
    img_l, al_l = rl.render(ds, cams[0], mask, planes, bg)
    torch.cuda.synchronize()
    assert torch.equal(img_l, imgs[0]) and torch.equal(al_l, als[0])
    # right eye: oracle lists in the shared order
    pre_l = oracle.preprocess(sc, cams[0], mask, planes, "f32")
    pre_r = oracle.preprocess(sc, cams[1], mask, planes, "f32")
    shared = dict(pre_r)
    shared["depth"] = np.where(pre_l["vis"] > 0, pre_l["depth"], pre_r["depth"])
    ranges, lst = oracle.bin_tiles(shared)
    ws = read_ws(r[1])
    assert ws["status"].error == 0
    compare_lists(ws, ranges, lst)
    co = oracle.composite(pre_r, ranges, lst, bg)
    st = compare_image(imgs[1].cpu().numpy(), als[1].cpu().numpy(), ws["n_contrib"].astype(np.int64), co, TOL)
    assert st["n_bad"] == 0, st
    # the approximation against the exact right eye
    rr = Rasterizer(sc.n, cams[1].width, cams[1].height)
    img_r, _ = rr.render(ds, cams[1], mask, planes, bg)
    torch.cuda.synchronize()
    p = psnr(imgs[1].cpu().numpy(), img_r.cpu().numpy())
    print("shared-sort right eye vs exact: PSNR %.2f dB, max |diff| %.3g"
          % (p, float((imgs[1] - img_r).abs().max())))
    assert p > 40.0


def test_stereo_rejects_shared_workspace():
    sc, cams, mask, planes = _stereo(0.002, 32, 32)
    ds = DeviceScene.from_host(sc)
    r = Rasterizer(sc.n, 32, 32)
    img = torch.empty((3, 32, 32), device="cuda")
    with pytest.raises(_lib.GsError):
        _lib.gs_render_stereo(ds.c_struct(), _lib.make_camera(cams[0]), _lib.make_camera(cams[1]), mask, [],
                              (0, 0, 0), r.workspace, r.ws_bytes, r.workspace, r.ws_bytes, img, None, img, None,
                              True, 0)


def test_shared_sort_full_size_quality():
    """The 3M-Gaussian stereo workload (2 x 2064x2208): the shared-sort right
    eye against the exact right eye (printed; the paper reports the shared
    order as visually equivalent)."""
    w = synth.scene_c4()
    sc, cams = w["scene"], w["cameras"]
    ds, r, imgs, _ = _run(sc, cams, w["layer_mask"], w["planes"], (0.0, 0.0, 0.0), True)
    rr = Rasterizer(sc.n, cams[1].width, cams[1].height)
    img_r, _ = rr.render(ds, cams[1], w["layer_mask"], w["planes"], (0.0, 0.0, 0.0))
    torch.cuda.synchronize()
    d = (imgs[1] - img_r).abs()
    p = psnr(imgs[1].cpu().numpy(), img_r.cpu().numpy())
    print("c4 shared-sort right eye vs exact: PSNR %.2f dB, max |diff| %.3g, pixels differing %d of %d"
          % (p, float(d.max()), int((d.amax(0) > 0).sum()), d.shape[1] * d.shape[2]))
    assert p >= 50.0


@pytest.mark.parametrize("eye", [0, 1])
def test_shared_sort_backward_per_eye(eye):
    """The backward of each eye after a shared-sort stereo render (the right
    eye's workspace holds a copy of the shared visible list): gradients within
    the field-normalised 1e-5 bar of the oracle's backward over that eye's
    lists (the left eye's own order, the right eye's shared order)."""
    from tests.gpu_util import f64_scene
    sc, cams, mask, planes = _stereo()
    bg = (0.1, 0.2, 0.3)
    ds, r, imgs, als = _run(sc, cams, mask, planes, bg, True)
    cam = cams[eye]
    rng = np.random.default_rng(11 + eye)
    dimg = rng.standard_normal((3, cam.height, cam.width)).astype(np.float32)
    dal = rng.standard_normal((cam.height, cam.width)).astype(np.float32)
    g = r[eye].backward(ds, cam, bg, torch.from_numpy(dimg).cuda(), torch.from_numpy(dal).cuda())
    torch.cuda.synchronize()
    pre_l = oracle.preprocess(sc, cams[0], mask, planes, "f32")
    pre = oracle.preprocess(sc, cam, mask, planes, "f32")
    keyed = dict(pre)
    if eye == 1:
        keyed["depth"] = np.where(pre_l["vis"] > 0, pre_l["depth"], pre["depth"])
    ranges, lst = oracle.bin_tiles(keyed)
    cb = oracle.composite_backward(pre, ranges, lst, bg, dimg, dal)
    ref = oracle.chain(f64_scene(sc), cam, pre["vis"], cb["rec_grad"])
    ok = cb["touched_fragile"] == 0
    assert ok.mean() > 0.6
    for f in ("means", "log_scales", "quats", "opacity_logit", "sh"):
        a = g[f].cpu().numpy().reshape(sc.n, -1)[ok].astype(np.float64)
        b = ref[f].reshape(sc.n, -1)[ok]
        assert np.abs(a - b).max() <= 1e-5 * np.abs(b).max(), (eye, f)
    vis = pre["vis"] > 0
    assert np.all(g["sh"].cpu().numpy()[~vis] == 0)


def test_shared_sort_with_gaussians_only_one_eye_sees():
    """A narrow view cuts off Gaussians at one eye's image border that the
    other eye sees.  They are in the shared order of both eyes, but the eye
    that does not see them has no record of them (its workspace holds whatever
    was there before: here random bytes) and must not list them."""
    sc = synth.scene_c4(scale=0.004)["scene"]
    centre = synth.look_at_camera((0.0, 0.0, 4.0), fov_x_deg=9.0, width=208, height=80)
    cams = list(synth.stereo_pair(centre, 0.064))
    pre = [oracle.preprocess(sc, c, 0b11111, [], "f32") for c in cams]
    vis = [p["vis"] > 0 for p in pre]
    assert (vis[0] & ~vis[1]).sum() > 50 and (vis[1] & ~vis[0]).sum() > 50
    ds = DeviceScene.from_host(sc)
    g = torch.Generator("cuda").manual_seed(5)
    r = [Rasterizer(sc.n, c.width, c.height) for c in cams]
    for rr in r:
        rr.workspace.random_(0, 256, generator=g)
    imgs = [torch.empty((3, c.height, c.width), device="cuda") for c in cams]
    _lib.gs_render_stereo(ds.c_struct(), _lib.make_camera(cams[0]), _lib.make_camera(cams[1]), 0b11111, [],
                          (0.1, 0.2, 0.3), r[0].workspace, r[0].ws_bytes, r[1].workspace, r[1].ws_bytes, imgs[0],
                          None, imgs[1], None, True, 0)
    torch.cuda.synchronize()
    for e in range(2):
        keyed = dict(pre[e])
        if e == 1:
            keyed["depth"] = np.where(vis[0], pre[0]["depth"], pre[1]["depth"])
        ranges, lst = oracle.bin_tiles(keyed)
        ws = read_ws(r[e])
        assert ws["status"].error == 0
        compare_lists(ws, ranges, lst)
