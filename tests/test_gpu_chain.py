"""The kernels of a call start ahead of the end of the one before them and wait
for it: back-to-back calls on one workspace, two streams at once and a captured
graph all give the bits of a call that ran alone."""
import pytest
import torch

import synth
from paper_2410_16978_gb300 import DeviceScene, Rasterizer, _lib
from paper_2410_16978_gb300.train import image_loss

pytestmark = pytest.mark.gpu
BG = (0.1, 0.2, 0.3)


class _Work:
    """One workspace and the buffers of a render, its image loss and its backward."""

    def __init__(self, w, k):
        self.sc, self.cam, self.mask = DeviceScene.from_host(w["scene"]), _lib.make_camera(w["cameras"][k]), w["layer_mask"]
        self.r = Rasterizer(self.sc.n, self.cam.width, self.cam.height)
        self.r.render(self.sc, self.cam, self.mask, (), BG)
        h, wd = self.cam.height, self.cam.width
        self.image, self.alpha = torch.empty((3, h, wd), device="cuda"), torch.empty((h, wd), device="cuda")
        self.d = torch.ones((3, h, wd), device="cuda")
        self.cmax = torch.zeros(self.sc.n, device="cuda")

    def step(self):
        self.cmax.zero_()
        self.r.render(self.sc, self.cam, self.mask, (), BG, self.image, self.alpha, check=False)
        self.r.backward(self.sc, self.cam, BG, self.d, None, 0xFFFFFFFF, None, self.cmax, self.grads)

    def alloc(self):
        self.grads = {k: torch.empty(p.shape, device="cuda") for k, p in
                      zip(("means", "log_scales", "quats", "opacity_logit", "sh"), self.sc.params())}
        return self

    def state(self):
        # (record-gradient sums are atomic: their last bits vary, so they are compared to rounding below)
        return [t.clone() for t in (self.image, self.alpha, self.cmax)], [g.clone() for g in self.grads.values()]


def _same(a, b):
    for x, y in zip(a[0], b[0]):
        assert torch.equal(x, y)
    for x, y in zip(a[1], b[1]):
        assert float((x - y).norm()) <= 1e-5 * float(y.norm()) + 1e-12


@pytest.mark.parametrize("scale", [0.002, 0.05])
def test_streams_repeats_and_capture(scale):
    w = synth.scene_c4(scale=scale, width=160, height=176)
    A, B = _Work(w, 0).alloc(), _Work(w, 1).alloc()
    A.step(), torch.cuda.synchronize()
    B.step(), torch.cuda.synchronize()
    ra, rb = A.state(), B.state()
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(20):
        for s, x in ((sa, A), (sb, B)):
            with torch.cuda.stream(s):
                x.step()
    torch.cuda.synchronize()
    _same(A.state(), ra)
    _same(B.state(), rb)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        A.step()
    A.image.zero_(), A.alpha.zero_()
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    _same(A.state(), ra)


def test_loss_after_itself():
    g = torch.Generator("cuda").manual_seed(1)
    x, t = torch.rand((3, 97, 131), generator=g, device="cuda"), torch.rand((3, 97, 131), generator=g, device="cuda")
    a, ta = torch.rand((97, 131), generator=g, device="cuda"), torch.rand((97, 131), generator=g, device="cuda")
    ref = image_loss(x, a, t, ta, BG, 0.2, 0.8).item()
    ws = torch.empty(_lib.gs_image_loss_workspace_size(131, 97), dtype=torch.uint8, device="cuda")
    got = torch.stack([image_loss(x, a, t, ta, BG, 0.2, 0.8, ws) for _ in range(20)])
    assert bool((got == got[0]).all()) and abs(float(got[0]) - ref) <= 1e-6
