"""The work this library is used for, as cases that can be timed and checked.

Scenes are shaped like the layered anatomical models the library renders: nested ellipsoid shells of Gaussians (one
layer per shell) of 10^4 to 3 10^6 Gaussians, seen from about four scene radii away, with layers toggled and clip
planes; the smallest is the 4,096-Gaussian cube of the tests.  `exact` evaluates the method's definition in double
precision with plain torch operations: EWA projection, front-to-back compositing of every tile list, the analytic
gradient of the compositing (the projection's by autograd), the image loss, Adam and the k-means round.
"""
import ctypes
import math
from types import SimpleNamespace

import torch

import paper_2410_16978_gb300 as gs
from paper_2410_16978_gb300 import _lib, train

DEV = "cuda"
SHELLS = ((400, 0.9), (300, 0.75), (250, 0.5), (100, 0.4), (150, 0.3))     # relative counts and radii of the layers
FIELDS = ("means", "log_scales", "quats", "opacity_logit", "sh")
LR = (1.6e-4, 5e-3, 1e-3, 5e-2, 2.5e-3)
PRUNE_AT = 0.005


def _view(name, n, w, h, **more):
    c = {"name": name, "kind": "view", "n": n, "w": w, "h": h, "deg": 3, "layers": 5, "mask": 31, "planes": 0,
         "dist": 4.0, "sh": "f32", "sr": "f32", "views": 1}
    c.update(more)
    return c


def listed():
    return [
        # the library's smallest scene through its default call: launch latency
        _view("view_128", 4096, 128, 128, deg=0, layers=2),
        # one served request of the small resident model, one clip plane
        _view("view_512", 500_000, 512, 512, planes=1),
        # a compressed model (16-bit storage) in a window of odd size, two clip planes
        _view("view_16bit_1037x771", 1_500_000, 1037, 771, planes=2, sh="f16", sr="bf16"),
        # a model with the SH codebook at a desktop resolution
        _view("view_codebook_1920x1080", 1_200_000, 1920, 1080, sh="cb", sr="f16"),
        # the large model close up at one headset eye's resolution, every layer on: the longest lists
        _view("view_2064x2208_near", 3_000_000, 2064, 2208, dist=3.6),
        # the headset frame: both eyes of the large model, two layers toggled on, one depth order for both eyes
        _view("stereo_2064x2208", 3_000_000, 2064, 2208, kind="stereo", mask=0b10100, planes=1),
        # continuous batching: eight small views of one resident model in one call
        _view("batch_8x512", 500_000, 512, 512, kind="batch", views=8),
        # forward, backward with blend weights and the contribution prune of one full frame
        _view("frame_1024", 1_200_000, 1024, 1024, kind="frame", mask=0b01111, planes=1),
        # a training step's forward, image loss and backward through autograd, every layer trainable
        _view("train_800", 500_000, 800, 800, kind="train", layers=3, mask=0b111),
        # the same on a small model and a ragged image, low SH degree
        _view("train_397x243", 40_000, 397, 243, kind="train", layers=3, mask=0b111, deg=1),
        # the optimiser's update of that training step
        {"name": "adam_500k", "kind": "adam", "n": 500_000, "deg": 3, "layers": 3, "frozen": 0b001},
        # one Lloyd round of the codebook over the usual sample, SH degree 3
        {"name": "kmeans_200k_16k", "kind": "kmeans", "n": 200_000, "k": 16384, "deg": 3},
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("view", "view", "view", "stereo", "batch", "frame", "frame", "train", "train", "adam", "kmeans"))
    deg = rng.choice((0, 1, 2, 3, 3, 3))
    if kind == "adam":
        return {"kind": kind, "n": _spread(rng, 20_000, 1_200_000), "deg": deg, "layers": 3,
                "frozen": rng.choice((0, 0b001, 0b011))}
    if kind == "kmeans":
        return {"kind": kind, "n": _spread(rng, 20_000, 200_000), "k": _spread(rng, 256, 16384), "deg": max(1, deg)}
    c = _view("", _spread(rng, 4096, 3_000_000), _spread(rng, 96, 2208), _spread(rng, 96, 2208), kind=kind, deg=deg,
              layers=5, mask=rng.randint(1, 31), planes=rng.randint(0, 2), dist=round(rng.uniform(3.6, 5.0), 2))
    del c["name"]
    if kind in ("view", "stereo", "batch"):
        c["sh"] = rng.choice(("f32", "f32", "f16", "bf16") + (("cb",) if deg > 0 else ()))
        c["sr"] = rng.choice(("f32", "f32", "f16", "bf16"))
    if kind == "stereo":                                         # an eye's image is upright, as in a headset
        c.update(w=min(c["w"], c["h"]), h=max(c["w"], c["h"]))
    if kind == "batch":
        c.update(n=min(c["n"], 500_000), w=min(c["w"], 800), h=min(c["h"], 800), views=rng.randint(2, 8))
    if kind in ("frame", "train"):
        c.update(n=min(c["n"], 1_200_000), w=min(c["w"], 1400), h=min(c["h"], 1400))
    if kind == "train":
        c.update(layers=3, mask=0b111, planes=0)
    return c


# ---------------------------------------------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(DEV).manual_seed(int(seed))


def _scene_arrays(case, g):
    """The model as float32 tensors: means, log-scales, quaternions, opacity logits, SH [n, K, 3], layer."""
    n, K = case["n"], (case["deg"] + 1) ** 2
    if case["n"] <= 4096:                                        # the small cube
        means = torch.rand((n, 3), generator=g, device=DEV) * 2 - 1
        ls = torch.randn((n, 3), generator=g, device=DEV) * 0.5 - 3.5
        sh = torch.zeros((n, K, 3), device=DEV)
        sh[:, 0] = (torch.rand((n, 3), generator=g, device=DEV) * 2 - 1) * math.sqrt(math.pi)
        layer = (torch.arange(n, device=DEV) * case["layers"] // n).to(torch.uint8)
    else:
        shells = SHELLS[: case["layers"]]
        total = sum(c for c, _ in shells)
        edges = [round(n * sum(c for c, _ in shells[:i]) / total) for i in range(len(shells) + 1)]
        layer = torch.zeros(n, dtype=torch.uint8, device=DEV)
        radius = torch.zeros((n, 1), device=DEV)
        for i, (_, r) in enumerate(shells):
            layer[edges[i]:edges[i + 1]] = i
            radius[edges[i]:edges[i + 1]] = r
        d = torch.randn((n, 3), generator=g, device=DEV)
        d = d / d.norm(dim=1, keepdim=True).clamp_min(1e-6)
        radius = radius * (1 + 0.02 * torch.randn((n, 1), generator=g, device=DEV))
        means = d * radius * torch.tensor([1.0, 0.8, 1.25], device=DEV)
        ls = torch.randn((n, 3), generator=g, device=DEV) * 0.7 - 4.5
        sh = torch.randn((n, K, 3), generator=g, device=DEV) * 0.2
    q = torch.randn((n, 4), generator=g, device=DEV)
    q = q / q.norm(dim=1, keepdim=True).clamp_min(1e-6)
    ol = torch.randn(n, generator=g, device=DEV)
    return means.contiguous(), ls, q, ol, sh, layer


def _camera(eye, w, h, shift=0.0):
    """Pinhole camera at `eye` looking at the origin (50 degrees across), moved by `shift` along its x axis."""
    def unit(v):
        s = math.sqrt(sum(x * x for x in v))
        return [x / s for x in v]

    def cross(a, b):
        return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]
    z = unit([-x for x in eye])
    x = unit(cross(z, [0.0, 1.0, 0.0] if abs(z[1]) < 0.999 else [0.0, 0.0, 1.0]))
    y = cross(z, x)
    R = torch.tensor([x, y, z], dtype=torch.float32)
    t = [-sum(r[i] * eye[i] for i in range(3)) for r in (x, y, z)]
    t[0] -= shift
    f = 0.5 * w / math.tan(math.radians(25.0))
    return SimpleNamespace(R=R.tolist(), t=torch.tensor(t, dtype=torch.float32).tolist(),
                           fx=ctypes.c_float(f).value, fy=ctypes.c_float(f).value, cx=0.5 * w, cy=0.5 * h,
                           width=w, height=h, znear=ctypes.c_float(0.2).value)


def _direction(g):
    v = torch.randn(3, generator=g, device=DEV).double().tolist()
    s = math.sqrt(sum(x * x for x in v))
    return [x / s for x in v]


def _inputs(case, seed):
    """Everything a call takes, the same for `prepare` and `exact`."""
    g = _gen(seed)
    s = SimpleNamespace()
    if case["kind"] == "kmeans":
        K = (case["deg"] + 1) ** 2
        s.sh = torch.randn((case["n"], K, 3), generator=g, device=DEV) * 0.2
        pick = torch.randperm(case["n"], generator=g, device=DEV)[: min(case["k"], case["n"])]
        # centroids as after a few rounds: near a sample, drawn towards the mean
        s.cent = (s.sh[pick, 1:].reshape(len(pick), -1) * 0.7).contiguous()
        return s
    s.means, s.log_scales, s.quats, s.opacity_logit, s.sh, s.layer = _scene_arrays(case, g)
    if case["kind"] == "adam":
        s.grads = [torch.randn(p.shape, generator=g, device=DEV) * 1e-3 for p in
                   (s.means, s.log_scales, s.quats, s.opacity_logit, s.sh)]
        s.m = [torch.randn(p.shape, generator=g, device=DEV) * 1e-3 for p in s.grads]
        s.v = [torch.rand(p.shape, generator=g, device=DEV) * 1e-5 + 1e-8 for p in s.grads]
        return s
    dt = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
    s.log_scales, s.quats = s.log_scales.to(dt[case["sr"]]), s.quats.to(dt[case["sr"]])
    s.index = s.table = None
    if case["sh"] == "cb":
        K = (case["deg"] + 1) ** 2
        rows = min(16384, case["n"])
        s.table = torch.zeros((rows, (3 * (K - 1) + 7) // 8 * 8), dtype=torch.float16, device=DEV)
        s.table[:, : 3 * (K - 1)] = (torch.randn((rows, 3 * (K - 1)), generator=g, device=DEV) * 0.2).half()
        s.index = torch.randint(0, rows, (case["n"],), generator=g, device=DEV).to(torch.int16)
        s.sh = s.sh[:, 0].contiguous()                           # the DC coefficient stays per Gaussian
    else:
        s.sh = s.sh.to(dt[case["sh"]])
    s.planes = []
    for _ in range(case["planes"]):
        nrm = torch.tensor(_direction(g), dtype=torch.float32).tolist()
        s.planes.append((nrm, ctypes.c_float(float(torch.rand(1, generator=g, device=DEV)) * 0.6 - 0.3).value, 0xFFFFFFFF))
    s.bg = tuple(torch.rand(3, generator=g, device=DEV).tolist())
    w, h = case["w"], case["h"]
    eyes = [[case["dist"] * x for x in _direction(g)] for _ in range(case["views"])]
    s.cams = [_camera(e, w, h) for e in eyes]
    if case["kind"] == "stereo":
        s.cams = [_camera(eyes[0], w, h, -0.032), _camera(eyes[0], w, h, 0.032)]
    if case["kind"] == "frame":                                  # upstream gradients of an unnormalised loss
        s.d_image = torch.randn((3, h, w), generator=g, device=DEV)
        s.d_alpha = torch.randn((h, w), generator=g, device=DEV)
    if case["kind"] == "train":                                  # a smooth target close to what the model shows
        yy, xx = torch.meshgrid(torch.arange(h, device=DEV) / h, torch.arange(w, device=DEV) / w, indexing="ij")
        a = torch.rand(4, 4, generator=g, device=DEV)
        wave = torch.stack([torch.sin(6.28 * (2 * a[i, 0] * xx + 2 * a[i, 1] * yy + a[i, 2])) for i in range(4)])
        s.target_alpha = (0.6 + 0.4 * wave[3]).clamp(0, 1).contiguous()
        s.target_rgb = ((0.5 + 0.4 * wave[:3] + 0.05 * torch.randn((3, h, w), generator=g, device=DEV)).clamp(0, 1)
                        * s.target_alpha).contiguous()
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s.case = case
    if case["kind"] == "kmeans":
        s.dim = s.cent.shape[1]
        s.k = s.cent.shape[0]
        s.assign = torch.empty(case["n"], dtype=torch.int32, device=DEV)
        s.moved = s.cent.clone()                                 # an empty cluster keeps its centroid
        s.scratch = torch.empty(_lib.gs_kmeans_scratch_size(s.k, s.dim), dtype=torch.uint8, device=DEV)
        return s
    s.scene = gs.DeviceScene(s.means, s.log_scales, s.quats, s.opacity_logit, s.sh, s.layer, case["deg"],
                             case.get("sh", "f32"), case.get("sr", "f32"), sh_index=getattr(s, "index", None),
                             sh_table=getattr(s, "table", None))
    if case["kind"] == "adam":
        s.step = 10
        return s
    # one workspace per view in flight, sized by rendering the view once with the overflow check on
    s.rasts = []
    for cam in s.cams:
        r = gs.Rasterizer(case["n"], case["w"], case["h"])
        r.render(s.scene, cam, case["mask"], s.planes, s.bg)
        s.rasts.append(r)
    h, w = case["h"], case["w"]
    s.images = [torch.empty((3, h, w), device=DEV) for _ in s.cams]
    s.alphas = [torch.empty((h, w), device=DEV) for _ in s.cams]
    if case["kind"] == "batch":
        s.c_scene = s.scene.c_struct()
    if case["kind"] in ("frame", "train"):
        s.contrib_sum = torch.zeros(case["n"], device=DEV)
        s.contrib_max = torch.zeros(case["n"], device=DEV)
    if case["kind"] == "frame":
        s.grads = {f: torch.empty(p.shape, device=DEV) for f, p in zip(FIELDS, s.scene.params())}
    if case["kind"] == "train":
        for p in s.scene.params():
            p.requires_grad_(True)
        s.loss_ws = torch.empty(_lib.gs_image_loss_workspace_size(w, h), dtype=torch.uint8, device=DEV)
    return s


# ---------------------------------------------------------------------------------------------------- one pass

def _stream():
    return int(torch.cuda.current_stream().cuda_stream)


def _run_view(s):
    c = s.case
    if c["n"] <= 4096:                                           # a first program's call: everything at its default
        return s.rasts[0].render(s.scene, s.cams[0], c["mask"], s.planes, s.bg)
    return s.rasts[0].render(s.scene, s.cams[0], c["mask"], s.planes, s.bg, s.images[0], s.alphas[0], check=False)


def _run_stereo(s):
    a, b = s.rasts
    _lib.gs_render_stereo(s.scene.c_struct(), gs.make_camera(s.cams[0]), gs.make_camera(s.cams[1]), s.case["mask"],
                          s.planes, s.bg, a.workspace, a.ws_bytes, b.workspace, b.ws_bytes, s.images[0], s.alphas[0],
                          s.images[1], s.alphas[1], True, _stream())
    return s.images[0], s.alphas[0], s.images[1], s.alphas[1]


def _run_batch(s):
    gs.gs_render_batch([dict(scene=s.c_scene, camera=gs.make_camera(cam), layer_mask=s.case["mask"], planes=s.planes,
                             bg=s.bg, workspace=r.workspace, ws_bytes=r.ws_bytes, image=i, alpha=a)
                        for cam, r, i, a in zip(s.cams, s.rasts, s.images, s.alphas)], _stream())
    return s.images + s.alphas


def _run_frame(s):
    r, cam, c = s.rasts[0], s.cams[0], s.case
    r.render(s.scene, cam, c["mask"], s.planes, s.bg, s.images[0], s.alphas[0], check=False)
    r.backward(s.scene, cam, s.bg, s.d_image, s.d_alpha, 0xFFFFFFFF, s.contrib_sum, s.contrib_max, s.grads)
    keep, _, n_keep = gs.contrib_prune(s.contrib_max, PRUNE_AT)
    return [s.images[0], s.alphas[0], [s.grads[f] for f in FIELDS], s.contrib_sum, s.contrib_max, keep, n_keep]


def _run_train(s):
    for p in s.scene.params():
        p.grad = None
    image, alpha = gs.render(s.scene, s.rasts[0], s.cams[0], s.case["mask"], s.planes, s.bg, 0xFFFFFFFF,
                             s.contrib_sum, s.contrib_max)
    loss = train.image_loss(image, alpha, s.target_rgb, s.target_alpha, s.bg, 0.2, 0.8, s.loss_ws)
    loss.backward()
    return [image.detach(), alpha.detach(), [p.grad for p in s.scene.params()], s.contrib_sum, s.contrib_max,
            loss.detach()]


def _run_adam(s):
    g, st = _lib.gs_grads(), _lib.gs_adam_state()
    g.means, g.log_scales, g.quats, g.opacity_logit, g.sh = (x.data_ptr() for x in s.grads)
    for k in range(5):
        st.m[k], st.v[k] = s.m[k].data_ptr(), s.v[k].data_ptr()
    _lib.gs_adam_step(s.scene.c_struct(), g, st, LR, 0.9, 0.999, 1e-15, s.step, 0xFFFFFFFF & ~s.case["frozen"],
                      _stream())
    s.step += 1
    return [s.scene.params(), s.m, s.v]


def _run_kmeans(s):
    row = 3 * (s.case["deg"] + 1) ** 2
    pts = s.sh.data_ptr() + 12                                   # the coefficients after the DC term
    _lib.gs_kmeans_assign(pts, s.case["n"], s.dim, row, s.cent, s.k, s.assign, _stream())
    _lib.gs_kmeans_update(pts, s.case["n"], s.dim, row, s.assign, s.k, s.moved, s.scratch, s.scratch.numel(), _stream())
    return s.assign, s.moved


RUN = {"view": _run_view, "stereo": _run_stereo, "batch": _run_batch, "frame": _run_frame, "train": _run_train,
       "adam": _run_adam, "kmeans": _run_kmeans}


def run(state):
    return RUN[state.case["kind"]](state)


# ---------------------------------------------------------------------------------------------------- work

def work(case):
    n, K = case["n"], (case["deg"] + 1) ** 2
    if case["kind"] == "kmeans":
        dim, k = 3 * (K - 1), min(case["k"], n)
        return {"bytes": 4.0 * (n * dim + n + 2 * k * dim), "flops": 3.0 * n * k * dim}
    width = 11 + 3 * K
    if case["kind"] == "adam":
        part = 1 - sum(c for i, (c, _) in enumerate(SHELLS[:3]) if case["frozen"] >> i & 1) / sum(c for c, _ in SHELLS[:3])
        return {"bytes": n * (28.0 * width * part + 1), "flops": n * 14.0 * width * part}
    shells = SHELLS[: case["layers"]]
    seen = sum(c for i, (c, _) in enumerate(shells) if case["mask"] >> i & 1) / sum(c for c, _ in shells)
    size = {"f32": 4, "f16": 2, "bf16": 2, "cb": 0}
    sh = 12 + 2 if case["sh"] == "cb" else 3 * K * size[case["sh"]]
    scene = n * (12.0 + 4 + 1 + seen * (7 * size[case["sr"]] + sh))
    px = float(case["w"] * case["h"])
    eyes = 2 if case["kind"] == "stereo" else case["views"]
    # about 25 blends of 24 flops a pixel (the alpha and the blend), five times that with the backward
    b, f = scene + eyes * 16 * px, eyes * px * 25 * 24
    if case["kind"] in ("frame", "train"):
        b += scene + 4.0 * n * width + 16 * n + 16 * px
        f *= 5
    if case["kind"] == "train":
        b += 32 * px
        f += 3 * px * 350
    return {"bytes": b, "flops": f + eyes * n * seen * 400}


# ---------------------------------------------------------------------------------------------------- in 64 bits

def _sh_basis(d, deg):
    x, y, z = d.unbind(1)
    b = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if deg > 0:
        c = math.sqrt(3 / (4 * math.pi))
        b += [-c * y, c * z, -c * x]
    if deg > 1:
        c = math.sqrt(15 / (4 * math.pi))
        b += [c * x * y, -c * y * z, math.sqrt(5 / (16 * math.pi)) * (2 * z * z - x * x - y * y), -c * x * z,
              c / 2 * (x * x - y * y)]
    if deg > 2:
        a, m, o = math.sqrt(35 / (32 * math.pi)), math.sqrt(105 / (4 * math.pi)), math.sqrt(21 / (32 * math.pi))
        b += [-a * y * (3 * x * x - y * y), m * x * y * z, -o * y * (4 * z * z - x * x - y * y),
              math.sqrt(7 / (16 * math.pi)) * z * (2 * z * z - 3 * x * x - 3 * y * y),
              -o * x * (4 * z * z - x * x - y * y), m / 2 * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(b, 1)


def _project(P, case, s, cam):
    """The splats of the Gaussians that are drawn: their indices, records [V, 9] (centre, conic, opacity, colour;
    differentiable in the parameters P), depths and tile rectangles."""
    f8 = torch.float64
    R, t = torch.tensor(cam.R, dtype=f8, device=DEV), torch.tensor(cam.t, dtype=f8, device=DEV)
    with torch.no_grad():
        keep = (torch.tensor(case["mask"], device=DEV) >> s.layer.long()) & 1 > 0
        for nrm, d, _ in s.planes:
            keep &= P[0] @ torch.tensor(nrm, dtype=f8, device=DEV) + d >= 0
        keep &= P[0] @ R[2] + t[2] > cam.znear
        idx = keep.nonzero()[:, 0]
    mean, ls, q, ol = (p[idx] for p in P[:4])
    p = mean @ R.T + t
    z = p[:, 2]
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, zz = q.unbind(1)
    rot = torch.stack([1 - 2 * (y * y + zz * zz), 2 * (x * y - w * zz), 2 * (x * zz + w * y), 2 * (x * y + w * zz),
                       1 - 2 * (x * x + zz * zz), 2 * (y * zz - w * x), 2 * (x * zz - w * y), 2 * (y * zz + w * x),
                       1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    M = rot * ls.exp()[:, None, :]
    lx, ly = 1.3 * 0.5 * cam.width / cam.fx, 1.3 * 0.5 * cam.height / cam.fy
    ix, iy = p[:, 0] / z, p[:, 1] / z
    o = torch.zeros_like(z)
    J = torch.stack([cam.fx / z, o, -cam.fx * ix.clamp(-lx, lx) / z, o, cam.fy / z, -cam.fy * iy.clamp(-ly, ly) / z],
                    1).view(-1, 2, 3)
    TM = (J @ R) @ M
    S = TM @ TM.transpose(1, 2)
    a, b, c = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    det = a * c - b * b
    u, v = cam.fx * ix + cam.cx, cam.fy * iy + cam.cy
    tx, ty = (cam.width + 15) // 16, (cam.height + 15) // 16
    with torch.no_grad():
        mid = 0.5 * (a + c)
        r = (3 * (mid + (mid * mid - det).clamp_min(0.1).sqrt()).sqrt()).ceil()
        x0, y0 = ((u - r) / 16).trunc().clamp(0, tx), ((v - r) / 16).trunc().clamp(0, ty)
        x1, y1 = ((u + r + 15) / 16).trunc().clamp(0, tx), ((v + r + 15) / 16).trunc().clamp(0, ty)
        on = ((det > 0) & (x1 > x0) & (y1 > y0)).nonzero()[:, 0]
        rect = torch.stack([x0, y0, x1, y1], 1)[on].long()
    deg, K = case["deg"], (case["deg"] + 1) ** 2
    who = idx[on]
    if case["sh"] == "cb":
        rest = s.table.double()[s.index[who].long() & 0xFFFF][:, : 3 * (K - 1)].view(-1, K - 1, 3)
        sh = torch.cat([P[4][who][:, None, :], rest], 1)
    else:
        sh = P[4][who]
    d = mean[on] + R.T @ t
    basis = _sh_basis(d / d.norm(dim=1, keepdim=True), deg)
    rgb = ((basis[:, :, None] * sh).sum(1) + 0.5).clamp_min(0)
    rec = torch.cat([torch.stack([u, v, c / det, -b / det, a / det], 1)[on], torch.sigmoid(ol[on])[:, None], rgb], 1)
    return who, rec, z.detach()[on].float(), rect


def _lists(depth, rect, tx, tn):
    """The splats of every tile in depth order: one list and each tile's first position in it."""
    order = torch.sort(depth, stable=True)[1]
    r = rect[order]
    w, h = r[:, 2] - r[:, 0], r[:, 3] - r[:, 1]
    cnt = w * h
    at = torch.repeat_interleave(torch.arange(len(order), device=DEV), cnt)
    k = torch.arange(len(at), device=DEV) - (cnt.cumsum(0) - cnt)[at]
    wa = w[at]
    tile = ((r[at, 1] + torch.div(k, wa, rounding_mode="floor")) * tx + r[at, 0] + k % wa).int()
    del k, wa
    tile, by = torch.sort(tile, stable=True)
    first = torch.searchsorted(tile, torch.arange(tn + 1, device=DEV, dtype=torch.int32))
    return order[at[by]].int(), first


class _Walk:
    """Front-to-back walk over all tiles, `step` list positions of the tiles still open at a time."""

    def __init__(self, rec, ids, first, cam, step=32, most=1024):
        self.rec, self.ids, self.first, self.step, self.most = rec, ids, first, step, most
        self.tx, self.ty = (cam.width + 15) // 16, (cam.height + 15) // 16
        tn = self.tx * self.ty
        px = torch.arange(256, device=DEV)
        t = torch.arange(tn, device=DEV)
        self.x = ((t % self.tx) * 16)[:, None] + (px % 16)[None, :]
        self.y = (torch.div(t, self.tx, rounding_mode="floor") * 16)[:, None] + (px // 16)[None, :]
        self.inside = (self.x < cam.width) & (self.y < cam.height)
        self.tn = tn

    def __call__(self, visit, C):
        """visit(tiles, ids, ok, dx, dy, ex, alpha, on, T) for each part; C carries what the caller adds up."""
        T = torch.ones((self.tn, 256), dtype=torch.float64, device=DEV)
        open_ = self.inside.clone()
        length = self.first[1:] - self.first[:-1]
        at = 0
        while True:
            live = ((length > at) & open_.any(1)).nonzero()[:, 0]
            if not len(live):
                return T
            for k in range(0, len(live), self.most):
                tl = live[k:k + self.most]
                pos = at + torch.arange(self.step, device=DEV)
                ok = pos[None, :] < length[tl][:, None]
                ids = self.ids[(self.first[tl][:, None] + pos).clamp_max(len(self.ids) - 1)].long()
                q = self.rec[ids]
                dx = self.x[tl][:, None, :] + 0.5 - q[..., 0:1]
                dy = self.y[tl][:, None, :] + 0.5 - q[..., 1:2]
                ex = (-0.5 * (q[..., 2:3] * dx * dx + 2 * q[..., 3:4] * dx * dy + q[..., 4:5] * dy * dy)).exp()
                al = (q[..., 5:6] * ex).clamp_max(0.99)
                hit = (al >= 1 / 255) & ok[:, :, None] & open_[tl][:, None, :]
                Tinc = T[tl][:, None, :] * torch.where(hit, 1 - al, torch.ones_like(al)).cumprod(1)
                on = hit & (Tinc >= 1e-4)                        # T only falls: all after the stop fail too
                stop = hit & ~on
                f = torch.where(on, 1 - al, torch.ones_like(al))
                Tb = T[tl][:, None, :] * f.cumprod(1) / f        # before each splat
                visit(tl, ids, q, dx, dy, ex, al, on, Tb)
                T[tl] = Tb[:, -1] * f[:, -1]
                open_[tl] = open_[tl] & ~stop.any(1)
            at += self.step


def _composite(rec, depth, rect, cam, bg):
    tx, ty = (cam.width + 15) // 16, (cam.height + 15) // 16
    ids, first = _lists(depth, rect, tx, tx * ty)
    walk = _Walk(rec, ids, first, cam)
    C = torch.zeros((walk.tn, 256, 3), dtype=torch.float64, device=DEV)

    def visit(tl, ids, q, dx, dy, ex, al, on, T):
        w = torch.where(on, al * T, torch.zeros_like(al))
        C[tl] += torch.einsum("tsp,tsc->tpc", w, q[..., 6:9])
    T = walk(visit, C) if len(ids) else torch.ones((walk.tn, 256), dtype=torch.float64, device=DEV)
    C = C + T[..., None] * torch.tensor(bg, dtype=torch.float64, device=DEV)
    return walk, C, T


def _to_image(a, cam):
    tx, ty = (cam.width + 15) // 16, (cam.height + 15) // 16
    a = a.view(ty, tx, 16, 16, -1).permute(4, 0, 2, 1, 3).reshape(-1, ty * 16, tx * 16)
    return a[:, : cam.height, : cam.width]


def _to_tiles(img, cam):
    tx, ty = (cam.width + 15) // 16, (cam.height + 15) // 16
    full = torch.zeros((img.shape[0], ty * 16, tx * 16), dtype=torch.float64, device=DEV)
    full[:, : cam.height, : cam.width] = img
    return full.view(-1, ty, 16, tx, 16).permute(1, 3, 2, 4, 0).reshape(ty * tx, 256, -1)


def _backward(walk, C, T, cam, bg, d_image, d_alpha, V):
    """Gradients of the records [V, 9], and each splat's sum and largest blend weight."""
    f8 = torch.float64
    dC, dA = _to_tiles(d_image.double(), cam), _to_tiles(d_alpha.double()[None], cam)[..., 0]
    g = torch.zeros((V, 9), dtype=f8, device=DEV)
    csum, cmax = torch.zeros(V, dtype=f8, device=DEV), torch.zeros(V, dtype=f8, device=DEV)
    left = C.clone()                                             # colour behind (with the background)

    def visit(tl, ids, q, dx, dy, ex, al, on, Tb):
        w = torch.where(on, al * Tb, torch.zeros_like(al))
        dc = torch.einsum("tpc,tsc->tsp", dC[tl], q[..., 6:9])
        behind = torch.einsum("tpc,tpc->tp", left[tl], dC[tl])[:, None, :] - (w * dc).cumsum(1)
        da = Tb * dc - (behind - (dA * T)[tl][:, None, :]) / (1 - al)
        da = torch.where(on, da, torch.zeros_like(da))
        do = torch.where(q[..., 5:6] * ex < 0.99, da, torch.zeros_like(da))
        de = do * q[..., 5:6] * ex
        part = torch.stack([(de * (q[..., 2:3] * dx + q[..., 3:4] * dy)).sum(2),
                            (de * (q[..., 3:4] * dx + q[..., 4:5] * dy)).sum(2), (-0.5 * de * dx * dx).sum(2),
                            (-de * dx * dy).sum(2), (-0.5 * de * dy * dy).sum(2), (do * ex).sum(2)], 2)
        part = torch.cat([part, torch.einsum("tsp,tpc->tsc", w, dC[tl])], 2)
        g.index_add_(0, ids.reshape(-1), part.reshape(-1, 9))
        csum.index_add_(0, ids.reshape(-1), w.sum(2).reshape(-1))
        cmax.scatter_reduce_(0, ids.reshape(-1), w.amax(2).reshape(-1), "amax")
        left[tl] -= torch.einsum("tsp,tsc->tpc", w, q[..., 6:9])
    if V:
        walk(visit, left)
    return g, csum, cmax


def _loss(X, A, s):
    """0.8 L1 + 0.2 (1 - SSIM) + 0.8 L1(alpha); 11x11 Gaussian window (sigma 1.5), zero outside the image."""
    bg = torch.tensor(s.bg, dtype=torch.float64, device=DEV)[:, None, None]
    Y = s.target_rgb.double() + (1 - s.target_alpha.double()) * bg
    g = torch.exp(-(torch.arange(11, dtype=torch.float64, device=DEV) - 5) ** 2 / 4.5)
    g = (g / g.sum()).tolist()

    def win(v):
        h, w = v.shape[1:]
        v = torch.nn.functional.pad(v, (5, 5, 5, 5))
        v = sum(g[i] * v[:, :, i:i + w] for i in range(11))
        return sum(g[i] * v[:, i:i + h] for i in range(11))
    mx, my = win(X), win(Y)
    sx, sy, sxy = win(X * X) - mx * mx, win(Y * Y) - my * my, win(X * Y) - mx * my
    ssim = (2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sx + sy + 9e-4))
    return 0.8 * (X - Y).abs().mean() + 0.2 * (1 - ssim.mean()) + 0.8 * (A - s.target_alpha.double()).abs().mean()


def _exact_kmeans(case, s):
    x = s.sh[:, 1:].reshape(case["n"], -1).double()
    c = s.cent.double()
    near = torch.cat([((c * c).sum(1) - 2 * (p @ c.T)).argmin(1) for p in x.split(16384)])
    total = torch.zeros_like(c).index_add_(0, near, x)
    count = torch.zeros(len(c), dtype=torch.float64, device=DEV).index_add_(0, near, torch.ones_like(x[:, 0]))
    return None, torch.where(count[:, None] > 0, total / count.clamp_min(1)[:, None], c)


def _exact_adam(case, s):
    on = (0xFFFFFFFF & ~case["frozen"]) >> s.layer.long() & 1 > 0
    ps, ms, vs = [], [], []
    for p, g, m, v, lr in zip((s.means, s.log_scales, s.quats, s.opacity_logit, s.sh), s.grads, s.m, s.v, LR):
        p, g, m, v = p.double(), g.double(), m.double(), v.double()
        k = on.view(-1, *([1] * (p.dim() - 1)))
        m2, v2 = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p2 = p - lr / (1 - 0.9 ** 10) * m2 / ((v2 / (1 - 0.999 ** 10)).sqrt() + 1e-15)
        ps, ms, vs = ps + [torch.where(k, p2, p)], ms + [torch.where(k, m2, m)], vs + [torch.where(k, v2, v)]
    return [ps, ms, vs]


def exact(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "kmeans":
        return _exact_kmeans(case, s)
    if case["kind"] == "adam":
        return _exact_adam(case, s)
    P = [p.double() for p in (s.means, s.log_scales, s.quats, s.opacity_logit, s.sh)]
    back = case["kind"] in ("frame", "train")
    for p in P:
        p.requires_grad_(back)
    images, alphas = [], []
    for cam in s.cams:
        with torch.set_grad_enabled(back):
            who, rec, depth, rect = _project(P, case, s, cam)
        with torch.no_grad():
            walk, C, T = _composite(rec.detach(), depth, rect, cam, s.bg)
            images.append(_to_image(C, cam).contiguous())
            alphas.append(_to_image(1 - T, cam)[0].contiguous())
    if case["kind"] == "view":
        return images[0], alphas[0]
    if case["kind"] == "stereo":
        return images[0], alphas[0], images[1], alphas[1]
    if case["kind"] == "batch":
        return images + alphas
    loss = None
    if case["kind"] == "train":
        X, A = images[0].clone().requires_grad_(True), alphas[0].clone().requires_grad_(True)
        loss = _loss(X, A, s)
        loss.backward()
        s.d_image, s.d_alpha, loss = X.grad, A.grad, loss.detach()
    with torch.no_grad():
        g, vsum, vmax = _backward(walk, C, T, cam, s.bg, s.d_image, s.d_alpha, len(rec))
    rec.backward(g)
    csum, cmax = torch.zeros(case["n"], dtype=torch.float64, device=DEV), torch.zeros(case["n"], dtype=torch.float64, device=DEV)
    csum[who], cmax[who] = vsum, vmax
    out = [images[0], alphas[0], [p.grad for p in P], csum, cmax]
    return out + ([loss] if loss is not None else [None, None])
