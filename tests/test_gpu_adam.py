"""Adam's 16-byte path against its element-wise path."""
import pytest
import torch

from paper_2410_16978_gb300 import DeviceScene, _lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,coeffs", [(1, 1), (5, 16), (171, 4), (4099, 9)])
def test_adam_units_equal_elements(n, coeffs):
    """The 16-byte path against the element-wise one (moments 4 bytes off a
    boundary), bit for bit: arrays shorter than a unit, units that are all
    frozen, all trained and mixed, several blocks with a partial last one.
    Frozen elements keep NaN moments and parameters untouched by NaN gradients."""
    g = torch.Generator("cuda").manual_seed(n)
    deg = {1: 0, 4: 1, 9: 2, 16: 3}[coeffs]
    shapes = [(n, 3), (n, 3), (n, 4), (n,), (n, coeffs, 3)]
    layer = (torch.arange(n, device="cuda") // 3 % 3).to(torch.uint8)
    P = [torch.randn(s, generator=g, device="cuda") for s in shapes]
    M = [0.1 * torch.randn(s, generator=g, device="cuda") for s in shapes]
    V = [0.1 * torch.rand(s, generator=g, device="cuda") for s in shapes]
    G = [torch.randn(s, generator=g, device="cuda") for s in shapes]
    for a in M + G:
        a[layer == 0] = float("nan")

    def run(off):
        m, v = ([torch.empty(a.numel() + off, device="cuda")[off:].view(a.shape).copy_(a) for a in x] for x in (M, V))
        sc = DeviceScene(*[a.clone() for a in P], layer, deg)
        gr, st = _lib.gs_grads(), _lib.gs_adam_state()
        gr.means, gr.log_scales, gr.quats, gr.opacity_logit, gr.sh = (x.data_ptr() for x in G)
        for k in range(5):
            st.m[k], st.v[k] = m[k].data_ptr(), v[k].data_ptr()
        _lib.gs_adam_step(sc.c_struct(), gr, st, (1e-3,) * 5, 0.9, 0.999, 1e-15, 7, 0b110, 0)
        torch.cuda.synchronize()
        return sc.params() + m + v

    for a, b in zip(run(0), run(1)):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
