"""Size of a render workspace and the regions of it that callers can see."""
import pytest

from paper_2410_16978_gb300 import _lib


@pytest.mark.parametrize("n,w,h,pairs,most", [
    (500_000, 512, 512, 4_000_000, 186_327_552), (1_200_000, 1024, 1024, 9_600_000, 461_958_656),
    (3_000_000, 2064, 2208, 150_000_000, 5_023_811_840), (4_096, 128, 128, 65_536, 2_928_128),
    (0, 4096, 4096, 0, 413_435_392), (500_000, 800, 800, 1_000_000, 110_245_888)])
def test_size_stays_below_that_without_the_second_copy_of_the_geometry(n, w, h, pairs, most):
    """The compositors read a copy of every Gaussian's geometry (32 bytes) beside its record; the workspace takes no
    more for it, as the sort's and the binning's buffers share their place with what the compositor writes."""
    assert _lib.gs_render_workspace_size(n, w, h, pairs) <= most


@pytest.mark.parametrize("n,w,h,pairs", [(1000, 100, 70, 5000), (1, 1, 1, 0), (70_000, 33, 4096, 10), (5000, 4096, 17, 900_000)])
def test_visible_regions_are_disjoint(n, w, h, pairs):
    size = _lib.gs_render_workspace_size(n, w, h, pairs)
    lay = _lib.gs_workspace_layout(n, w, h, size)
    assert lay["dup_capacity"] >= pairs
    tn = ((w + 15) // 16) * ((h + 15) // 16)
    bytes_of = dict(ctl=128, rec=48 * n, tiles=4 * n, depth=4 * n, list=4 * lay["dup_capacity"], ranges=8 * tn,
                    t_final=4 * w * h, n_contrib=4 * w * h, rec_grad=48 * n)
    spans = sorted((lay[k], lay[k] + v) for k, v in bytes_of.items())
    assert all(a[1] <= b[0] for a, b in zip(spans, spans[1:]))
    assert spans[-1][1] <= lay["total"] <= size
