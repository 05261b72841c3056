"""k-means assignment through the tensor cores (calls of 1,024 points and 128
centroids on): the same assignment, bit for bit, as the brute-force scan that
smaller calls take, at ragged counts, all widths of a row, ties, duplicates,
values that underflow, and values that are not finite."""
import numpy as np
import pytest
import torch

from paper_2410_16978_gb300 import _lib

pytestmark = pytest.mark.gpu


def _assign(pts, cent, dim, stride, off, n0, n1):
    out = torch.full((n1 - n0,), -2, dtype=torch.int32, device="cuda")
    _lib.gs_kmeans_assign(pts.data_ptr() + 4 * (n0 * stride + off), n1 - n0, dim, stride, cent, cent.shape[0], out,
                          int(torch.cuda.current_stream().cuda_stream))
    return out


def _check(pts, cent, dim, stride, off):
    n = pts.shape[0]
    got = _assign(pts, cent, dim, stride, off, 0, n)
    want = torch.cat([_assign(pts, cent, dim, stride, off, i, min(n, i + 1000)) for i in range(0, n, 1000)])
    torch.cuda.synchronize()
    bad = (got != want).nonzero()
    assert bad.numel() == 0, (bad.numel(), bad[:5, 0].tolist(), got[bad[:5, 0]].tolist(), want[bad[:5, 0]].tolist())


def _data(n, k, dim, stride, off, seed, spread=0.2):
    g = torch.Generator("cuda").manual_seed(seed)
    pts = torch.randn((n, stride), generator=g, device="cuda") * spread
    cent = pts[torch.randperm(n, generator=g, device="cuda")[:k], off:off + dim] * 0.7
    return pts, cent.contiguous()


@pytest.mark.parametrize("n,k,dim,stride,off", [
    (1024, 128, 45, 48, 3), (1025, 129, 45, 48, 3), (1279, 255, 24, 27, 3), (2048, 257, 9, 12, 3),
    (5000, 1000, 48, 48, 0), (4097, 160, 46, 51, 2), (3000, 511, 1, 1, 0), (1500, 1313, 31, 33, 1),
    (30_000, 4096, 45, 48, 3),
])
def test_same_as_the_scan(n, k, dim, stride, off):
    _check(*_data(n, k, dim, stride, off, n + k), dim, stride, off)


def test_centroids_not_16_byte_aligned():
    pts, cent = _data(2000, 301, 45, 48, 3, 5)
    buf = torch.empty(301 * 45 + 1, device="cuda")
    moved = buf[1:].view(301, 45)
    moved.copy_(cent)
    assert moved.data_ptr() % 16 == 4
    _check(pts, moved, 45, 48, 3)


def test_points_equal_to_centroids_and_duplicates():
    pts, cent = _data(6000, 900, 45, 48, 3, 6)
    cent = torch.cat([cent, cent, pts[:300, 3:]]).contiguous()      # every centroid twice, 300 points themselves
    _check(pts, cent, 45, 48, 3)


@pytest.mark.parametrize("case", ["zeros", "constant", "clusters", "tiny", "huge", "nan", "inf", "mixed"])
def test_values_the_bounds_cannot_separate(case):
    dim, stride, off = 45, 48, 3
    pts, cent = _data(3000, 2100, dim, stride, off, 9)
    if case == "zeros":
        pts.zero_()
        cent.zero_()
    elif case == "constant":
        pts.fill_(0.3)
        cent.fill_(0.3)
    elif case == "clusters":                       # a few centres, many points a last bit apart
        pts = (pts[:7].repeat(429, 1) * (1 + 1e-7 * torch.randn((3003, 1), device="cuda"))).contiguous()
        cent = pts[:2100, off:].contiguous()
    elif case == "tiny":
        pts *= 1e-22
        cent *= 1e-22
    elif case == "huge":
        pts[::3] *= 1e17
        cent[::5] *= 1e17
    elif case == "nan":
        pts[5, 10] = float("nan")
        cent[7, 3] = float("nan")
        cent[2000, 0] = float("nan")
    elif case == "inf":
        pts[5, 10] = float("inf")
        cent[7, 3] = float("inf")
        cent[1999] = float("-inf")
    else:
        pts[::2] = 0
        cent[:1500] = 0
    _check(pts, cent, dim, stride, off)


@pytest.mark.parametrize("n,k,dim", [(50_000, 4096, 24), (50_000, 2048, 24), (20_000, 2048, 48), (50_000, 2048, 40)])
def test_same_on_every_run(n, k, dim):
    """Row widths whose reads from shared memory conflict most, so that a row still being read when its buffer is
    filled again would show."""
    g = torch.Generator("cuda").manual_seed(3)
    pal = torch.randn((k, dim), generator=g, device="cuda") * 0.2
    pts = pal[torch.randint(k, (n,), generator=g, device="cuda")]
    pts = pts + 0.02 * torch.randn((n, dim), generator=g, device="cuda")
    cent = pts[torch.randperm(n, generator=g, device="cuda")[:k]].contiguous()
    want = torch.cat([_assign(pts, cent, dim, dim, 0, i, min(n, i + 1000)) for i in range(0, n, 1000)])
    for _ in range(40):
        assert torch.equal(_assign(pts, cent, dim, dim, 0, 0, n), want)


@pytest.mark.parametrize("dim", [1, 2, 3])
@pytest.mark.parametrize("k", [129, 130, 257, 258, 259])
def test_last_tile_of_a_few_values(k, dim):
    """Rows of one to three coordinates: a last tile of one to three centroids may hold fewer values than the
    16-byte unit of the copy that fetches a tile."""
    _check(*_data(1024, k, dim, dim + 1, 1, 10 * k + dim), dim, dim + 1, 1)


def test_release_and_debug_library_in_one_process():
    """Each library sets up its own kernels (their shared memory is above the default limit)."""
    pts, cent = _data(2000, 256, 45, 48, 3, 8)
    _check(pts, cent, 45, 48, 3)
    with _lib.use(_lib.load_debug()):
        _check(pts, cent, 45, 48, 3)
    _check(pts, cent, 45, 48, 3)


@pytest.mark.parametrize("limit", [1, 2, 3, 5, 20])
@pytest.mark.parametrize("k,dim", [(4096, 45), (300, 24), (1000, 46)])
def test_waits_that_run_out(k, dim, limit):
    """Waits cut short (test hook of the debug build) end a CTA's walk with copies and MMAs under way: it lets them
    finish, and its points are scanned in full."""
    lib = _lib.load_debug()
    pts, cent = _data(5000, k, dim, dim + 3, 3, k)
    with _lib.use(lib):
        try:
            _lib.gs_debug_kmeans_wait(limit)
            for _ in range(3):
                _check(pts, cent, dim, dim + 3, 3)
        finally:
            _lib.gs_debug_kmeans_wait(0)
        _check(pts, cent, dim, dim + 3, 3)


@pytest.mark.parametrize("n,k", [(1, 1), (5, 2), (129, 3), (700, 5), (300, 63), (300, 64), (257, 65), (900, 127), (2000, 130),
                                 (1500, 515)])
@pytest.mark.parametrize("dim", [1, 2, 9, 10, 11, 24, 25, 45, 46, 47, 48])
def test_whole_numbers(n, k, dim):
    """Coordinates of -2 .. 2: every distance is exact in single precision and many are equal, so the assignment is
    that of whole-number arithmetic, ties to the lower index, in the scan of every width and behind the tensor cores."""
    rng = np.random.default_rng(1000 * dim + k)
    x, c = rng.integers(-2, 3, (n, dim)), rng.integers(-2, 3, (k, dim))
    want = ((x[:, None, :] - c[None]) ** 2).sum(2).argmin(1)
    pts = torch.full((n, dim + 2), 7.0)
    pts[:, 1:dim + 1] = torch.from_numpy(x).float()
    pts = pts.cuda()
    got = _assign(pts, torch.from_numpy(c).float().cuda(), dim, dim + 2, 1, 0, n)
    assert np.array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("colours,spread", [(64, 0.3), (64, 0.1), (8, 0.1), (4, 0.05), (1, 0.0)])
@pytest.mark.parametrize("n,k,dim", [(6000, 2048, 45), (3000, 500, 24), (2100, 160, 9)])
def test_palettes(n, k, dim, colours, spread):
    """Points around a few colours: more candidates than a point remembers, or too large a share of the centroids."""
    g = torch.Generator("cuda").manual_seed(colours + n)
    pal = torch.randn((colours, dim + 3), generator=g, device="cuda") * 0.2
    pts = pal[torch.randint(colours, (n,), generator=g, device="cuda")]
    pts = pts + 0.2 * spread * torch.randn((n, dim + 3), generator=g, device="cuda")
    cent = pts[torch.randperm(n, generator=g, device="cuda")[:k], 3:].contiguous()
    _check(pts, cent, dim, dim + 3, 3)
