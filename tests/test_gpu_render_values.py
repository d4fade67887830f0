"""What a Gaussian's values make of its pixels: the rounding of colours and
opacities (evaluated in FP64, rounded once to FP32), and values that are not
ordinary numbers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

VIEW = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, 0]], dtype=np.float64)


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_05650_gb300 import gsnfs
    return gsnfs


def test_nan_opacity_covers_its_tiles(G):
    """alpha = min(0.99, NaN) = 0.99 at every pixel of the 16 x 16 tiles that the footprint square overlaps."""
    a = np.zeros((1, 56), dtype=np.float32)
    a[0, 0:3] = np.log(0.1)  # 10 pixels at z = 1: radius ceil(3 sqrt(100.3 + sqrt(0.1))) = 31, tiles 2 .. 5
    a[0, 3] = 1.0
    a[0, 7] = np.nan
    p = np.array([[0, 0, 1.0]], dtype=np.float32)
    img = G.render(torch.from_numpy(p).cuda(), torch.from_numpy(a).cuda(), VIEW, 100.0, 100.0, 64.0, 64.0, 128, 128,
                   background=(0.0, 0.0, 0.0)).cpu().numpy()
    want = np.zeros((128, 128, 3), dtype=np.float32)
    want[32:96, 32:96] = np.float32(0.5) * np.float32(0.99)
    assert np.array_equal(img, want)


def _grid(G, attr, side):
    """Image of side x side splats of 0.3 square pixels, each alone at its pixel (alpha at two pixels' distance is below
    the cut) and exactly at its centre: pixel (2 i, 2 j) is colour * min(0.99, opacity)."""
    i, j = np.meshgrid(np.arange(side), np.arange(side))
    f = 2048.0
    pos = np.stack([2 * i / f, 2 * j / f, np.ones_like(i)], -1).reshape(-1, 3).astype(np.float32)
    attr[:, 0:3] = -12.0
    attr[:, 3] = 1.0
    img = G.render(torch.from_numpy(pos).cuda(), torch.from_numpy(attr).cuda(), VIEW, f, f, 0.5, 0.5, 2 * side, 2 * side,
                   background=(0.0, 0.0, 0.0)).cpu().numpy()
    return pos, img[::2, ::2].reshape(-1, 3)


def _basis(d):
    x, y, z = d.T
    pi = np.arccos(np.asarray(-1, dtype=d.dtype))
    c1, c2a, c2b, c2c = np.sqrt(3 / (4 * pi)), 0.5 * np.sqrt(15 / pi), 0.25 * np.sqrt(5 / pi), 0.25 * np.sqrt(15 / pi)
    c3a, c3b, c3c = 0.25 * np.sqrt(35 / (2 * pi)), 0.5 * np.sqrt(105 / pi), 0.25 * np.sqrt(21 / (2 * pi))
    c3d, c3e = 0.25 * np.sqrt(7 / pi), 0.25 * np.sqrt(105 / pi)
    return np.stack([np.full_like(x, 0.5 / np.sqrt(pi)), -c1 * y, c1 * z, -c1 * x, c2a * x * y, -c2a * y * z,
                     c2b * (2 * z * z - x * x - y * y), -c2a * x * z, c2c * (x * x - y * y),
                     -c3a * y * (3 * x * x - y * y), c3b * x * y * z, -c3c * y * (4 * z * z - x * x - y * y),
                     c3d * z * (2 * z * z - 3 * x * x - 3 * y * y), -c3c * x * (4 * z * z - x * x - y * y),
                     c3e * z * (x * x - y * y), -c3a * x * (x * x - 3 * y * y)], -1)


def test_colours_are_rounded_from_fp64(G):
    """Dark colours, sums of 16 terms that cancel to 1e-6 .. 0.1.  Every pixel's float is that of a number within 2^-46
    of the terms' magnitudes of the exact sum, as an FP64 evaluation's is; and as FP64's usual error is below 2^-53 of the
    magnitudes (32 roundings of some 2^-55 of partial sums that are a quarter of them, of random signs), no more floats
    differ from the exact sum's than an error of 2^-53 would let differ."""
    side = 512
    rng = np.random.default_rng(3)
    n = side * side
    a = np.zeros((n, 56), dtype=np.float32)
    a[:, 7] = 30.0  # opacity 1: alpha 0.99
    a[:, 11:] = rng.normal(0, 0.3, (n, 45))
    i, j = np.meshgrid(np.arange(side), np.arange(side))
    L = np.longdouble
    d = np.stack([2 * i / 2048, 2 * j / 2048, np.ones_like(i)], -1).reshape(-1, 3).astype(L)
    Y = _basis(d / np.sqrt((d * d).sum(1, keepdims=True)))
    want = np.empty((n, 3), dtype=L)
    mag = np.empty((n, 3))
    for c in range(3):
        ac = a[:, 11 + 15 * c:26 + 15 * c].astype(L)
        rest = (Y[:, 1:] * ac).sum(1) + L(0.5)
        a[:, 8 + c] = (10 ** rng.uniform(-6, -1, n) - rest) / Y[:, 0]
        want[:, c] = Y[:, 0] * a[:, 8 + c].astype(L) + rest
        mag[:, c] = 0.5 + np.abs(a[:, 8 + c]) + np.abs(ac).sum(1)
    _, img = _grid(G, a, side)
    lo, mid, hi = (np.maximum(w, 0).astype(np.float32) * np.float32(0.99)
                   for w in (want - 2.0 ** -46 * mag, want, want + 2.0 ** -46 * mag))
    bad = (img < lo) | (img > hi)
    assert not bad.any(), int(bad.sum())
    on = mid > 0
    expected = (2.0 ** -53 * mag[on] / np.spacing(mid[on].astype(np.float64).astype(np.float32))).clip(0, 1).sum()
    assert (img != mid)[on].sum() <= expected, (int((img != mid)[on].sum()), float(expected))


def test_opacities_are_rounded_from_fp64(G):
    side = 512
    a = np.zeros((side * side, 56), dtype=np.float32)  # colour 0.5
    a[:, 7] = np.random.default_rng(4).normal(0, 2, side * side).clip(-5, 4)  # above the alpha cut, below 0.99
    _, img = _grid(G, a, side)
    op = 1.0 / (1.0 + np.exp(-a[:, 7].astype(np.float64)))
    lo, hi = (op * (1 - 2.0 ** -50)).astype(np.float32), (op * (1 + 2.0 ** -50)).astype(np.float32)
    assert ((img[:, 0] >= 0.5 * lo) & (img[:, 0] <= 0.5 * hi)).all()


def test_infinite_and_huge_coefficients(G):
    """An infinite coefficient makes its colour infinite, or 0 where the product is negative or not a number; the rest
    are as FP64 has them."""
    a = np.zeros((16, 56), dtype=np.float32)
    a[:, 7] = 30.0
    a[1, 11] = np.inf   # times -y = -0: not a number
    a[2, 12] = np.inf   # times z > 0
    a[3, 12] = -np.inf
    a[5, 8] = np.nan
    a[6, 8:11] = [3e38, -3e38, 1e38]
    _, img = _grid(G, a, 4)
    want = np.full((16, 3), np.float32(0.5) * np.float32(0.99))
    want[1, 0] = 0.0
    want[2, 0] = np.inf
    want[3, 0] = 0.0
    want[5, 0] = 0.0
    c0 = 0.5 / np.sqrt(np.pi)
    want[6] = np.maximum(np.float64(np.float32([3e38, -3e38, 1e38])) * c0 + 0.5, 0).astype(np.float32) * np.float32(0.99)
    assert np.array_equal(img, want)
