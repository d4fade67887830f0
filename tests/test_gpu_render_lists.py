"""The rasteriser's tile lists against the oracle, pixel by pixel: images of
one, two and three tile-sort passes, wide and tall ones, a single Gaussian,
fewer Gaussians than a warp; footprints from below a pixel to many tiles,
elongated ones, opacities down to below the alpha cut."""
import numpy as np
import pytest

from paper_2606_05650_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_05650_gb300 import gsnfs
    return gsnfs


def _scene(n, seed, spread):
    pos, attr = syn.static_gs_frame(seed, n=n)
    rng = np.random.default_rng(seed + 100)
    if spread:
        attr[:, 0:3] = rng.uniform(-7.5, -1.5, (n, 3)).astype(np.float32)
        attr[:, 7] = rng.normal(-1.0, 4.0, n).astype(np.float32)
    return pos, attr


@pytest.mark.parametrize("n,W,H,f,spread", [(1, 40, 30, 32, False), (31, 16, 16, 13, False), (400, 17, 700, 100, True),
                                            (400, 3000, 16, 200, True), (400, 3000, 16, 2400, False),
                                            (33, 1000, 1100, 880, False), (3000, 130, 90, 104, True)])
def test_lists(G, orc, n, W, H, f, spread):
    pos, attr = _scene(n, n + W, spread)
    view = syn.orbit_views(3)[n % 3]
    bg = (0.2, 0.1, 0.3)
    img = G.render(torch.from_numpy(pos).cuda(), torch.from_numpy(attr).cuda(), view, f, f, W / 2, H / 2, W, H,
                   background=bg).cpu().numpy()
    want, flag, tol = orc.render(pos, attr, view, f, f, W / 2, H / 2, W, H, bg=bg, check=True)
    bad = (flag == 0) & (np.abs(img.astype(np.float64) - want).max(axis=2) > tol)
    assert not bad.any(), int(bad.sum())
    assert flag.mean() < 1e-2  # the oracle could judge nearly every pixel
