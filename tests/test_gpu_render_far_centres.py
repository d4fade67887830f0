"""Gaussians beside the camera near its plane, whose centres project tens of
thousands to ten million pixels off the image while their footprints cover
it, against the oracle pixel by pixel: in x, in y and in both, to either
side, round in space and drawn out."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

VIEW = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, 0]], dtype=np.float64)
W, H, F = 200, 120, 864.0


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_05650_gb300 import gsnfs
    return gsnfs


def far_scene(off, sx, sy, long):
    """Four Gaussians of camera-space centres (sx, sy) * off * z / F, at depths z just past the near plane: each
    covers the image (the image lies within z / scale standard deviations of its centre)."""
    z = np.array([0.0105, 0.02, 0.05, 0.1])
    attr = np.zeros((4, 56), dtype=np.float32)
    if long:
        # thin across the diagonal that leads to the centre, so that cov_xx cov_yy / det = 3e8, of which the perspective
        # of a round one at this distance makes (off / F)^2 / 2
        sx = sy = sx + sy if sx * sy == 0 else 1
        attr[:, 0:3] = 2.0
        attr[:, 1] -= 0.5 * np.log(3e8 / (0.5 * (off / F) ** 2))
        attr[:, 3:7] = [0.9238795, 0.0, 0.0, 0.3826834]  # 45 degrees about z
    else:
        attr[:, 3] = 1.0
    pos = np.stack([sx * off * z / F, sy * off * z / F, z], 1).astype(np.float32)
    attr[:, 7] = [-1.0, -0.5, 0.0, 0.5]
    attr[:, 8:11] = np.random.default_rng(int(off)).uniform(-1, 2, (4, 3))
    return pos, attr


@pytest.mark.parametrize("long", [False, True])
@pytest.mark.parametrize("sx,sy", [(1, 0), (-1, 0), (0, 1), (0, -1), (1, 1)])
@pytest.mark.parametrize("off", [66e3, 1e5, 1e6, 1e7])
def test_far_centres(G, orc, off, sx, sy, long):
    pos, attr = far_scene(off, sx, sy, long)
    bg = (0.1, 0.2, 0.3)
    want, flag, tol = orc.render(pos, attr, VIEW, F, F, W / 2, H / 2, W, H, bg=bg, check=True)
    assert np.abs(want - np.asarray(bg)).max() > 0.1  # the splats show
    img = G.render(torch.from_numpy(pos).cuda(), torch.from_numpy(attr).cuda(), VIEW, F, F, W / 2, H / 2, W, H,
                   background=bg).cpu().numpy()
    bad = (flag == 0) & (np.abs(img.astype(np.float64) - want).max(axis=2) > tol)
    assert not bad.any(), int(bad.sum())
    assert flag.mean() < 0.05
