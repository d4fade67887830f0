"""What a Gaussian's values make of its pixels where they are not ordinary
numbers: a NaN opacity logit."""
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
