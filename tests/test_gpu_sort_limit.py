"""Sorts on both sides of the pair count up to which one launch does all
passes: Morton codes against the oracle, and images, whose lists are by depth
and input index."""
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


@pytest.mark.parametrize("n", [4097, 8191, 8192, 8193, 10_241])
@pytest.mark.parametrize("J", [1, 8, 10, 21])
def test_codes(G, orc, n, J):
    pos = np.random.default_rng(n + J).random((n, 3)).astype(np.float32)
    pos[n // 2:] = pos[: n - n // 2]
    codes, _, _ = G.voxelize(torch.from_numpy(pos).cuda(), J)
    ref = orc.voxelize(pos, np.zeros((n, 1), np.float32), J)[0]
    assert np.array_equal(codes.cpu().numpy().astype(np.uint64), np.asarray(ref).astype(np.uint64))


@pytest.mark.parametrize("n", [8192, 8193])
def test_image(G, orc, n):
    pos, attr = syn.static_gs_frame(n, n=n)
    pos[n // 2:] = pos[: n - n // 2]  # equal depths: input order
    view, W, H = syn.orbit_views(3)[1], 90, 70
    img = G.render(torch.from_numpy(pos).cuda(), torch.from_numpy(attr).cuda(), view, 80, 80, W / 2, H / 2, W, H).cpu().numpy()
    want, flag, tol = orc.render(pos, attr, view, 80, 80, W / 2, H / 2, W, H, check=True)
    bad = (flag == 0) & (np.abs(img.astype(np.float64) - want).max(axis=2) > tol)
    assert not bad.any(), int(bad.sum())
