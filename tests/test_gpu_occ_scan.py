"""Octree occupancy of voxel counts at which the scan of the CTAs' counts
takes one turn, exactly one, two, and its most (256 counts a turn, one per 256
voxels), against the oracle byte for byte."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("nv", [1, 255, 256, 2047, 65_279, 65_280, 65_536, 130_816, 400_003])
def test_occupancy(G, orc, nv):
    J = 9
    k = np.random.default_rng(nv).choice(8 ** J, nv, replace=False)
    vox = np.stack([k % 2 ** J, k // 2 ** J % 2 ** J, k // 4 ** J], 1).astype(np.uint32)
    codes = np.sort(orc.morton_codes(vox, J))
    occ, lsz = G.octree_encode(torch.from_numpy(codes.astype(np.int64)).cuda(), J)
    want, wlsz = orc.octree_encode(vox, J)
    assert np.array_equal(lsz, wlsz) and np.array_equal(occ.cpu().numpy(), want)
