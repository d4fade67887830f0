"""The one-CTA sort of small frames at its edges (a lane, a warp, a round, its
largest size and one more, which takes the grid-wide passes) over every key
width: the distinct Morton codes and the merged frame against the oracle."""
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


@pytest.mark.parametrize("n", [2, 31, 33, 1023, 1024, 1025, 5000, 16384, 16385])
@pytest.mark.parametrize("J", [1, 3, 10, 21])
def test_codes_and_merge(G, orc, n, J):
    rng = np.random.default_rng(n * 100 + J)
    pos = rng.random((n, 3)).astype(np.float32)
    pos[n // 2:] = pos[rng.integers(0, n // 2, n - n // 2)]  # duplicates: equal keys keep their order
    attr = rng.normal(0, 1, (n, 3)).astype(np.float32)
    codes, lo, ext = G.voxelize(torch.from_numpy(pos).cuda(), J)
    ref = orc.encode_frame(pos, attr, J, np.zeros(3, np.uint8), [0.05])
    assert np.array_equal(codes.cpu().numpy().astype(np.uint64), np.asarray(ref["codes"]).astype(np.uint64))
    bs = G.encode_frame(torch.from_numpy(pos).cuda(), torch.from_numpy(attr).cuda(), J,
                        G.QuantParams(np.zeros(3, np.uint8), [0.05]))[0].cpu().numpy()
    dec, want = orc.decode_frame(bs), orc.decode_frame(ref["bitstream"])
    assert np.array_equal(dec["codes"], want["codes"])
    assert (dec["q"] != want["q"]).sum() <= 2  # rounding boundaries only: a wrong merge order moves far more
