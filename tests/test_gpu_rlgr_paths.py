"""The RLGR coders' code paths against the oracle, byte for byte: codewords by
table and beyond it (long prefixes, the escape, every Golomb-Rice parameter),
run mode, warps whose lanes are in different modes, blocks of different
lengths in one warp; and whole frames on both sides of the stream count at
which the encoder changes kernels."""
import numpy as np
import pytest

from parity import compare_stream
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


def _indices(kind, nv, C, rng):
    if kind == "zeros":
        return np.zeros((nv, C), np.int32)
    if kind == "runs":
        return (rng.integers(-3, 4, (nv, C)) * (rng.random((nv, C)) < 0.02)).astype(np.int32)
    if kind == "table edge":  # magnitudes around the tables' largest, after small ones and after large ones
        return (rng.choice([0, 1, 125, 126, 127, 128, 129, 4000], (nv, C)) * rng.choice([-1, 1], (nv, C))).astype(np.int32)
    if kind == "huge":
        return rng.integers(-2 ** 31, 2 ** 31, (nv, C)).astype(np.int32) >> rng.integers(0, 31, (nv, C)).astype(np.int32)
    scale = 10.0 ** rng.uniform(-1.5, 3.5, C)  # each channel of its own size: mixed modes and parameters in a warp
    return np.round(rng.laplace(0, 1.0, (nv, C)) * scale).astype(np.int32)


@pytest.mark.parametrize("kind", ["zeros", "runs", "table edge", "huge", "mixed"])
@pytest.mark.parametrize("nv,C,B", [(5, 1, 32), (515, 56, 256), (1027, 33, 512), (700, 200, 64), (4101, 3, 2048)])
def test_indices_byte_identical(G, orc, kind, nv, C, B):
    rng = np.random.default_rng(nv + C + len(kind))
    q = _indices(kind, nv, C, rng)
    q[q == -2 ** 31] = 0
    slots, bw = G.rlgr_encode_indices(torch.from_numpy(q).cuda(), B)
    words, lens = slots.cpu().numpy().view(np.uint32), bw.cpu().numpy()
    sw = G.rlgr_slot_words(B)
    for k in range(lens.size):
        b, c = divmod(k, C)
        ref = orc.rlgr_encode(q[b * B:(b + 1) * B, c])
        assert lens[k] == ref.size and np.array_equal(words[k * sw:k * sw + ref.size], ref), (b, c)
    assert np.array_equal(G.rlgr_decode_indices(slots, bw, nv, C, B).cpu().numpy(), q)


@pytest.mark.parametrize("n,scale", [(182_200, 1.0), (183_000, 1.0), (183_000, 12.0)])
def test_frames_around_the_kernel_change(G, orc, n, scale):
    pos, attr = syn.DynamicScene(3).frame(0, n=n)
    groups, steps = syn.gs_channel_groups(), syn.GS_BASE_STEPS * scale
    bs = G.encode_frame(torch.from_numpy(pos).cuda(), torch.from_numpy(attr).cuda(), 14, G.QuantParams(groups, steps))[0]
    gpos, gattr = G.decode_frame(bs)
    compare_stream(orc, bs.cpu().numpy(), pos, attr, 14, groups, steps, 0.5, 512, 4096,
                   gpu_decoded=(gpos.cpu().numpy(), gattr.cpu().numpy()))
