"""The RLGR decoder by arithmetic, which takes over from the one by table where
there are many streams of long codewords: frames on both sides of that, and of
both at once (channels of zeros and runs beside channels past the escape),
against the oracle's reading of the same stream; one frame and batches."""
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


# 68,096 streams on 152 SMs: 1,216 row blocks of 32 at 56 channels.  Steps of channels 0-27 / 28-41 / 42-55: one side
# has short codewords throughout, the others long ones, with runs (a step far above the values) or the escape beside
@pytest.mark.parametrize("steps", [(0.3, 0.3, 0.3), (0.004, 0.004, 0.004), (1e-3, 50.0, 0.1), (1e-7, 1e-2, 50.0)])
@pytest.mark.parametrize("n", [38_000, 40_007])
def test_frames(G, orc, n, steps):
    rng = np.random.default_rng(n)
    k = rng.choice(64 ** 3, n, replace=False)  # distinct voxels of a 2^6 grid
    pos = np.stack([k % 64, k // 64 % 64, k // 4096], 1).astype(np.float32)
    pos[:2] = [[0, 0, 0], [64, 64, 64]]
    attr = rng.normal(0, 1, (n, 56)).astype(np.float32)
    groups = np.repeat([0, 1, 2], [28, 14, 14]).astype(np.uint8)
    qp = G.QuantParams(groups, steps, rlgr_block=32)
    bs = G.encode_frame(torch.from_numpy(pos).cuda(), torch.from_numpy(attr).cuda(), 6, qp)[0].clone()
    gpos, gattr = G.decode_frame(bs)
    dec = orc.decode_frame(bs.cpu().numpy())
    assert np.array_equal(gpos.cpu().numpy(), dec["pos"])
    scale = np.sqrt((dec["attr"] ** 2).mean(0)) + np.asarray(steps)[groups]
    err = np.abs(gattr.cpu().numpy().astype(np.float64) - dec["attr"]) / scale  # FP32 dequantisation and transform
    assert err.max() < 1e-4, err.max()
    # the same frame between an empty one and a small one in a batch
    small = (torch.from_numpy(pos[:77]).cuda(), torch.from_numpy(attr[:77]).cuda())
    none = (torch.zeros(0, 3, device="cuda"), torch.zeros(0, 56, device="cuda"))
    frames = [none, (torch.from_numpy(pos).cuda(), torch.from_numpy(attr).cuda()), small, none]
    out, offs = G.encode_batch([f[0] for f in frames], [f[1] for f in frames], [6] * 4, [1.0], qp)
    bpos, battr, rows = G.decode_batch(out, offs, 56, n + 77)
    a, b = int(rows[1]), int(rows[2])
    assert torch.equal(bpos[a:b], gpos) and torch.equal(battr[a:b], gattr)


@pytest.mark.parametrize("cut", [0.3, 0.7, 0.999])
def test_cut_payload(G, cut):
    """A stream whose payload was overwritten with ones from some point on: an error or a decode, no hang."""
    n = 40_000
    g = torch.Generator(device="cuda").manual_seed(1)
    pos, attr = torch.rand(n, 3, generator=g, device="cuda"), torch.randn(n, 56, generator=g, device="cuda")
    bs = G.encode_frame(pos, attr, 12, G.QuantParams(np.zeros(56, np.uint8), [0.004], rlgr_block=32))[0].clone()
    bs[int(cut * bs.numel()):] = 0xFF
    try:
        G.decode_frame(bs)
    except G.GsnfsError:
        pass
    torch.cuda.synchronize()
