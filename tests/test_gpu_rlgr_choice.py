"""Frames whose points are too many for the encoder of few streams, whose
voxels may not be: on both sides of its limit (152 SMs x 32 streams: 4,864) the
bytes are those of the frame inside a batch of far more streams."""
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


# voxels: 2,744 to 110k of at most n points; blocks of 32 rows
@pytest.mark.parametrize("C,rungs", [(56, [1.0]), (3, [1.0, 8.0, 0.1])])
@pytest.mark.parametrize("J,side", [(4, 14), (5, 25), (5, 32), (6, 64)])
def test_same_bytes(G, C, rungs, J, side):
    n = 5_000 if C == 56 else 60_000  # 8,792 and 16,875 streams by points
    g = torch.Generator(device="cuda").manual_seed(side)
    pos = torch.randint(0, side, (n, 3), generator=g, device="cuda").float()
    pos[0], pos[1] = 0.0, 2.0 ** J
    attr = torch.randn(n, C, generator=g, device="cuda")
    qp = G.QuantParams([0] * C, [0.05], rlgr_block=32)
    one, offs = G.encode_batch([pos], [attr], [J], rungs, qp)
    copies = 6
    many, moffs = G.encode_batch([pos] * copies, [attr] * copies, [J] * copies, rungs, qp)
    for f in (0, copies - 1):
        for r in range(len(rungs)):
            k = f * len(rungs) + r
            assert torch.equal(one[int(offs[r]):int(offs[r + 1])], many[int(moffs[k]):int(moffs[k + 1])]), (f, r)
