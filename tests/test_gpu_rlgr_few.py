"""The RLGR encoder for few streams against the one for many: a frame encoded
on its own (few streams) and as one of many copies in a batch (more than the
count at which the encoder changes) gives the same bytes, over block sizes
around a segment, partial blocks, stream counts that do not fill a CTA, run
mode, long prefixes and the escape, several rungs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FEW = 20_000  # streams (row blocks x rungs x channels)


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_05650_gb300 import gsnfs
    return gsnfs


@pytest.mark.parametrize("n,C,B,rungs", [(161, 56, 32, [1.0]), (3407, 3, 32, [1.0]), (1000, 56, 64, [1.0]),
                                         (1411, 56, 512, [1.0, 30.0]), (515, 67, 128, [1.0]), (5003, 120, 2048, [1.0]),
                                         (2600, 120, 512, [1.0, 4.0, 0.02, 9.0])])
@pytest.mark.parametrize("step", [1e-6, 0.02, 1.0, 6.0])
def test_same_bytes(G, n, C, B, rungs, step):
    g = torch.Generator(device="cuda").manual_seed(n + C)
    pos = torch.rand(n, 3, generator=g, device="cuda")
    attr = torch.randn(n, C, generator=g, device="cuda") ** 3
    qp = G.QuantParams([c % 3 for c in range(C)], [step, 3 * step, 0.4 * step], rlgr_block=B)
    one, offs = G.encode_batch([pos], [attr], [10], rungs, qp)
    streams = -(-n // B) * len(rungs) * C
    copies = min(64, FEW // streams + 2)
    many, moffs = G.encode_batch([pos] * copies, [attr] * copies, [10] * copies, rungs, qp)
    assert streams <= FEW < copies * streams
    for f in (0, copies - 1):
        for r in range(len(rungs)):
            a = one[int(offs[r]):int(offs[r + 1])]
            k = f * len(rungs) + r
            assert torch.equal(a, many[int(moffs[k]):int(moffs[k + 1])]), (f, r)
