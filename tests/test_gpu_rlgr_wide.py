"""Ladders of more than 512 streams per row block (rungs x channels, up to the
1,024 that the library accepts), by each of the encoder's kernels: every
rung's stream is that of the rung coded on its own, byte for byte, with the
same distortion sums, and decodes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RUNGS = [1.0, 2.5, 0.1, 30.0, 8.0, 0.01, 4.0, 100.0]


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_05650_gb300 import gsnfs
    return gsnfs


# streams in all (row blocks of 512 x rungs x channels): 1,500 to 61,440, on both sides of the limit (4,864) of the
# kernel that splits the work, and of four times that by points
@pytest.mark.parametrize("n", [700, 4500, 20_000])
@pytest.mark.parametrize("C,rungs", [(171, 3), (129, 4), (65, 8), (256, 3), (128, 8), (256, 4)])
def test_wide_ladder(G, n, C, rungs):
    g = torch.Generator(device="cuda").manual_seed(n + C)
    pos = [torch.rand(n, 3, generator=g, device="cuda"), torch.rand(77, 3, generator=g, device="cuda")]
    attr = [torch.randn(p.shape[0], C + (-C) % 4, generator=g, device="cuda")[:, :C].contiguous() ** 3 for p in pos]
    scales = RUNGS[:rungs]
    qp = G.QuantParams([c % 2 for c in range(C)], [0.1, 0.4])
    out, offs = G.encode_batch(pos, attr, [10, 8], scales, qp)
    _, _, dist = G.encode_batch(pos, attr, [10, 8], scales, qp, distortion=True)
    for r, s in enumerate(scales):
        one, o1 = G.encode_batch(pos, attr, [10, 8], [s], qp)
        _, _, d1 = G.encode_batch(pos, attr, [10, 8], [s], qp, distortion=True)
        for f in range(2):
            k = f * rungs + r
            a = out[int(offs[k]):int(offs[k + 1])]
            assert torch.equal(a, one[int(o1[f]):int(o1[f + 1])]), (f, r)
            assert np.allclose(dist[f, r], d1[f, 0], rtol=1e-12)  # sums of the same terms, in any order
    nv = G.peek_frame(out[int(offs[0]):int(offs[0]) + 96].cpu())[0]
    p, a = G.decode_frame(out[int(offs[0]):int(offs[1])].clone())
    assert p.shape[0] == nv and a.shape == (nv, C)
