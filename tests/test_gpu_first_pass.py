"""First transform pass: the pipelined kernel and the plain pass compute the
same butterflies in the same order, so every result is the same bit for bit,
for any channel count, ragged last tiles, tiles holding several frames and
voxels holding several points."""
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
    yield gsnfs
    for k in gsnfs.TUNABLES:
        gsnfs.tune_set(k, 0)


def both(G, run):
    out = []
    for pipe in (1, 0):
        G.tune_set("raht_pipe", pipe)
        out.append(run())
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("C", [4, 12, 48, 56, 60, 100, 256])
@pytest.mark.parametrize("nv", [1, 256, 257, 20_003, 130_000])
def test_plan(G, nv, C):
    g = torch.Generator(device="cuda").manual_seed(nv + C)
    codes = torch.randint(0, 1 << 42, (nv + nv // 8 + 8,), generator=g, device="cuda") >> 3
    codes = torch.unique(codes)[:nv].contiguous()
    A = torch.randn(nv, C, generator=g, device="cuda")
    qp = G.QuantParams([c % 3 for c in range(C)], [0.1, 0.03, 0.5], tau=0.4)

    def run():
        plan = G.RahtPlan(codes, 14, C)
        Y = plan.forward(A)
        return Y, plan.inverse(Y), plan.inverse(Y, qp=qp)

    both(G, run)


@pytest.mark.parametrize("C,color", [(8, False), (56, False), (56, True)])
@pytest.mark.parametrize("sizes", [(1,), (70_001,), (3, 90, 1, 400, 30_000, 7)])
def test_frames(G, sizes, C, color):
    g = torch.Generator(device="cuda").manual_seed(len(sizes) + C)
    pos = [torch.rand(n, 3, generator=g, device="cuda") for n in sizes]
    attr = [torch.randn(n, C, generator=g, device="cuda") for n in sizes]
    J = [4 if n < 1000 else 5 for n in sizes]  # voxels of several points
    qp = G.QuantParams([c % 2 for c in range(C)], [0.05, 0.2], color=color)

    def run():
        data, offs = G.encode_batch(pos, attr, J, [1.0], qp)
        n = int(offs[-1])
        p, a, rows = G.decode_batch(data[:n], offs, C, sum(sizes))
        return data[:n], p, a

    both(G, run)
