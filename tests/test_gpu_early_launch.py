"""Kernels whose CTAs take their places before the kernel before them has ended:
calls queued behind a producer and before a consumer on one stream, without a
wait between them, give what they give one at a time; grids on either side of
the size up to which the launch is early."""
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


@pytest.mark.parametrize("nv,C", [(300, 8), (20_000, 56), (400_000, 8)])
def test_transforms_between_producers_and_consumers(G, nv, C):
    g = torch.Generator(device="cuda").manual_seed(nv)
    codes = torch.unique(torch.randint(0, 1 << 42, (nv + nv // 8 + 8,), generator=g, device="cuda") >> 3)[:nv].contiguous()
    A = torch.randn(nv, C, generator=g, device="cuda")
    plan = G.RahtPlan(codes, 14, C)
    qps = [G.QuantParams([c % 2 for c in range(C)], [s, 3 * s]) for s in (0.01, 0.2, 0.05)]

    def run(wait):
        out, x, y = [], torch.empty_like(A), torch.empty_like(A)
        for k, qp in enumerate(qps * 3):
            torch.mul(A, 1.0 + 0.25 * k, out=x)
            plan.forward(x, out=y)
            wait()
            x.zero_()
            plan.inverse(y, out=x, qp=qp)
            wait()
            y.fill_(float(k))
            out.append(x.clone())
            wait()
        torch.cuda.synchronize()
        return out

    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        got = run(lambda: None)
    for a, b in zip(got, run(torch.cuda.synchronize)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n", [500, 30_000, 700_000])
def test_frames_back_to_back(G, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    pos, attr = torch.rand(n, 3, generator=g, device="cuda"), torch.randn(n, 11, generator=g, device="cuda")
    qp = G.QuantParams([c % 2 for c in range(11)], [0.05, 0.2])
    want = []
    for k in range(4):
        p = (pos * (1.0 + k)).contiguous()
        torch.cuda.synchronize()
        bs = G.encode_frame(p, attr, 12, qp)[0].clone()
        torch.cuda.synchronize()
        want.append((bs, *[t.clone() for t in G.decode_frame(bs)]))
        torch.cuda.synchronize()
    p = torch.empty_like(pos)
    for k in range(4):
        torch.mul(pos, 1.0 + k, out=p)
        bs = G.encode_frame(p, attr, 12, qp)[0]
        p.fill_(7.0)
        dp, da = G.decode_frame(bs)
        for a, b in zip((bs, dp, da), want[k]):
            assert torch.equal(a, b)
