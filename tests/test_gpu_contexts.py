"""Contexts on threads and streams of their own whose calls take different
amounts of shared memory in the same kernels: every call succeeds and gives
what it gives alone."""
import ctypes as ct
import threading

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


def _p(t):
    return ct.c_void_p(t.data_ptr())


class RlgrDecode:
    def __init__(self, G, ctx, nv, C, B):
        g = torch.Generator(device="cuda").manual_seed(nv)
        self.want = (torch.randn(nv, C, generator=g, device="cuda") * 3).to(torch.int32)
        self.slots, self.bw = G.rlgr_encode_indices(self.want, B)
        self.out = torch.empty_like(self.want)
        self.f, self.args = G.lib().gsnfs_rlgr_decode_indices, (ctx,)
        self.rest = (_p(self.slots), _p(self.bw), nv, C, B, _p(self.out))

    def call(self, stream):
        return self.f(*self.args, stream, *self.rest)


class Forward:
    def __init__(self, G, ctx, nv, C, _):
        g = torch.Generator(device="cuda").manual_seed(nv)
        codes = G.voxelize(torch.rand(nv, 3, generator=g, device="cuda"), 12)[0].clone()
        self.lib, self.plan = G.lib(), ct.c_void_p()
        assert self.lib.gsnfs_raht_plan_create(ctx, None, _p(codes), codes.shape[0], 12, C, ct.byref(self.plan)) == 0
        self.x = torch.randn(codes.shape[0], C, generator=g, device="cuda")
        self.out = torch.empty_like(self.x)
        assert self.call(None) == 0
        torch.cuda.synchronize()
        self.want = self.out.clone()

    def call(self, stream):
        return self.lib.gsnfs_raht_forward(self.plan, stream, _p(self.x), _p(self.out))


# the decoder's CTAs are smaller for few streams; a tile's rows take more shared memory with more channels
@pytest.mark.parametrize("kind,small,large", [(RlgrDecode, (64, 1, 32), (90_000, 56, 32)), (Forward, (500, 12, 0), (500, 56, 0))])
def test_threads(G, kind, small, large):
    lib = G.lib()
    ctxs = [ct.c_void_p() for _ in range(4)]
    for c in ctxs:
        assert lib.gsnfs_create(ct.byref(c), 0) == 0
    work = [kind(G, c, *(large if k == 0 else small)) for k, c in enumerate(ctxs)]
    streams = [torch.cuda.Stream() for _ in work]
    torch.cuda.synchronize()
    bad, stop = [], threading.Event()

    def run(k):
        s, n = ct.c_void_p(streams[k].cuda_stream), 0
        while n < 8000 if k == 0 else not stop.is_set():
            rc = work[k].call(s)
            n += 1
            if rc != 0:
                bad.append((k, rc))
            if n % 64 == 0:
                streams[k].synchronize()
        if k == 0:
            stop.set()

    threads = [threading.Thread(target=run, args=(k,)) for k in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not bad, (len(bad), bad[:5])
    for w in work:
        assert torch.equal(w.out, w.want)
    for w in work:
        if kind is Forward:
            lib.gsnfs_raht_plan_destroy(w.plan)
    for c in ctxs:
        lib.gsnfs_destroy(c)
