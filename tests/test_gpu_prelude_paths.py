"""RAHT schedules built by a CTA and by a warp per tile: the transform does not
depend on the tiling, so a plan on either path gives the same coefficients bit
for bit, and the inverse gives the rows back."""
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
    gsnfs.tune_set("raht_tile", 0)
    gsnfs.tune_set("prelude_grid", 0)


@pytest.mark.parametrize("nv,C", [(1, 4), (255, 56), (257, 3), (65_537, 4), (1_400_003, 4)])
@pytest.mark.parametrize("tile,grid", [(256, 0), (256, 1), (512, 0), (1024, 32)])
def test_same_coefficients(G, nv, C, tile, grid):
    g = torch.Generator(device="cuda").manual_seed(nv + C)
    codes = torch.randint(0, 1 << 42, (nv + nv // 8 + 8,), generator=g, device="cuda") >> 3  # a third of the octants
    codes = torch.unique(codes)[:nv].contiguous()
    assert codes.shape[0] == nv
    A = torch.randn(nv, C, generator=g, device="cuda")
    G.tune_set("raht_tile", 0)
    G.tune_set("prelude_grid", 0)
    want = G.RahtPlan(codes, 14, C).forward(A)
    G.tune_set("raht_tile", tile)
    G.tune_set("prelude_grid", grid)
    plan = G.RahtPlan(codes, 14, C)
    got = plan.forward(A)
    assert torch.equal(got, want)
    assert np.isclose(float((got.double() ** 2).sum()), float((A.double() ** 2).sum()), rtol=1e-5)
    assert (plan.inverse(got) - A).abs().max() < 1e-4
