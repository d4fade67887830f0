"""Octree of a batch, a CTA per run of last-level nodes, against the one-frame
decoder: node counts around a CTA's share, dense octrees (more voxels than are
gathered at a time), depths from 1 to 21, empty frames in between; and bytes
that are not an octree's are refused."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHARE = 1016  # last-level nodes of a CTA


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_05650_gb300 import gsnfs
    return gsnfs


def _chain(n, J, rng):  # n voxels, each the only child of its parent
    x = np.sort(rng.choice(1 << max(J - 1, 1), n, replace=False)) * 2
    return np.stack([x, x[::-1], (x * 7) % (1 << J)], 1).astype(np.float32) / np.float32(1 << J)


def _frames(kind, rng):
    if kind == "edges":
        return [(_chain(n, 13, rng), 13) for n in (1, SHARE - 1, SHARE, SHARE + 1, 2 * SHARE, 2 * SHARE + 1)]
    if kind == "dense":  # every voxel of a cube, and half of one
        g = np.stack(np.meshgrid(*[np.arange(64)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.float32) / 64
        return [(g, 6), (g[rng.random(len(g)) < 0.5], 6), (g[:1], 6)]
    if kind == "depths":
        return [(rng.random((n, 3)).astype(np.float32), J) for n, J in ((3, 1), (40, 2), (5000, 21), (5000, 9), (1, 21), (20_000, 14))]
    return [(np.zeros((0, 3), np.float32), 8), (rng.random((3000, 3)).astype(np.float32), 8), (np.zeros((0, 3), np.float32), 8),
            (rng.random((100_000, 3)).astype(np.float32), 7)]


@pytest.mark.parametrize("kind", ["edges", "dense", "depths", "empty"])
def test_same_as_one_frame(G, kind):
    rng = np.random.default_rng(len(kind))
    qp = G.QuantParams([0, 0, 0], [0.05])
    streams, pos, attr = [], [], []
    for p, J in _frames(kind, rng):
        a = rng.normal(0, 1, (len(p), 3)).astype(np.float32)
        bs = G.encode_frame(torch.from_numpy(p).cuda(), torch.from_numpy(a).cuda(), J, qp)[0]
        dp, da = G.decode_frame(bs)
        streams.append(bs)
        pos.append(dp)
        attr.append(da)
    pad = [torch.cat([b, b.new_zeros(-len(b) % 8)]) for b in streams]
    offs = np.cumsum([0] + [len(b) for b in pad])
    got_p, got_a, rows = G.decode_batch(torch.cat(pad), offs, 3, sum(len(p) for p in pos))
    assert rows.tolist() == np.cumsum([0] + [len(p) for p in pos]).tolist()
    assert torch.equal(got_p, torch.cat(pos)) and torch.equal(got_a, torch.cat(attr))


@pytest.mark.parametrize("change", ["zero byte", "bit more", "bit less", "moved to the level below"])
def test_bytes_of_no_octree_are_refused(G, change):
    J = 6
    p = np.ascontiguousarray(np.random.default_rng(7).random((60, 3)), np.float32)
    pd = torch.from_numpy(p).cuda()
    good = G.encode_frame(pd, None, J, G.geometry_only())[0].cpu().numpy()
    codes = G.voxelize(pd, J)[0].cpu().numpy().astype(np.uint64)
    occ, level = [], []  # breadth first
    for d in range(J):
        parents = codes >> np.uint64(3 * (J - d))
        bits = np.uint64(1) << ((codes >> np.uint64(3 * (J - d - 1))) & np.uint64(7))
        for q in np.unique(parents):
            occ.append(int(np.bitwise_or.reduce(bits[parents == q])))
            level.append(d)
    body = good.tobytes().find(bytes(occ))
    assert body > 0  # so few that the section holds the bytes as they are
    bad, lvl = good.copy(), np.array(level)
    leaf = body + int(np.flatnonzero(lvl == J - 1)[3])
    two = body + next(i for i in range(len(occ)) if lvl[i] == J - 2 and bin(occ[i]).count("1") > 1)
    if change == "zero byte":
        bad[leaf] = 0
    if change in ("bit more", "moved to the level below"):
        bad[leaf] |= 1 if not bad[leaf] & 1 else 2 if not bad[leaf] & 2 else 4
        assert bad[leaf] != good[leaf]
    if change in ("bit less", "moved to the level below"):
        bad[two] &= bad[two] - 1
    one, other = (np.concatenate([b, np.zeros(-len(b) % 8, np.uint8)]) for b in (bad, good))
    with pytest.raises(G.GsnfsError):
        G.decode_batch(torch.from_numpy(np.concatenate([other, one])).cuda(), [0, len(other), 2 * len(other)], 0, 200)
    pos, _, _ = G.decode_batch(torch.from_numpy(np.concatenate([other, other])).cuda(),
                               [0, len(other), 2 * len(other)], 0, 200)
    assert torch.equal(pos[:len(pos) // 2], G.decode_frame(torch.from_numpy(good).cuda())[0])
