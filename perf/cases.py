"""Workloads of the GS-NFS codec: what a program that uses this framework has it do.

Each case is one call (or one layer's forward and backward) through the public
entry points of paper_2606_05650_gb300.gsnfs: frames encoded and decoded one
at a time and in batches, from ten thousand Gaussians to sixteen frames of a
million, three-channel point clouds, the colour-decorrelated mode with the
encoder's reconstruction, the bandwidth ladder, the differentiable attribute
codec and the splat rasteriser.

Frames are drawn on the GPU from the case's seed with the shapes and
distributions of paper_2606_05650_gb300.synthetic: Gaussians on moving, warped
parametric surfaces (plus a uniform part for static scenes) with 3DGS
attributes, and points on capsule figures with smooth colour.  `exact` is the
codec's reconstruction, the layer's result and the rendered image evaluated in
64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_05650_gb300 import gsnfs
from paper_2606_05650_gb300 import synthetic as syn

DEVICE = "cuda"
GS_CHANNELS = syn.GS_CHANNELS
CLOUD_CHANNELS = 3
CLOUD_STEP = 0.05
RUNG_SCALES = [float(s) for s in syn.LADDER_RUNG_SCALES]
BYTES_PER_POINT = {"gs": 33.0, "colour": 19.0, "cloud": 0.6}  # typical stream size at the base steps
LADDER_STREAM_SHARE = [1.0, 0.80, 0.60, 0.39, 0.25]           # of it at each rung


# ---- the cases ------------------------------------------------------------------
def _frame(kind, n, J, scene, colour=False, recon=False, block=512, tau=0.5):
    return {"kind": kind, "n": n, "J": J, "scene": scene, "colour": colour, "recon": recon, "block": block, "tau": tau}


def _batch(kind, frames, n_lo, n_hi, sizes, J, scene="dynamic", rungs=1, block=512):
    return {"kind": kind, "frames": frames, "n_lo": n_lo, "n_hi": n_hi, "sizes": sizes, "J": J, "scene": scene,
            "rungs": rungs, "block": block}


def listed():
    cases = []

    def add(name, case):
        case["name"] = name
        cases.append(case)

    # a small static asset (an object, an avatar's head), coded on its own: launches and waits count
    add("frame_10k_encode", _frame("encode", 10_000, 10, "static"))
    add("frame_10k_decode", _frame("decode", 10_000, 10, "static"))
    # one frame of a live 30 fps Gaussian sequence, sent and received as it comes
    add("frame_250k_encode", _frame("encode", 247_313, 16, "dynamic"))
    add("frame_250k_decode", _frame("decode", 247_313, 16, "dynamic"))
    # captured point clouds of two people on a 10-bit grid, YCbCr: a frame as it is captured, four for playback
    add("cloud_1m_encode", _frame("encode", 1_000_000, 10, "cloud"))
    add("cloud_4x1m_decode", _batch("decode_batch", 4, 1_000_000, 1_000_000, 0, 10, scene="cloud"))
    # a large scene stored with SH colour decorrelation, the encoder returning the decoded frame
    add("colour_1m_encode_recon", _frame("encode", 1_000_000, 16, "dynamic", colour=True, recon=True))
    # sixteen frames of a sequence at a time, for a server that stores or forwards them
    add("batch_16x1m_encode", _batch("encode_batch", 16, 1_000_000, 1_000_000, 0, 16))
    add("batch_16x1m_decode", _batch("decode_batch", 16, 1_000_000, 1_000_000, 0, 16))
    # eight frames of very different sizes and depths at five quantisation rungs, for adaptive streaming
    add("ladder_8x5_encode", _batch("encode_batch", 8, 50_000, 2_000_000, 5, 0, rungs=5))
    # one step of compression-aware fine-tuning through the attribute codec
    add("codec_layer_500k", {"kind": "layer", "n": 500_003, "J": 16})
    # a decoded frame drawn for a viewer
    add("render_1m_960x540", {"kind": "render", "n": 1_000_000, "width": 960, "height": 540})
    return cases


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["encode", "encode", "decode", "decode", "cloud", "cloud", "colour", "batch", "batch", "ladder",
                       "layer", "render"])
    block = rng.choice([256, 512, 512, 1024])
    if kind in ("encode", "decode"):
        n = _log_int(rng, 3_000, 1_500_000)
        J = rng.randint(10, 12) if n < 30_000 else rng.randint(13, 18)
        return _frame(kind, n, J, rng.choice(["static", "dynamic"]), recon=kind == "encode" and rng.random() < 0.3,
                      block=block, tau=rng.choice([0.5, 0.5, 1.0 / 3.0]))
    if kind == "cloud":
        n, J = _log_int(rng, 50_000, 2_000_000), rng.randint(9, 11)
        if rng.random() < 0.5:
            return _frame("encode", n, J, "cloud", block=block)
        return _batch("decode_batch", rng.randint(1, 6), n * 4 // 5, n, rng.randint(0, 999), J, scene="cloud", block=block)
    if kind == "colour":
        return _frame(rng.choice(["encode", "decode"]), _log_int(rng, 50_000, 1_000_000), rng.randint(14, 17), "dynamic",
                      colour=True, recon=rng.random() < 0.5)
    if kind == "batch":
        n = _log_int(rng, 100_000, 1_000_000)
        return _batch(rng.choice(["encode_batch", "decode_batch"]), rng.randint(3, 16), n * 9 // 10, n,
                      rng.randint(0, 999), rng.randint(14, 18), block=block)
    if kind == "ladder":
        return _batch("encode_batch", rng.randint(2, 8), 50_000, _log_int(rng, 200_000, 1_500_000), rng.randint(0, 999), 0,
                      rungs=rng.randint(2, 5), block=block)
    if kind == "layer":
        return {"kind": "layer", "n": _log_int(rng, 20_000, 1_000_000), "J": rng.randint(13, 17)}
    return {"kind": "render", "n": _log_int(rng, 8_000, 1_000_000), "width": rng.randint(200, 1280),
            "height": rng.randint(150, 720)}


# ---- frames ----------------------------------------------------------------------
class _Rand:
    """Random numbers of one seed: bulk draws on the GPU, a scene's few parameters on the host."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEVICE).manual_seed(int(seed))
        self.h = np.random.default_rng(int(seed))

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device=DEVICE)

    def uniform(self, lo, hi, *shape):
        return torch.rand(*shape, generator=self.g, device=DEVICE) * (hi - lo) + lo

    def perm(self, n):
        return torch.randperm(n, generator=self.g, device=DEVICE)


def _rotation(r):
    q, _ = np.linalg.qr(r.h.normal(size=(3, 3)))
    return torch.tensor(q, dtype=torch.float32, device=DEVICE)


def _vec(v):
    return torch.tensor(np.asarray(v), dtype=torch.float32, device=DEVICE)


def _surface_points(r, n, uniform):
    """n points: a sphere, a torus, a cylinder and a plane patch, rotated, warped and jittered; the share `uniform`
    spread over the unit cube."""
    nu = int(round(uniform * n))
    m = n - nu
    counts = r.h.multinomial(m, [0.3, 0.3, 0.2, 0.2])
    parts = []
    for s, k in enumerate(int(c) for c in counts):
        if s == 0:
            v = r.normal(k, 3)
            p = 0.15 * v / v.norm(dim=1, keepdim=True).clamp_min(1e-12)
        elif s == 1:
            u, w = r.uniform(0, 2 * math.pi, k), r.uniform(0, 2 * math.pi, k)
            p = torch.stack([(0.14 + 0.05 * w.cos()) * u.cos(), (0.14 + 0.05 * w.cos()) * u.sin(), 0.05 * w.sin()], 1)
        elif s == 2:
            u, h = r.uniform(0, 2 * math.pi, k), r.uniform(-0.15, 0.15, k)
            p = torch.stack([0.07 * u.cos(), 0.07 * u.sin(), h], 1)
        else:
            p = torch.stack([r.uniform(-0.2, 0.2, k), r.uniform(-0.2, 0.2, k), torch.zeros(k, device=DEVICE)], 1)
        p = p @ _rotation(r)
        p = p + float(r.h.uniform(0.005, 0.02)) * torch.sin(_vec(r.h.uniform(4, 12, 3)) * p[:, [1, 2, 0]])
        parts.append(p + _vec(r.h.uniform(0.3, 0.7, 3)))
    pos = torch.cat(parts)
    pos = pos + 1e-3 * r.normal(m, 3)
    if nu:
        pos = torch.cat([pos, r.uniform(0.0, 1.0, nu, 3)])
    return pos[r.perm(n)].contiguous()


def _gs_attributes(r, n, correlated=False):
    a = r.normal(n, GS_CHANNELS)
    a[:, 0:3] = a[:, 0:3] * 0.5 - 4.0
    a[:, 3:7] /= a[:, 3:7].norm(dim=1, keepdim=True).clamp_min(1e-12)
    a[:, 7] *= 2.0
    a[:, 8:11] *= 0.5
    a[:, 11:56] *= 0.05
    if correlated:  # SH colours sharing a luminance, energy falling with the degree, functions mixed
        mix = _vec(np.random.default_rng(12345).normal(0, 1, (15, 15)) * 0.35 + np.eye(15))
        sig = _vec(0.08 / np.array([1] * 3 + [2] * 5 + [3] * 7))
        w = (0.95, 1.0, 0.9)
        lum = (r.normal(n, 15) * sig) @ mix.T
        for col in range(3):
            a[:, 11 + 15 * col:26 + 15 * col] = lum * w[col] + r.normal(n, 15) * (0.15 * sig)
        a[:, 8:11] = 0.5 * r.normal(n, 1) * _vec(w) + 0.05 * r.normal(n, 3)
    return a


_BONES = [[0.0, 0.0, 0.9, 0.0, 0.0, 1.45, 0.12], [0.0, 0.0, 1.5, 0.0, 0.0, 1.7, 0.09],
          [0.0, -0.2, 1.4, 0.0, -0.45, 1.1, 0.04], [0.0, -0.45, 1.1, 0.0, -0.55, 0.8, 0.035],
          [0.0, 0.2, 1.4, 0.0, 0.45, 1.1, 0.04], [0.0, 0.45, 1.1, 0.0, 0.55, 0.8, 0.035],
          [0.0, -0.1, 0.9, 0.0, -0.12, 0.45, 0.06], [0.0, -0.12, 0.45, 0.0, -0.12, 0.02, 0.05],
          [0.0, 0.1, 0.9, 0.0, 0.12, 0.45, 0.06], [0.0, 0.12, 0.45, 0.0, 0.12, 0.02, 0.05]]


def _cloud_frame(r, n):
    """n points on two capsule figures with swung limbs, YCbCr colours in [0, 1]."""
    counts = r.h.multinomial(n, np.full(20, 1 / 20))
    parts = []
    for fig in range(2):
        swing = 0.3 * math.sin(float(r.h.uniform(0, 6.28)))
        for bi, b in enumerate(_BONES):
            k = int(counts[10 * fig + bi])
            a, e, rad = np.array(b[0:3]), np.array(b[3:6]), b[6]
            if bi >= 2:
                c, s = math.cos(swing if bi % 2 == 0 else -swing), math.sin(swing if bi % 2 == 0 else -swing)
                e = a + np.array([[c, 0, s], [0, 1, 0], [-s, 0, c]]) @ (e - a)
            d = (e - a) / np.linalg.norm(e - a)
            e1 = np.cross(d, [1.0, 0, 0] if abs(d[0]) < 0.9 else [0, 1.0, 0])
            e1 /= np.linalg.norm(e1)
            e2 = np.cross(d, e1)
            u, th = r.uniform(0, 1, k, 1), r.uniform(0, 2 * math.pi, k, 1)
            parts.append(_vec(a + [0, fig - 0.5, 0]) + u * _vec(e - a) + rad * (th.cos() * _vec(e1) + th.sin() * _vec(e2)))
    pos = torch.cat(parts)
    lo, hi = pos.amin(0), pos.amax(0)
    pos = (pos - lo) / (hi - lo).amax()
    f = 2 * math.pi
    rgb = torch.stack([128 + 90 * torch.sin(f * 1.3 * pos[:, 0] + 0.5) * torch.cos(f * 0.7 * pos[:, 2]),
                       128 + 90 * torch.sin(f * 0.9 * pos[:, 1] + 1.1), 128 + 90 * torch.cos(f * 1.1 * pos[:, 2])], 1)
    rgb = (rgb + 4.0 * r.normal(n, 3)).round().clamp(0, 255)
    R, G, B = rgb[:, 0], rgb[:, 1], rgb[:, 2]
    attr = torch.stack([0.299 * R + 0.587 * G + 0.114 * B, 128 - 0.168736 * R - 0.331264 * G + 0.5 * B,
                        128 + 0.5 * R - 0.418688 * G - 0.081312 * B], 1) / 255.0
    p = r.perm(n)
    return pos[p].contiguous(), attr[p].contiguous()


def _in_distinct_voxels(pos, J, n):
    """Indices of n points that lie in n voxels of the grid of all points, those that span the grid among them."""
    lo, hi = pos.amin(0), pos.amax(0)
    v = ((pos.double() - lo.double()) * ((1 << J) / float((hi.double() - lo.double()).amax()))).floor().long()
    v = v.clamp_max((1 << J) - 1)
    key = (v[:, 0] << (2 * J)) | (v[:, 1] << J) | v[:, 2]
    rank = torch.arange(pos.shape[0], device=pos.device)
    rank[((pos == lo) | (pos == hi)).any(1)] -= pos.shape[0]
    order = torch.argsort(rank)
    _, first = torch.unique(key[order], return_inverse=True)
    head = torch.full((int(first.amax()) + 1,), pos.shape[0], device=pos.device)
    head.scatter_reduce_(0, first, torch.arange(pos.shape[0], device=pos.device), "amin")
    return order[head.sort()[0][:n]]


def _one_frame(seed, n, scene, colour=False, voxels=0):
    """Positions and attributes of n points, in n distinct voxels of a grid of depth `voxels` where one is given (a
    stream holds voxels, so its decoder sees n of them)."""
    r = _Rand(seed)
    if scene == "cloud":
        return _cloud_frame(r, n)
    pos = _surface_points(r, n + (n // 16 + 64 if voxels else 0), 0.3 if scene == "static" else 0.0)
    if voxels:
        pos = pos[_in_distinct_voxels(pos, voxels, n)][r.perm(n)].contiguous()
    return pos, _gs_attributes(r, n, correlated=colour)


def _case_frame(case, seed):
    fixed = case["kind"] == "decode" or case["recon"]
    return _one_frame(seed, case["n"], case["scene"], case["colour"], case["J"] if fixed else 0)


def _batch_shape(case):
    """Sizes and depths of a batch's frames: log-uniform sizes, depths 16, 17, 18 in turn where the case gives none."""
    rng = np.random.default_rng(int(case["sizes"]))
    F = case["frames"]
    n = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), F)).round().astype(int)
    J = [case["J"] or 16 + f % 3 for f in range(F)]
    return [min(max(int(v), case["n_lo"]), case["n_hi"]) for v in n], J


def _batch_frames(case, seed):
    n, J = _batch_shape(case)
    frames = [_one_frame(seed * 1000 + f, n[f], case["scene"]) for f in range(len(n))]
    return [p for p, _ in frames], [a for _, a in frames], J


def _gs_quant(block=512, tau=0.5, colour=False):
    return gsnfs.QuantParams(syn.gs_channel_groups(), syn.GS_BASE_STEPS, tau=tau, rlgr_block=block, color=colour)


def _quant(case):
    if case.get("scene") == "cloud":
        return gsnfs.QuantParams(np.zeros(CLOUD_CHANNELS, np.uint8), [CLOUD_STEP], rlgr_block=case["block"])
    return _gs_quant(case["block"], case.get("tau", 0.5), case.get("colour", False))


def _stream_bytes(case, n):
    """Typical size of the streams of n points."""
    kind = "cloud" if case.get("scene") == "cloud" else "colour" if case.get("colour") else "gs"
    return BYTES_PER_POINT[kind] * n * sum(LADDER_STREAM_SHARE[:case.get("rungs", 1)])


def _room(case, n):
    """Bytes that hold those streams with room to spare."""
    return int(1.5 * _stream_bytes(case, n)) + 65536 * case.get("frames", 1) * case.get("rungs", 1)


def _camera(width, height):
    f = 0.9 * width
    return syn.orbit_views(3)[1], f, f, width / 2.0, height / 2.0


# ---- what a program holds, and one pass ---------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("encode", "decode"):
        pos, attr = _case_frame(case, seed)
        qp = _quant(case)
        if kind == "decode":
            return {"case": case, "stream": gsnfs.encode_frame(pos, attr, case["J"], qp)[0].clone()}
        out = torch.zeros(gsnfs.max_bitstream_bytes(case["n"], case["J"], qp), dtype=torch.uint8, device=DEVICE)
        return {"case": case, "pos": pos, "attr": attr, "qp": qp, "out": out, "room": _room(case, case["n"])}
    if kind in ("encode_batch", "decode_batch"):
        pos, attr, J = _batch_frames(case, seed)
        qp = _quant(case)
        N, C = sum(p.shape[0] for p in pos), qp.C
        scales = RUNG_SCALES[:case["rungs"]]
        out = torch.zeros(_room(case, N), dtype=torch.uint8, device=DEVICE)
        if kind == "encode_batch":
            return {"case": case, "pos": pos, "attr": attr, "J": J, "qp": qp, "scales": scales, "out": out}
        out, offs, hdr = gsnfs.encode_batch(pos, attr, J, scales, qp, headers=True, out=out)
        return {"case": case, "data": out[:int(offs[-1])].clone(), "offs": offs, "hdr": hdr, "N": N, "C": C,
                "pos": torch.zeros((N, 3), device=DEVICE), "attr": torch.zeros((N, C), device=DEVICE),
                "status": torch.zeros(1, dtype=torch.int32, device=DEVICE)}
    if kind == "layer":
        pos, attr = _one_frame(seed, case["n"], "dynamic", voxels=case["J"])
        codes, _, _ = gsnfs.voxelize(pos, case["J"])
        return {"case": case, "attr": attr.requires_grad_(), "qp": _gs_quant(),
                "plan": gsnfs.RahtPlan(codes.clone(), case["J"], GS_CHANNELS),
                "grad": _Rand(seed + 7).normal(case["n"], GS_CHANNELS)}
    pos, attr = _one_frame(seed, case["n"], "dynamic")
    return {"case": case, "pos": pos, "attr": attr}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "encode":
        stream, nv, rpos, rattr = gsnfs.encode_frame(state["pos"], state["attr"], case["J"], state["qp"],
                                                     recon=case["recon"], out=state["out"])
        res = [state["out"][:state["room"]], stream.numel(), nv]  # the kept buffer: zeros after the stream
        return res + [rpos, rattr] if case["recon"] else res
    if kind == "decode":
        return list(gsnfs.decode_frame(state["stream"]))
    if kind == "encode_batch":
        if case["rungs"] == 1:  # for a decoder that is handed the header records
            return list(gsnfs.encode_batch(state["pos"], state["attr"], state["J"], state["scales"], state["qp"],
                                           out=state["out"], headers=True))
        return list(gsnfs.encode_batch(state["pos"], state["attr"], state["J"], state["scales"], state["qp"],
                                       out=state["out"]))
    if kind == "decode_batch":  # into kept buffers: rows past the last frame's stay zero
        rows = gsnfs.decode_batch_async(state["data"], state["offs"], state["hdr"], state["C"], state["N"], state["pos"],
                                        state["attr"], state["status"])
        return [state["pos"], state["attr"], state["status"], rows]
    if kind == "layer":
        out = gsnfs.AttrCodecFn.apply(state["attr"], state["plan"], state["qp"])
        (grad,) = torch.autograd.grad(out, state["attr"], state["grad"])
        return [out.detach(), grad]
    view, fx, fy, cx, cy = _camera(case["width"], case["height"])
    return gsnfs.render(state["pos"], state["attr"], view, fx, fy, cx, cy, case["width"], case["height"],
                        background=(0.1, 0.2, 0.3))


# ---- the work that a pass cannot do without -------------------------------------------
def work(case):
    kind = case["kind"]
    if kind in ("encode", "decode", "encode_batch", "decode_batch"):
        C = CLOUD_CHANNELS if case["scene"] == "cloud" else GS_CHANNELS
        n = sum(_batch_shape(case)[0]) if "frames" in case else case["n"]
        both = 2 if case.get("recon") and kind == "encode" else 1
        return {"bytes": 4.0 * (3 + C) * n * both + _stream_bytes(case, n), "flops": (6.0 * C * both + 40.0) * n}
    if kind == "layer":  # attributes and the gradient in, the reconstruction and its gradient out
        return {"bytes": 16.0 * GS_CHANNELS * case["n"], "flops": 24.0 * GS_CHANNELS * case["n"]}
    px = case["width"] * case["height"]
    return {"bytes": 4.0 * (3 + GS_CHANNELS) * case["n"] + 12.0 * px, "flops": 500.0 * case["n"] + 20.0 * 100.0 * px}


# ---- results in 64 bits -------------------------------------------------------------
def _spread(v):
    """Bits of v to every third position."""
    out = torch.zeros_like(v)
    for b in range(21):
        out |= ((v >> b) & 1) << (3 * b)
    return out


def _gather_bits(m):
    out = torch.zeros_like(m)
    for b in range(21):
        out |= ((m >> (3 * b)) & 1) << b
    return out


def _voxels(pos, J):
    """Ascending distinct Morton codes, the voxel of each point, and the voxel centres."""
    p = pos.double()
    lo = p.amin(0)
    ext = float((p.amax(0) - lo).amax())
    ext = ext if ext > 0.0 else 1.0
    v = ((p - lo) * ((1 << J) / ext)).floor().long().clamp_max((1 << J) - 1)
    m = _spread(v[:, 0]) | (_spread(v[:, 1]) << 1) | (_spread(v[:, 2]) << 2)
    codes, inv = torch.unique(m, return_inverse=True)
    grid = torch.stack([_gather_bits(codes >> a) for a in range(3)], 1)
    return codes, inv, lo + (grid.double() + 0.5) * (ext / (1 << J))


def _raht_levels(codes, J):
    """Butterflies of every level: rows of the two children and the rotation (a, b)."""
    rows = torch.arange(codes.shape[0], device=codes.device)
    w = torch.ones(codes.shape[0], dtype=torch.float64, device=codes.device)
    c = codes
    levels = []
    for _ in range(3 * J):
        c = c >> 1
        pair = torch.zeros_like(c, dtype=torch.bool)
        pair[:-1] = c[1:] == c[:-1]  # a node and its right sibling
        left = pair.nonzero()[:, 0]
        if left.numel():
            w0, w1 = w[left], w[left + 1]
            levels.append((rows[left], rows[left + 1], (w0 / (w0 + w1)).sqrt()[:, None], (w1 / (w0 + w1)).sqrt()[:, None]))
            w = w.clone()
            w[left] = w0 + w1
            keep = torch.ones_like(pair)
            keep[left + 1] = False
            rows, w, c = rows[keep], w[keep], c[keep]
    return levels


def _raht(levels, V, inverse=False):
    for i0, i1, a, b in reversed(levels) if inverse else levels:
        x, y = V[i0], V[i1]
        V[i0], V[i1] = (a * x - b * y, b * x + a * y) if inverse else (a * x + b * y, a * y - b * x)
    return V


def _reconstruct(levels, A, qp):
    """Forward transform, quantise, dequantise, inverse transform."""
    step = torch.tensor(qp.steps[qp.groups.astype(int)], dtype=torch.float64, device=A.device)
    Y = _raht(levels, A)
    Y = torch.sign(Y) * (Y.abs() / step + qp.tau).floor() * step
    return _raht(levels, Y, inverse=True)


_YUV = [[0.299, 0.587, 0.114], [-0.14713, -0.28886, 0.436], [0.615, -0.51499, -0.10001]]


def _exact_frame(pos, attr, J, qp):
    """Decoded positions and attributes of one frame."""
    codes, inv, centres = _voxels(pos, J)
    a = attr.double()
    klt = M = None
    if qp.color:  # YUV on every SH function, then the KLT of each channel's 15 AC functions over the first points
        M = torch.tensor(_YUV, dtype=torch.float64, device=a.device)
        sh = torch.cat([a[:, 8:11, None], a[:, 11:56].reshape(-1, 3, 15)], 2)
        sh = torch.einsum("ij,njk->nik", M, sh)
        s = sh[:4096, :, 1:]
        d = s - s.mean(0, keepdim=True)
        _, vec = torch.linalg.eigh(torch.einsum("nij,nik->ijk", d, d) / d.shape[0])
        klt = vec.transpose(1, 2).flip(1).float().double()  # rows: eigenvectors, largest eigenvalue first
        ac = torch.einsum("irk,nik->nir", klt, sh[:, :, 1:])
        a = torch.cat([a[:, :8], sh[:, :, 0], ac.reshape(-1, 45)], 1)
    cnt = torch.zeros(codes.shape[0], dtype=torch.float64, device=a.device).index_add_(0, inv, torch.ones_like(inv, dtype=torch.float64))
    V = torch.zeros((codes.shape[0], a.shape[1]), dtype=torch.float64, device=a.device).index_add_(0, inv, a) / cnt[:, None]
    V = _reconstruct(_raht_levels(codes, J), V, qp)
    if qp.color:
        ac = torch.einsum("irk,nir->nik", klt, V[:, 11:56].reshape(-1, 3, 15))
        sh = torch.einsum("ij,njk->nik", torch.linalg.inv(M), torch.cat([V[:, 8:11, None], ac], 2))
        V = torch.cat([V[:, :8], sh[:, :, 0], sh[:, :, 1:].reshape(-1, 45)], 1)
    return centres, V


def _sh_basis(d):
    x, y, z = d[:, 0], d[:, 1], d[:, 2]
    pi = math.pi
    c1, c2, c3 = math.sqrt(3 / (4 * pi)), math.sqrt(15 / pi), math.sqrt(35 / (2 * pi))
    t, s = math.sqrt(105 / pi), math.sqrt(21 / (2 * pi))
    return torch.stack([
        torch.full_like(x, 0.5 / math.sqrt(pi)), -c1 * y, c1 * z, -c1 * x, 0.5 * c2 * x * y, -0.5 * c2 * y * z,
        0.25 * math.sqrt(5 / pi) * (2 * z * z - x * x - y * y), -0.5 * c2 * x * z, 0.25 * c2 * (x * x - y * y),
        -0.25 * c3 * y * (3 * x * x - y * y), 0.5 * t * x * y * z, -0.25 * s * y * (4 * z * z - x * x - y * y),
        0.25 * math.sqrt(7 / pi) * z * (2 * z * z - 3 * x * x - 3 * y * y), -0.25 * s * x * (4 * z * z - x * x - y * y),
        0.25 * t * z * (x * x - y * y), -0.25 * c3 * x * (x * x - 3 * y * y)], 1)


def _exact_render(pos, attr, case, background=(0.1, 0.2, 0.3), znear=0.01):
    W, H = case["width"], case["height"]
    view, fx, fy, cx, cy = _camera(W, H)
    view = torch.tensor(np.asarray(view), dtype=torch.float64, device=pos.device).reshape(3, 4)
    R, t = view[:, :3], view[:, 3]
    p, a = pos.double(), attr.double()
    pc = p @ R.T + t
    keep = pc[:, 2] > znear
    p, a, pc = p[keep], a[keep], pc[keep]
    x, y, z = pc.unbind(1)
    w, i, j, k = (a[:, 3:7] / a[:, 3:7].norm(dim=1, keepdim=True)).unbind(1)
    rot = torch.stack([1 - 2 * (j * j + k * k), 2 * (i * j - w * k), 2 * (i * k + w * j),
                       2 * (i * j + w * k), 1 - 2 * (i * i + k * k), 2 * (j * k - w * i),
                       2 * (i * k - w * j), 2 * (j * k + w * i), 1 - 2 * (i * i + j * j)], 1).reshape(-1, 3, 3)
    m = rot * a[:, None, 0:3].exp()
    zero = torch.zeros_like(z)
    jac = torch.stack([fx / z, zero, -fx * x / z ** 2, zero, fy / z, -fy * y / z ** 2], 1).reshape(-1, 2, 3)
    tm = jac @ R @ m
    cov = tm @ tm.transpose(1, 2)
    ca, cb, cc = cov[:, 0, 0] + 0.3, cov[:, 0, 1], cov[:, 1, 1] + 0.3
    det = ca * cc - cb * cb
    mid = 0.5 * (ca + cc)
    rad = (3 * (mid + (mid * mid - det).clamp_min(0.1).sqrt()).sqrt()).ceil()
    u, v = fx * x / z + cx, fy * y / z + cy
    TX, TY = (W + 15) // 16, (H + 15) // 16
    tx0, tx1 = ((u - rad) / 16).floor().clamp_min(0), ((u + rad) / 16).floor().clamp_max(TX - 1)
    ty0, ty1 = ((v - rad) / 16).floor().clamp_min(0), ((v + rad) / 16).floor().clamp_max(TY - 1)
    d = p + R.T @ t  # from the camera centre -R^T t
    basis = _sh_basis(d / d.norm(dim=1, keepdim=True))
    col = torch.einsum("nk,nck->nc", basis, torch.cat([a[:, 8:11, None], a[:, 11:56].reshape(-1, 3, 15)], 2)) + 0.5
    order = torch.argsort(z.float(), stable=True)  # depth, then index
    tx0, tx1, ty0, ty1 = (q[order] for q in (tx0, tx1, ty0, ty1))
    q00, q01, q11 = (q[order] for q in (cc / det, -cb / det, ca / det))
    u, v, col, opa = u[order], v[order], col[order].clamp_min(0), torch.sigmoid(a[order, 7])
    bg = torch.tensor(background, dtype=torch.float64, device=pos.device)
    img = torch.empty((TY * 16, TX * 16, 3), dtype=torch.float64, device=pos.device)
    g = torch.arange(16, device=pos.device, dtype=torch.float64) + 0.5
    for ty in range(TY):
        row = ((ty0 <= ty) & (ty <= ty1)).nonzero()[:, 0]
        for tx in range(TX):
            s = row[(tx0[row] <= tx) & (tx <= tx1[row])]
            T = torch.ones((16, 16), dtype=torch.float64, device=pos.device)
            c = torch.zeros((16, 16, 3), dtype=torch.float64, device=pos.device)
            live = torch.ones((16, 16), dtype=torch.bool, device=pos.device)
            for b in range(0, s.numel(), 4096):
                e = s[b:b + 4096]
                dx, dy = (u[e] - (16 * tx + g)[:, None])[None], (v[e] - (16 * ty + g)[:, None])[:, None]
                al = (opa[e] * torch.exp(-0.5 * (q00[e] * dx * dx + 2 * q01[e] * dx * dy + q11[e] * dy * dy))).clamp_max(0.99)
                al = torch.where(al < 1.0 / 255.0, torch.zeros_like(al), al)
                live = live[..., None] & (T[..., None] * torch.cumprod(1 - al, 2) >= 1e-4)  # the splat past the stop is out
                al = al * live
                after = T[..., None] * torch.cumprod(1 - al, 2)
                c += (al * torch.cat([T[..., None], after[..., :-1]], 2)) @ col[e]
                T, live = after[..., -1], live[..., -1]
            img[16 * ty:16 * ty + 16, 16 * tx:16 * tx + 16] = c + T[..., None] * bg
    return img[:H, :W].contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("encode", "decode"):
        if kind == "encode" and not case["recon"]:
            return None  # bytes and counts
        frame = _exact_frame(*_case_frame(case, seed), case["J"], _quant(case))
        return list(frame) if kind == "decode" else [None, None, None, *frame]
    if kind == "encode_batch":
        return None
    if kind == "decode_batch":
        qp = _quant(case)
        pos, attr, J = _batch_frames(case, seed)
        N = sum(p.shape[0] for p in pos)
        res = [torch.zeros((N, 3), dtype=torch.float64, device=DEVICE), torch.zeros((N, qp.C), dtype=torch.float64, device=DEVICE)]
        row = 0
        for f in range(len(J)):
            frame = _exact_frame(pos[f], attr[f], J[f], qp)
            for r, x in zip(res, frame):
                r[row:row + x.shape[0]] = x
            row += frame[0].shape[0]
        return res + [None, None]
    if kind == "layer":
        pos, attr = _one_frame(seed, case["n"], "dynamic", voxels=case["J"])
        out = _reconstruct(_raht_levels(_voxels(pos, case["J"])[0], case["J"]), attr.double(), _gs_quant())
        return [out, _Rand(seed + 7).normal(case["n"], GS_CHANNELS).double()]  # T^T T g = g: the transform is orthonormal
    pos, attr = _one_frame(seed, case["n"], "dynamic")
    return _exact_render(pos, attr, case)
