// Batch-wide decoding steps: many frames (streams) decoded by one sequence
// of launches (Sec. 2.3 / Algorithms 2-3 for geometry, Sec. 3.4 and the
// inverse of Algorithm 6 for attributes, applied to every frame at once).
// Frames are described by a device table (DecFrame); every kernel finds the
// frame of its work item with a binary search over per-frame prefix sums.
#include "kernels.cuh"
#include "rans_dec.cuh"

namespace gsnfs {

namespace {

constexpr uint32_t kProbBits = 15;
constexpr uint32_t kM = 1u << kProbBits;

template <typename T>
__device__ __forceinline__ uint32_t find_frame(const T *pref, uint32_t F, uint64_t x)
{
    uint32_t lo = 0, hi = F;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if ((uint64_t)pref[mid] <= x) lo = mid; else hi = mid;
    }
    return lo;
}

// raw and constant occupancy sections: bytes straight into the batch buffer
__global__ void occ_bytes_kernel(const DecFrame *fr, uint8_t *occ_all)
{
    if (after_previous()) return;
    const DecFrame &d = fr[blockIdx.y];
    if (d.mode == 1) return;
    uint8_t *dst = occ_all + d.occ_off;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < d.n_occ; i += (uint64_t)gridDim.x * blockDim.x)
        dst[i] = (d.mode == 2) ? (uint8_t)d.aux : d.occ_sec[16 + i];
}

// per frame: slot -> symbol table and freq << 16 | cum, then a corruption flag; and the byte offset of
// every chunk inside the section (a scan of the chunk size table)
__global__ void __launch_bounds__(1024) tables_kernel(const DecFrame *fr, uint32_t *tabs, uint64_t tab_words,
                                                      uint64_t *cstart, DevState *st)
{
    if (after_previous()) return;
    const DecFrame &d = fr[blockIdx.x];
    if (d.mode != 1) return;
    uint32_t *tab = tabs + (uint64_t)blockIdx.x * tab_words;
    __shared__ uint32_t cum[257];
    const bool ok = ransdec::build_tables(d.occ_sec + 24, tab, cum);
    if (threadIdx.x == 0) {
        tab[kM / 4 + 256] = !ok;
        if (!ok) set_error(&st->err, kErrCorrupt);
    }
    // chunk offsets: after the section header, the frequency table and the size table (8-byte aligned)
    __shared__ uint64_t sh64[33];
    const uint32_t nch = d.aux;
    const uint8_t *ctab = d.occ_sec + 24 + 512;
    uint64_t run = (16 + 8 + 512 + 4 * (uint64_t)nch + 7) & ~7ull;
    for (uint32_t b = 0; b < nch; b += blockDim.x) {
        const uint32_t c = b + threadIdx.x;
        uint64_t sz = 0;
        if (c < nch) {
            const uint8_t *q = ctab + 4 * (uint64_t)c;
            sz = (uint32_t)q[0] | ((uint32_t)q[1] << 8) | ((uint32_t)q[2] << 16) | ((uint32_t)q[3] << 24);
        }
        uint64_t tot;
        const uint64_t ex = block_exclusive_sum<uint64_t>(sz, sh64, &tot);
        if (c < nch) cstart[d.chunk_off + c] = run + ex;
        run += tot;
    }
}

// grid (chunk groups, frames): warp per chunk of frame blockIdx.y, the chunk read in place, the tables in shared memory
constexpr uint32_t kRansWarps = 8;

__global__ void __launch_bounds__(32 * kRansWarps) rans_batch_kernel(const DecFrame *fr, const uint32_t *tabs,
                                                                     uint64_t tab_words, const uint64_t *cstart,
                                                                     uint8_t *occ_all, DevState *st)
{
    if (after_previous()) return;
    using namespace ransdec;
    extern __shared__ __align__(16) unsigned char dsm[];
    const DecFrame &d = fr[blockIdx.y];
    if (d.mode != 1) return;
    const uint32_t *tab = tabs + (uint64_t)blockIdx.y * tab_words;
    if (tab[kTabWords] != 0) return;
    const uint32_t nch = d.aux, chunk = d.chunk;
    const uint32_t lane = threadIdx.x & 31, wl = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    if (blockIdx.x * nwarps >= nch) return;  // no chunk of this frame for this CTA
    load_tables(reinterpret_cast<uint32_t *>(dsm), tab);
    __syncthreads();
    const uint8_t *slot2sym = dsm;
    const uint32_t *fc = reinterpret_cast<const uint32_t *>(dsm + kM);
    const uint8_t *ctab = d.occ_sec + 24 + 512;
    uint8_t *out = occ_all + d.occ_off;
    for (uint32_t c = blockIdx.x * nwarps + wl; c < nch; c += gridDim.x * nwarps) {
        const uint64_t start = cstart[d.chunk_off + c];
        const uint8_t *cp = ctab + 4 * c;
        const uint32_t cbytes = (uint32_t)cp[0] | ((uint32_t)cp[1] << 8) | ((uint32_t)cp[2] << 16) | ((uint32_t)cp[3] << 24);
        if (cbytes < 128 || (cbytes & 3) || (start & 3) || cbytes > 128 + 2 * chunk + 2 || start + cbytes > d.occ_bytes) {
            if (lane == 0) set_error(&st->err, kErrCorrupt);
            continue;
        }
        const uint64_t s0 = (uint64_t)c * chunk;
        const uint32_t len = (uint32_t)((d.n_occ - s0) < chunk ? (d.n_occ - s0) : chunk);
        if (decode_chunk(slot2sym, fc, d.occ_sec + start, (cbytes - 128) / 2, len, out + s0, lane) && lane == 0)
            set_error(&st->err, kErrCorrupt);
    }
}

__device__ __forceinline__ uint32_t compact3b(uint64_t m)
{
    m &= 0x1249249249249249ull;
    m = (m | (m >> 2)) & 0x10C30C30C30C30C3ull;
    m = (m | (m >> 4)) & 0x100F00F00F00F00Full;
    m = (m | (m >> 8)) & 0x001F0000FF0000FFull;
    m = (m | (m >> 16)) & 0x001F00000000FFFFull;
    m = (m | (m >> 32)) & 0x00000000001FFFFFull;
    return (uint32_t)m;
}

// ---- octree (Algorithm 3) ------------------------------------------------------
// P(x) = number of set bits in the batch occupancy bytes before byte x.  Node w
// of level d of frame f (byte x = occ_off + boff[d] + w) has its children at
// indices P(x) - pbase[d] .. of level d + 1, pbase[d] = P at the level's first
// byte, which the host knows (a level's popcounts add up to the next level's
// size).  The bytes are summed in tiles, P at every tile's first byte is one
// scan.
constexpr uint32_t kOccTile = 1024;  // bytes per tile

__device__ __forceinline__ uint32_t word_at(const uint8_t *occ, uint64_t n, uint64_t x)  // bytes >= n read 0
{
    if (x >= n) return 0u;
    uint32_t v = *reinterpret_cast<const uint32_t *>(occ + x);  // x % 4 == 0; the buffer has 8 bytes of slack
    if (x + 4 > n) v &= (1u << (8u * (uint32_t)(n - x))) - 1u;
    return v;
}

// tsum: set bits per tile; *broken and the error are set when a byte is zero (a node without children)
__global__ void __launch_bounds__(256) occ_tile_popc_kernel(const uint8_t *occ, uint64_t n,
                                                            uint64_t ntiles, uint32_t *tsum, uint32_t *broken,
                                                            DevState *st)
{
    if (after_previous()) return;
    const uint32_t lane = threadIdx.x & 31;
    for (uint64_t t = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < ntiles;
         t += ((uint64_t)gridDim.x * blockDim.x) >> 5) {
        uint32_t c = 0, zero = 0;
#pragma unroll
        for (uint32_t k = 0; k < kOccTile / 128; ++k) {
            const uint64_t x = t * kOccTile + 4ull * (lane + 32 * k);
            uint32_t v = word_at(occ, n, x);
            c += __popc(v);
            if (x + 4 > n) v |= x < n ? 0xFFFFFFFFu << (8u * (uint32_t)(n - x)) : 0xFFFFFFFFu;  // bytes past the end
            zero |= __vcmpeq4(v, 0u);
        }
        if (__any_sync(0xFFFFFFFFu, zero != 0u) && lane == 0) {
            *broken = 1;
            set_error(&st->err, kErrCorrupt);
        }
        c = __reduce_add_sync(0xFFFFFFFFu, c);
        if (lane == 0) tsum[t] = c;
    }
}

__device__ __forceinline__ void leaf_out(const DecFrame &d, const float *ctab, uint32_t v, uint64_t m,
                                         float *pos)
{
    if (d.ctab_off != ~0ull) {
        const float *t = ctab + d.ctab_off;
        float c[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) c[a] = *(t + ((uint64_t)a << d.J) + compact3b(m >> a));
#pragma unroll
        for (int a = 0; a < 3; ++a) pos[3ull * v + a] = c[a];
    } else {
        const FrameGrid g = d.grid;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double off = __dmul_rn(__dadd_rn((double)compact3b(m >> a), 0.5), g.cell);
            pos[3ull * v + a] = (float)__dadd_rn(g.lo[a], off);
        }
    }
}

// Going down level by level, every level reads and writes a code per node and
// waits for a launch.  Instead a CTA takes kLeafTile nodes of the last level and
// walks down their ancestors only, from the root, the codes in shared memory:
// global memory sees the occupancy bytes and the voxels' outputs.  A node has at
// least one child, so that no level has more ancestors than the last has nodes.
// Where a CTA begins in each level is found first, a warp per CTA going up by
// rank: the parent of node w of level d + 1 is the byte that holds set bit
// pbase[d] + w.  A CTA's last node is the next one's first, for that one's last
// child is the voxel before the next CTA's first (its gap level).
// 16 frames of 1M voxels, beside the RLGR decode: 1.57 ms in 16 launches, a tile
// of 1,024 nodes of a level per CTA -> 0.18 + 0.56 ms.  Bound by latency: a
// level is a scan and a loop over at most eight children between two barriers.
constexpr uint32_t kLeafTile = 1016, kLeafThreads = 256;
constexpr uint32_t kLeafNodes = kLeafTile + 1;  // of a level in a CTA at most; with the 3 bytes before, a word a thread
constexpr uint32_t kLeafStage = 2048;           // voxels gathered at a time
static_assert(kLeafNodes + 3 <= 4 * kLeafThreads && kLeafNodes <= kLeafStage, "a word of bytes per thread");

struct OctArgs {
    const DecFrame *fr;
    uint32_t F, Jmax;
    uint32_t Jtab, tables;      // deepest frame with a centre table, warps for the tables
    const uint32_t *tile_pref;  // F + 1: first CTA of each frame
    uint32_t tiles;             // tile_pref[F]
    const uint8_t *occ;
    uint64_t n_occ;
    const uint64_t *tbase;      // P at each tile's first byte, and the total
    uint2 *path;                // per CTA and level: first node, its children that belong to the CTA before
    uint32_t *leaf0;            // per CTA: voxels of the frame before the first node's
    float *ctab;
    float *pos;                 // or null: no centres
    uint8_t *gap;
    uint64_t nv_total;
    uint32_t *broken;           // set: the bytes are not an octree's with these level sizes
    DevState *st;
};

// P(x), by a warp
__device__ __forceinline__ uint64_t bits_before(const OctArgs &a, uint64_t x, uint32_t lane)
{
    const uint64_t t = x / kOccTile;
    const uint32_t part = (uint32_t)(x % kOccTile);
    uint32_t c = 0;
#pragma unroll
    for (uint32_t k = 0; k < kOccTile / 128; ++k) {
        const uint32_t o = 4 * (lane + 32 * k);
        if (o >= part) continue;
        uint32_t v = word_at(a.occ, a.n_occ, t * kOccTile + o);
        if (o + 4 > part) v &= (1u << (8u * (part - o))) - 1u;
        c += __popc(v);
    }
    return a.tbase[t] + __reduce_add_sync(0xFFFFFFFFu, c);
}

// The byte of [a0, a1) that holds set bit r, by a warp: its index from a0 and, in y, the set bits before r in it.
// (Any r and any bytes: the byte returned lies in the range.)
__device__ __forceinline__ uint2 byte_of_bit(const OctArgs &a, uint64_t a0, uint64_t a1, uint64_t r, uint32_t lane)
{
    uint64_t t = a0 / kOccTile, n = (a1 - 1) / kOccTile - t + 1;  // the last of n tiles from t that starts at or before r
    while (n > 1) {
        const uint64_t step = (n + 31) / 32, probe = lane * step;
        const uint32_t le = __ballot_sync(0xFFFFFFFFu, probe < n && a.tbase[t + probe] <= r);
        const uint32_t last = le ? 31u - (uint32_t)__clz(le) : 0u;
        t += last * step;
        n = min(step, n - last * step);
    }
    const uint64_t tx = t * kOccTile, tb = a.tbase[t];
    uint32_t rest = r > tb ? (uint32_t)min(r - tb, (uint64_t)(8 * kOccTile)) : 0u;
    uint32_t c = 0;
#pragma unroll
    for (uint32_t k = 0; k < kOccTile / 128; ++k) c += __popc(word_at(a.occ, a.n_occ, tx + lane * (kOccTile / 32) + 4 * k));
    uint32_t inc = warp_inclusive_sum(c);
    uint32_t m = __ballot_sync(0xFFFFFFFFu, inc > rest);
    const uint32_t part = m ? (uint32_t)__ffs(m) - 1u : 31u;  // 32 bytes
    rest -= min(rest, __shfl_sync(0xFFFFFFFFu, inc - c, part));
    const uint64_t x = tx + part * (kOccTile / 32) + lane;
    c = x < a.n_occ ? __popc(a.occ[x]) : 0u;
    inc = warp_inclusive_sum(c);
    m = __ballot_sync(0xFFFFFFFFu, inc > rest);
    const uint32_t byte = m ? (uint32_t)__ffs(m) - 1u : 31u;
    rest -= min(rest, __shfl_sync(0xFFFFFFFFu, inc - c, byte));
    const uint64_t y = min(max(tx + part * (kOccTile / 32) + byte, a0), a1 - 1);
    return make_uint2((uint32_t)(y - a0), min(rest, 8u));
}

// A warp per CTA of octree_leaves_kernel: where it begins in each level.  Then a warp per frame and level: that the
// level's bytes hold as many set bits as the next level has nodes.  Then kTableEntries of a frame's centre table a
// warp: entry a * 2^J + v = (float)(lo_a + (v + 0.5) * cell), the same FP64 expression as per voxel (Sec. 2.1).
constexpr uint32_t kTableEntries = 512;

__host__ __device__ inline uint32_t table_warps(uint32_t Jmax)  // of a frame; no table is larger than the voxels
{
    return (uint32_t)(((3ull << Jmax) + kTableEntries - 1) / kTableEntries);
}

__global__ void __launch_bounds__(256) octree_paths_kernel(OctArgs a)
{
    if (after_previous()) return;
    const uint32_t lane = threadIdx.x & 31, w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w == 0 && lane == 0) a.gap[a.nv_total] = (uint8_t)kInfLevel;  // sentinel after the last voxel
    if (w < a.tiles) {
        const uint32_t f = find_frame(a.tile_pref, a.F, w), k = w - a.tile_pref[f];
        const DecFrame &fd = a.fr[f];
        uint32_t d = fd.J - 1, i = k ? k * kLeafTile - 1 : 0u;  // the last node of the CTA before
        uint2 *path = a.path + (uint64_t)w * kMaxJ;
        const uint64_t leaf0 = bits_before(a, fd.occ_off + fd.boff[d] + i, lane) - fd.pbase[d];
        if (lane == 0) {
            path[d] = make_uint2(i, 0u);
            a.leaf0[w] = (uint32_t)min(leaf0, (uint64_t)fd.nv);
        }
        while (d > 0) {
            --d;
            const uint64_t a0 = fd.occ_off + fd.boff[d];
            const uint2 p = byte_of_bit(a, a0, a0 + fd.lsz[d], fd.pbase[d] + i, lane);
            if (lane == 0) path[d] = p;
            i = p.x;
        }
    } else if (w < a.tiles + a.F * a.Jmax) {
        const uint32_t f = (w - a.tiles) / a.Jmax, d = (w - a.tiles) - f * a.Jmax;
        const DecFrame &fd = a.fr[f];
        if (fd.nv == 0 || d >= fd.J) return;
        const uint64_t a0 = fd.occ_off + fd.boff[d];
        const uint64_t bits = bits_before(a, a0 + fd.lsz[d], lane) - bits_before(a, a0, lane);
        if (lane == 0 && bits != fd.lsz[d + 1]) {
            *a.broken = 1;
            set_error(&a.st->err, kErrCorrupt);
        }
    } else if (w < a.tiles + a.F * a.Jmax + a.tables) {
        const uint32_t x = w - a.tiles - a.F * a.Jmax, per = table_warps(a.Jtab), f = x / per;
        const DecFrame &fd = a.fr[f];
        if (fd.ctab_off == ~0ull) return;
        const uint64_t side = 1ull << fd.J, e0 = (uint64_t)(x - f * per) * kTableEntries;
        float *tab = a.ctab + fd.ctab_off;
        for (uint64_t e = e0 + lane; e < min(e0 + kTableEntries, 3 * side); e += 32) {
            const uint32_t axis = (uint32_t)(e >> fd.J);
            const double off = __dmul_rn(__dadd_rn((double)(e & (side - 1)), 0.5), fd.grid.cell);
            tab[e] = (float)__dadd_rn(fd.grid.lo[axis], off);
        }
    }
}

// the set bits of v as children of a node: calls put(rank, code) for each, rank counting from `rank`
template <typename Put>
__device__ __forceinline__ void children(uint64_t code, uint32_t v, uint32_t rank, Put put)
{
    for (; v; v &= v - 1u) put(rank++, (code << 3) + (uint32_t)(__ffs(v) - 1));
}

__global__ void __launch_bounds__(kLeafThreads) octree_leaves_kernel(OctArgs a)
{
    if (after_previous()) return;
    __shared__ uint64_t s_code[2][kLeafStage];  // a level's codes, the last level's in [0]; then the voxels' in [1]
    __shared__ uint2 s_path[kMaxJ];             // first node, its children of the CTA before
    __shared__ uint32_t s_cnt[kMaxJ];           // nodes
    __shared__ uint32_t s_word[kMaxJ][32];      // the bytes of a level of few nodes
    __shared__ uint32_t s_scan[2][kLeafThreads / 32];
    __shared__ uint64_t s_prev;
    const uint32_t g = blockIdx.x, t = threadIdx.x, lane = t & 31;
    if (*a.broken) {  // nothing to follow: every voxel on its own, for what reads the gap levels next
        const uint64_t per = (a.nv_total + a.tiles - 1) / a.tiles, lo = g * per, hi = min(lo + per, a.nv_total);
        for (uint64_t i = lo + t; i < hi; i += kLeafThreads) a.gap[i] = (uint8_t)kInfLevel;
        return;
    }
    const uint32_t f = find_frame(a.tile_pref, a.F, g), k = g - a.tile_pref[f];
    const bool last = g + 1 == a.tile_pref[f + 1];
    const DecFrame &fd = a.fr[f];
    const uint32_t J = fd.J;
    if (t < J) {
        const uint2 p = a.path[(uint64_t)g * kMaxJ + t];
        const uint32_t e = last ? fd.lsz[t] - 1u : a.path[(uint64_t)(g + 1) * kMaxJ + t].x;
        s_path[t] = p;
        s_cnt[t] = e >= p.x ? min(e - p.x + 1u, kLeafNodes) : 0u;
    }
    __syncthreads();
    // word t of the bytes of this CTA's nodes of level d (aligned: `lead` bytes before the first node), others zero
    auto lead_of = [&](uint32_t d) { return (uint32_t)((fd.occ_off + fd.boff[d] + s_path[d].x) & 3u); };
    auto word_of = [&](uint32_t d, uint32_t at) {
        const uint64_t x = fd.occ_off + fd.boff[d] + s_path[d].x;
        const uint32_t lead = (uint32_t)(x & 3u), cnt = s_cnt[d], o = 4 * at;
        if (o >= lead + cnt) return 0u;
        uint32_t v = *reinterpret_cast<const uint32_t *>(a.occ + (x - lead) + o);  // 8 bytes of slack after the last
        if (o < lead) v &= 0xFFFFFFFFu << (8u * (lead - o));
        if (o + 4 > lead + cnt) v &= (1u << (8u * (lead + cnt - o))) - 1u;
        return v;
    };
    auto few = [&](uint32_t d) { return s_cnt[d] + 3u <= 128u; };  // a warp's words
    for (uint32_t d = t >> 5; d < J; d += kLeafThreads / 32)
        if (few(d)) s_word[d][lane] = word_of(d, lane);
    if (t == 0) s_code[(J - 1) & 1u][0] = 0ull;  // the implicit root of Algorithm 2
    __syncthreads();
    uint32_t d = 0;
    while (d + 1 < J && few(d)) ++d;
    if (t < 32)  // levels of few nodes: one warp, a node per lane
        for (uint32_t e = 0; e < d; ++e) {
            const uint8_t *bytes = reinterpret_cast<const uint8_t *>(s_word[e]) + lead_of(e);
            const uint64_t *from = s_code[(J - 1 - e) & 1u];
            uint64_t *to = s_code[(J - e) & 1u];
            const uint32_t cnt = s_cnt[e], cnt1 = s_cnt[e + 1];
            uint32_t rank = 0u - s_path[e].y;  // of the next child; wraps for the children of the CTA before
            for (uint32_t n = lane; n < cnt + lane; n += 32) {
                const uint32_t byte = n < cnt ? bytes[n] : 0u, c = __popc(byte), inc = warp_inclusive_sum(c);
                children(byte ? from[n] : 0ull, byte, rank + inc - c, [&](uint32_t r, uint64_t m) {
                    if (r < cnt1) to[r] = m;
                });
                rank += __shfl_sync(0xFFFFFFFFu, inc, 31);
            }
            __syncwarp();
        }
    uint32_t v = word_of(d, t);
    __syncthreads();
    // set bits of the CTA's nodes before the thread's word (one barrier), and of all of them
    auto scan = [&](uint32_t d, uint32_t c, uint32_t *tot) {
        uint32_t *sh = s_scan[d & 1u];
        const uint32_t inc = warp_inclusive_sum(c);
        if (lane == 31) sh[t >> 5] = inc;
        __syncthreads();
        uint32_t before = inc - c, all = 0;
#pragma unroll
        for (uint32_t w = 0; w < kLeafThreads / 32; ++w) {
            const uint32_t x = sh[w];
            before += w < (t >> 5) ? x : 0u;
            all += x;
        }
        *tot = all;
        return before;
    };
    uint32_t tot;
    for (; d + 1 < J; ++d) {  // a word of bytes (four nodes) per thread
        const uint32_t next = word_of(d + 1, t);  // lands while this level is taken
        const uint32_t lead = lead_of(d), skip = s_path[d].y, cnt = s_cnt[d], cnt1 = s_cnt[d + 1];
        const uint64_t *from = s_code[(J - 1 - d) & 1u];
        uint64_t *to = s_code[(J - d) & 1u];
        uint32_t rank = scan(d, __popc(v), &tot) - skip;  // wraps for the children of the CTA before
#pragma unroll
        for (uint32_t b = 0; b < 4; ++b) {
            const uint32_t n = 4 * t + b - lead, byte = (v >> (8 * b)) & 0xFFu;  // n wraps before the first node
            if (n >= cnt) continue;
            children(from[n], byte, rank, [&](uint32_t r, uint64_t m) {
                if (r < cnt1) to[r] = m;
            });
            rank += __popc(byte);
        }
        __syncthreads();
        v = next;
    }
    // last level: the voxels, kLeafStage at a time
    const uint32_t lead = lead_of(d), cnt = s_cnt[d];
    const uint32_t before0 = scan(d, __popc(v), &tot);
    const uint64_t vb = (uint64_t)fd.vstart + a.leaf0[g];
    const uint64_t vend = (uint64_t)fd.vstart + fd.nv;
    // the first node's voxels are the CTA's before (but the frame's first CTA's)
    const uint32_t own = k == 0 ? 0u : (uint32_t)__popc(a.occ[fd.occ_off + fd.boff[d] + s_path[d].x]);
    uint64_t *out = s_code[1];
    for (uint32_t base = 0; base < tot; base += kLeafStage) {
        uint32_t before = before0;
#pragma unroll
        for (uint32_t b = 0; b < 4; ++b) {
            const uint32_t n = 4 * t + b - lead, byte = (v >> (8 * b)) & 0xFFu;
            if (n >= cnt) continue;
            children(s_code[0][n], byte, before - base, [&](uint32_t r, uint64_t c) {
                if (r < kLeafStage) out[r] = c;
            });
            before += __popc(byte);
        }
        __syncthreads();
        const uint32_t hi = min(tot - base, kLeafStage);
        for (uint32_t i = t; i < hi; i += kLeafThreads) {
            const uint32_t r = base + i;
            if (r < own || vb + r >= vend) continue;
            const uint64_t m = out[i];
            const uint32_t row = (uint32_t)(vb + r);
            const uint64_t prev = i ? out[i - 1] : s_prev;
            a.gap[row] = r ? (uint8_t)gap_level(prev, m, 64) : (uint8_t)kInfLevel;
            if (a.pos) leaf_out(fd, a.ctab, row, m, a.pos);
        }
        const uint64_t end = out[hi - 1];
        __syncthreads();
        if (t == 0) s_prev = end;
    }
}

__global__ void block_tables_kernel(const DecFrame *fr, uint32_t F, const uint64_t *blk_pref, uint64_t nblk,
                                    uint32_t *bw_all)
{
    if (after_previous()) return;
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nblk; k += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t f = find_frame(blk_pref, F, k);
        bw_all[k] = fr[f].bw[k - blk_pref[f]];
    }
}

uint32_t grid_for(uint64_t n, int num_sms)
{
    uint64_t b = (n + 255) / 256;
    const uint64_t cap = (uint64_t)num_sms * 8;
    if (b < 1) b = 1;
    return (uint32_t)(b < cap ? b : cap);
}

}  // namespace

void launch_batch_occ_bytes(const DecFrame *fr, uint32_t F, uint8_t *occ_all, uint64_t max_occ, int num_sms,
                            cudaStream_t s)
{
    if (max_occ == 0) return;
    uint32_t X = grid_for(max_occ, num_sms) / F + 1;
    launch_after(occ_bytes_kernel, dim3(X, F), 256, 0, s, fr, occ_all);
    count_launch();
}

void launch_batch_rans_decode(const DecFrame *fr, uint32_t F, uint32_t max_chunks_per_frame, uint32_t chunk_max,
                              uint8_t *occ_all, uint32_t *tabs, uint64_t *cstart, DevState *st, cudaStream_t s)
{
    (void)chunk_max;
    if (max_chunks_per_frame == 0) return;
    const uint64_t tab_words = kM / 4 + 256 + 4;
    launch_after(tables_kernel, F, 1024, 0, s, fr, tabs, tab_words, cstart, st);
    count_launch();
    const size_t smem = (size_t)ransdec::kTabWords * 4;
    allow_shared<rans_batch_kernel>();
    const uint32_t X = (max_chunks_per_frame + kRansWarps - 1) / kRansWarps;
    launch_after(rans_batch_kernel, dim3(X, F), 32 * kRansWarps, smem, s, fr, tabs, tab_words, cstart, occ_all, st);
    count_launch();
}

uint64_t occ_tiles(uint64_t n_occ) { return (n_occ + kOccTile - 1) / kOccTile; }

void launch_occ_tile_bases(const uint8_t *occ, uint64_t n_occ, uint32_t *tsum, uint64_t *tbase, uint64_t *partials,
                           uint32_t *broken, DevState *st, int num_sms, cudaStream_t s)
{
    const uint64_t nt = occ_tiles(n_occ);
    if (nt) {
        const uint64_t want = (nt + 7) / 8, cap = (uint64_t)num_sms * 8;
        launch_after(occ_tile_popc_kernel, (uint32_t)(want < cap ? want : cap), 256, 0, s, occ, n_occ, nt, tsum, broken, st);
        count_launch();
    }
    launch_scan_u32_to_u64(tsum, nt, tbase, partials, num_sms, s);
}

uint64_t octree_path_words(uint64_t tiles) { return 2 * tiles * kMaxJ; }

uint32_t octree_tiles(uint32_t nodes) { return (nodes + kLeafTile - 1) / kLeafTile; }

void launch_octree_leaves(const DecFrame *fr, uint32_t F, uint32_t Jmax, uint32_t Jtab, const uint32_t *tile_pref,
                          uint32_t tiles, const uint8_t *occ, uint64_t n_occ, const uint64_t *tbase, uint32_t *path,
                          uint32_t *leaf0, float *ctab, float *pos, uint8_t *gap, uint64_t nv_total, uint32_t *broken,
                          DevState *st, cudaStream_t s)
{
    OctArgs a{fr, F, Jmax, Jtab, Jtab ? F * table_warps(Jtab) : 0u, tile_pref, tiles, occ, n_occ, tbase,
              reinterpret_cast<uint2 *>(path), leaf0, ctab, pos, gap, nv_total, broken, st};
    launch_after(octree_paths_kernel, (tiles + F * Jmax + a.tables + 7) / 8, 256, 0, s, a);
    count_launch();
    if (tiles == 0) return;
    launch_after(octree_leaves_kernel, tiles, kLeafThreads, 0, s, a);
    count_launch();
}

void launch_batch_block_tables(const DecFrame *fr, uint32_t F, const uint64_t *blk_pref, uint64_t nblk,
                               uint32_t *bw_all, int num_sms, cudaStream_t s)
{
    if (nblk == 0) return;
    launch_after(block_tables_kernel, grid_for(nblk, num_sms), 256, 0, s, fr, F, blk_pref, nblk, bw_all);
    count_launch();
}

}  // namespace gsnfs
