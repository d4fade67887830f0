// Decoding side of the occupancy rANS (Sec. 2.3 entropy stage; format of the
// occupancy section: 32 interleaved 32-bit states per chunk, L = 2^16,
// 16-bit renormalisation words, M = 2^15), shared by the one-frame and the
// batched decoders.  One warp decodes one chunk: lane j owns state j and
// symbols j, j + 32, ...; the words each step needs are handed out in lane
// order by a ballot.
#pragma once
#include "common.cuh"

namespace gsnfs {
namespace ransdec {

constexpr uint32_t kProbBits = 15;
constexpr uint32_t kM = 1u << kProbBits;
constexpr uint32_t kL = 1u << 16;
constexpr uint32_t kTabWords = kM / 4 + 256;  // slot -> symbol bytes, then freq << 16 | cum per symbol
constexpr uint32_t kMaxWarps = 8;

// whole CTA: copies the decoding tables (16-byte aligned, kTabWords words) into shared memory
__device__ __forceinline__ void load_tables(uint32_t *dst, const uint32_t *tab)
{
    const uint4 *s = reinterpret_cast<const uint4 *>(tab);
    uint4 *d = reinterpret_cast<uint4 *>(dst);
    for (uint32_t k = threadIdx.x; k < kTabWords / 4; k += blockDim.x) d[k] = s[k];
}

// Whole CTA (a power of two of threads, at most kM / 4): the decoding tables of
// a section's frequency table `ftab` to tab (shared or global memory, kTabWords
// words); false (for every thread) when the frequencies do not add up to M.
// cum: 257 words of shared memory.  A thread fills a run of consecutive slots,
// walking the symbols from the first slot's.  Contains __syncthreads.
__device__ __forceinline__ bool build_tables(const uint8_t *ftab, uint32_t *tab, uint32_t *cum)
{
    if (threadIdx.x < 32) {
        uint32_t run = 0;
        for (int b = 0; b < 256; b += 32) {
            const int s = b + threadIdx.x;
            const uint32_t v = (uint32_t)(ftab[2 * s] | (ftab[2 * s + 1] << 8));
            const uint32_t inc = warp_inclusive_sum(v);
            cum[s] = run + inc - v;
            tab[kM / 4 + s] = (v << 16) | ((run + inc - v) & 0xFFFFu);
            run += __shfl_sync(0xFFFFFFFFu, inc, 31);
        }
        if (threadIdx.x == 0) cum[256] = run;
    }
    __syncthreads();
    if (cum[256] != kM) return false;
    const uint32_t per = kM / blockDim.x, t0 = threadIdx.x * per;
    uint32_t lo = 0, hi = 256;  // symbol of a slot: the last s with cum[s] <= slot
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (cum[mid] <= t0) lo = mid; else hi = mid;
    }
    uint32_t end = cum[lo + 1];
    for (uint32_t t = t0; t < t0 + per; t += 4) {
        uint32_t w = 0;
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            while (t + k >= end) end = cum[++lo + 1];  // ends: cum[256] = M is above every slot
            w |= lo << (8 * k);
        }
        tab[t / 4] = w;
    }
    __syncthreads();
    return true;
}

// One warp: decodes len symbols of a chunk (states then W words at src) to out;
// returns true if the chunk asked for more words than it holds.  W is even and
// src 4-byte aligned.  Lane l holds 32-bit words l, 32 + l, ... of the chunk
// from the reader's 32-word line on, the two lines after it on their way, and a
// step's 16-bit words are handed out by shuffles: loading them where they are
// needed put a first touch of an L2 sector into almost every step's chain (one
// frame of 10k Gaussians: 46 us for 128 steps; 1M-voxel batches the same).
__device__ __forceinline__ bool decode_chunk(const uint8_t *slot2sym, const uint32_t *fc, const uint8_t *src,
                                             uint32_t W, uint32_t len, uint8_t *out, uint32_t lane)
{
    const uint32_t *words = reinterpret_cast<const uint32_t *>(src + 128);
    const uint32_t n32 = W / 2;
    auto word = [&](uint32_t i) { return i < n32 ? words[i] : 0u; };
    uint32_t x = reinterpret_cast<const uint32_t *>(src)[lane];
    const uint32_t ltm = lanemask_lt();
    uint32_t line = 0, c0 = word(lane), c1 = word(32 + lane), c2 = word(64 + lane), c3 = word(96 + lane);
    uint32_t wp = 0;
    bool bad = false;
    for (uint32_t g = 0; g * 32 < len; ++g) {
        const uint32_t j = g * 32 + lane;
        bool need = false;
        if (j < len) {
            const uint32_t slot = x & (kM - 1);
            const uint32_t sy = slot2sym[slot];
            const uint32_t f = fc[sy];
            out[j] = (uint8_t)sy;
            x = (f >> 16) * (x >> kProbBits) + slot - (f & 0xFFFFu);
            need = x < kL;
        }
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, need);
        const uint32_t k = wp + __popc(m & ltm), i = (k >> 1) - line;  // i < 64
        const uint32_t v0 = __shfl_sync(0xFFFFFFFFu, c0, i), v1 = __shfl_sync(0xFFFFFFFFu, c1, i);
        if (need) {
            if (k < W) x = (x << 16) | (((i < 32 ? v0 : v1) >> (16 * (k & 1))) & 0xFFFFu);
            else bad = true;
        }
        wp += __popc(m);
        if (wp - 2 * line >= 64) {
            line += 32;
            c0 = c1;
            c1 = c2;
            c2 = c3;
            c3 = word(line + 96 + lane);
        }
    }
    return __any_sync(0xFFFFFFFFu, bad);
}

// one warp: byte offset of chunk c inside the chunk area (sum of the sizes before it)
__device__ __forceinline__ uint64_t chunk_offset(const uint8_t *ctab, uint32_t c, uint32_t lane)
{
    uint64_t off = 0;
    for (uint32_t k = lane; k < c; k += 32) {
        const uint8_t *p = ctab + 4 * k;
        off += (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) | ((uint32_t)p[3] << 24);
    }
    for (int o = 16; o > 0; o >>= 1) off += __shfl_xor_sync(0xFFFFFFFFu, off, o);
    return off;
}

}  // namespace ransdec
}  // namespace gsnfs
