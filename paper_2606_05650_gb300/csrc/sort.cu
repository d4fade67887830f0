// LSD radix sort of (64-bit Morton key, 32-bit point index) pairs
// (Algorithm 1: "RadixSort" of the Morton codes), and of pairs with 32-bit
// keys (the rasteriser's depths and tiles).  Only the 3J significant
// key bits are sorted, up to 8 bits per pass; the frames of a batch, which arrive
// grouped, are sorted as separate segments so that their id bits need no pass.
//
// Each pass is reduce-then-scan: every CTA owns one contiguous chunk of the
// array, counts its digits (upsweep), one CTA scans the digit-major count
// matrix, and every CTA re-reads its chunk tile by tile, ranks keys stably
// with warp votes, stages the tile digit-sorted in shared memory and
// writes it out in runs (downsweep).  No CTA waits on another CTA.
#include "kernels.cuh"

namespace gsnfs {

namespace {

constexpr int kRadix = 256;

// Threads, pairs per thread and CTAs resident per SM.  A downsweep writes a
// tile's pairs of a digit as one run, and what it costs is writes that fill
// their cache lines only in part: the longer the runs and the fewer CTAs write
// at a time, the less.  16 segments of 1M pairs (42-bit keys, six passes): 256
// threads x 8 pairs x 4 CTAs 0.98 ms, 256 x 8 x 2 0.81, 512 x 8 x 2 0.66, 512 x
// 12 x 2 0.75; one CTA per SM of any size 1.07 and more (nothing to do at its
// barriers).  Arrays that would not give every resident CTA two large tiles
// take the small ones.
template <int T, int K, int C>
struct SortCfg {
    static constexpr int threads = T, warps = T / 32, kpt = K, ctas = C, tile = T * K;
};
typedef SortCfg<256, 8, 4> SortSmall;
typedef SortCfg<512, 8, 2> SortLarge;
static_assert(SortLarge::tile >= SortSmall::tile && SortLarge::ctas <= SortSmall::ctas, "sort_ctas_bound");
constexpr uint64_t kLargeTiles = 2;  // per resident CTA

bool sort_large(uint64_t n, int num_sms)
{
    return n >= kLargeTiles * SortLarge::tile * SortLarge::ctas * (uint64_t)num_sms;
}

// Bits per pass: as few passes as 8-bit digits take, the bits spread evenly
// over them (fewer digits make longer runs: 11 bits as 6 + 5 instead of 8 + 3,
// 22M pairs, 0.49 -> 0.39 ms).
uint32_t digit_width(uint32_t nbits)
{
    const uint32_t passes = (nbits + 7) / 8;
    return (nbits + passes - 1) / passes;
}

struct SortGeom {
    uint32_t P;       // CTAs
    uint64_t chunk;   // elements per CTA
};

template <typename Cfg>
uint32_t sort_ctas(uint64_t n, int num_sms)
{
    const uint64_t tiles = (n + Cfg::tile - 1) / Cfg::tile, pmax = (uint64_t)num_sms * Cfg::ctas;
    return (uint32_t)(tiles < 1 ? 1 : (tiles < pmax ? tiles : pmax));
}

// CTAs of a sort of up to n pairs at most (a large array takes fewer than the largest small one)
uint32_t sort_ctas_bound(uint64_t n, int num_sms) { return sort_ctas<SortSmall>(n, num_sms); }

SortGeom sort_geom(uint64_t n, int num_sms)
{
    SortGeom g;
    g.P = sort_large(n, num_sms) ? sort_ctas<SortLarge>(n, num_sms) : sort_ctas<SortSmall>(n, num_sms);
    g.chunk = (n + g.P - 1) / g.P;
    return g;
}

// CTA p sorts elements [b, e): p * chunk onwards, or cta_lo[p] .. cta_lo[p + 1]
// when the array is cut into independently sorted segments
__device__ __forceinline__ void cta_range(const uint64_t *cta_lo, uint64_t chunk, uint64_t n, uint64_t &b,
                                          uint64_t &e)
{
    if (cta_lo) {
        b = cta_lo[blockIdx.x];
        e = cta_lo[blockIdx.x + 1];
    } else {
        b = (uint64_t)blockIdx.x * chunk;
        e = b + chunk;
        if (e > n) e = n;
    }
}

// Lanes of the warp (of those with ok) that hold the same digit: a vote per
// bit, whose time does not depend on the digits; __match_any_sync takes longer
// the more of them differ (10k keys in one CTA: 54 -> 41 us).
__device__ __forceinline__ uint32_t same_digit(uint32_t d, bool ok, uint32_t mask)
{
    uint32_t peers = __ballot_sync(0xFFFFFFFFu, ok);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        if (!(mask >> b)) break;
        const bool bit = (d >> b) & 1u;
        const uint32_t with = __ballot_sync(0xFFFFFFFFu, bit);
        peers &= bit ? with : ~with;
    }
    return peers;
}

template <typename Key, int kThreads>
__global__ void __launch_bounds__(kThreads) upsweep_kernel(const Key *keys, uint64_t n,
                                                           uint32_t shift, uint32_t mask, uint64_t chunk, uint32_t *hist,
                                                           const uint64_t *cta_lo)
{
    if (after_previous()) return;
    __shared__ uint32_t h[kRadix];
    if (threadIdx.x < kRadix) h[threadIdx.x] = 0;
    __syncthreads();
    uint64_t b, e;
    cta_range(cta_lo, chunk, n, b, e);
    uint64_t i = b + threadIdx.x;
    for (; i + 7 * kThreads < e; i += 8 * kThreads) {
        Key k[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) k[r] = keys[i + r * kThreads];
#pragma unroll
        for (int r = 0; r < 8; ++r) atomicAdd(&h[(uint32_t)(k[r] >> shift) & mask], 1u);
    }
    for (; i < e; i += kThreads) atomicAdd(&h[(uint32_t)(keys[i] >> shift) & mask], 1u);
    __syncthreads();
    if (threadIdx.x < kRadix) hist[(uint64_t)threadIdx.x * gridDim.x + blockIdx.x] = h[threadIdx.x];
}

// hist is digit-major [256][P]: warp d scans row d in place (exclusive) and
// stores the digit total at hist[256 * P + d]
__global__ void __launch_bounds__(256) scan_cols_kernel(uint32_t *hist, uint32_t P)
{
    if (after_previous()) return;
    const uint32_t d = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    uint32_t *row = hist + (uint64_t)d * P;
    uint32_t run = 0;
    for (uint32_t b = 0; b < P; b += 32) {
        const uint32_t c = b + lane;
        const uint32_t v = (c < P) ? row[c] : 0u;
        const uint32_t inc = warp_inclusive_sum(v);
        if (c < P) row[c] = run + inc - v;
        run += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
    if (lane == 0) hist[(uint64_t)kRadix * P + d] = run;
}

// A tile's pairs are loaded while the tile before is written out, into the
// registers that its pairs have left; every warp zeroes its own counters, so a
// tile takes four barriers.
template <typename Key, typename Cfg>
struct DownSmem {
    Key keys[Cfg::tile];
    uint32_t vals[Cfg::tile];
    uint16_t wcnt[Cfg::warps][kRadix];  // counts, then first slots, per warp and digit
    uint32_t out[kRadix];               // output position of slot 0, for the slots of each digit
    uint32_t scan[33];
};

template <typename Key, typename Cfg>
__global__ void __launch_bounds__(Cfg::threads, Cfg::ctas) downsweep_kernel(const Key *keys,
                                                             const uint32_t *vals, uint64_t n,
                                                             uint32_t shift, uint32_t mask, uint64_t chunk,
                                                             const uint32_t *hist,
                                                             Key *keys_out,
                                                             uint32_t *vals_out,
                                                             const uint64_t *cta_lo,
                                                             const uint32_t *cta_seg)
{
    if (after_previous()) return;
    constexpr int kWarps = Cfg::warps, kPairs = Cfg::kpt, kTile = Cfg::tile;
    extern __shared__ __align__(16) unsigned char sort_raw[];
    DownSmem<Key, Cfg> &S = *reinterpret_cast<DownSmem<Key, Cfg> *>(sort_raw);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t P = gridDim.x;
    const bool own = tid < kRadix;  // digit tid is this thread's
    uint32_t out = 0;               // where this CTA's pairs of it go
    if (!cta_seg) {  // digit d starts after all smaller digits, then after the same digit of earlier CTAs
        uint32_t tot;
        out = block_exclusive_sum<uint32_t>(own ? hist[(uint64_t)kRadix * P + tid] : 0u, S.scan, &tot);
        if (own) out += hist[(uint64_t)tid * P + blockIdx.x];
    } else {  // the same within this CTA's segment (CTAs p0 .. p1 - 1), which starts at element cta_lo[p0]
        const uint32_t p0 = cta_seg[2 * blockIdx.x], p1 = cta_seg[2 * blockIdx.x + 1];
        const uint32_t c0 = own ? hist[(uint64_t)tid * P + p0] : 0u;
        const uint32_t c1 = !own ? 0u : p1 < P ? hist[(uint64_t)tid * P + p1] : hist[(uint64_t)kRadix * P + tid];
        uint32_t tot;
        out = (uint32_t)cta_lo[p0] + block_exclusive_sum<uint32_t>(c1 - c0, S.scan, &tot);
        if (own) out += hist[(uint64_t)tid * P + blockIdx.x] - c0;
    }
    uint64_t cb, ce;
    cta_range(cta_lo, chunk, n, cb, ce);
    const uint32_t ltmask = lanemask_lt();
    const uint32_t at0 = (uint32_t)w * (32 * kPairs) + lane;  // this thread's pairs: at0 + 32 r
    Key k[kPairs];
    uint32_t v[kPairs], rk[(kPairs + 1) / 2];  // ranks: two 16-bit values each
    auto load = [&](uint64_t t0) {
#pragma unroll
        for (int r = 0; r < kPairs; ++r) {
            const uint64_t p = t0 + at0 + 32 * r;
            k[r] = p < ce ? keys[p] : Key(0);
            v[r] = p < ce ? vals[p] : 0u;
        }
    };
    auto zero_counters = [&]() {
#pragma unroll
        for (int i = 0; i < kRadix / 64; ++i) reinterpret_cast<uint32_t *>(S.wcnt[w])[lane + 32 * i] = 0u;
        __syncwarp();
    };
    load(cb);
    zero_counters();
    for (uint64_t t0 = cb; t0 < ce; t0 += kTile) {
        const uint32_t cnt = (uint32_t)((ce - t0) < (uint64_t)kTile ? (ce - t0) : (uint64_t)kTile);
#pragma unroll
        for (int r = 0; r < kPairs; ++r) {
            const bool ok = at0 + 32 * r < cnt;
            const uint32_t d = (uint32_t)(k[r] >> shift) & mask;
            const uint32_t peers = same_digit(d, ok, mask);
            const uint32_t before = __popc(peers & ltmask);
            const uint32_t base = S.wcnt[w][d];
            rk[r / 2] = (r & 1) ? (rk[r / 2] | ((base + before) << 16)) : (base + before);
            __syncwarp();
            if (ok && before == 0) S.wcnt[w][d] = (uint16_t)(base + __popc(peers));
            __syncwarp();
        }
        __syncthreads();
        // per digit: the tile's exclusive prefix over digits, then over the warps
        uint32_t run = 0;
        if (own) {
#pragma unroll
            for (int ww = 0; ww < kWarps; ++ww) run += S.wcnt[ww][tid];
        }
        const uint32_t inc = warp_inclusive_sum(run);
        if (lane == 31) S.scan[w] = inc;
        __syncthreads();
        if (own) {
            uint32_t at = inc - run;
#pragma unroll
            for (int ww = 0; ww < kRadix / 32; ++ww) at += ww < w ? S.scan[ww] : 0u;
            S.out[tid] = out - at;
            out += run;
#pragma unroll
            for (int ww = 0; ww < kWarps; ++ww) {
                const uint32_t c = S.wcnt[ww][tid];
                S.wcnt[ww][tid] = (uint16_t)at;
                at += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kPairs; ++r) {
            if (at0 + 32 * r < cnt) {
                const uint32_t slot = S.wcnt[w][(uint32_t)(k[r] >> shift) & mask] + ((rk[r / 2] >> (16 * (r & 1))) & 0xFFFFu);
                S.keys[slot] = k[r];
                S.vals[slot] = v[r];
            }
        }
        __syncwarp();
        zero_counters();  // of this warp, the only one that still reads them
        load(t0 + kTile);
        __syncthreads();
        for (uint32_t slot = tid; slot < cnt; slot += Cfg::threads) {
            const Key key = S.keys[slot];
            const uint32_t op = S.out[(uint32_t)(key >> shift) & mask] + slot;
            keys_out[op] = key;
            vals_out[op] = S.vals[slot];
        }
    }
}

// Few pairs: every pass in one CTA, the keys and the pairs' original places in
// shared memory (a launch instead of three per pass, and no trips through L2).
// A warp owns `rounds` x 32 consecutive pairs, in registers while a pass moves
// them; the values are fetched by place at the end.  By the launches of all
// passes / by this one, voxelisation and sort (us): 30-bit keys (12 launches), 2k
// points 121 / 109, 6k 129 / 121, 8k 130 / 123, 10k 131 / 134, 16k 131 / 159; 63
// bits (24 launches), 2k 158 / 120, 8k 171 / 158, 10k 169 / 171, 16k 172 / 210;
// 32-bit keys of a render, 3k Gaussians 171 / 155, 8k 211 / 209, 16k 240 / 260.
constexpr uint32_t kSmallMax = 8192, kSmallThreads = 1024, kSmallRounds = kSmallMax / kSmallThreads;

template <typename Key>
struct SmallSmem {
    Key keys[kSmallMax];
    uint16_t place[kSmallMax];
    uint16_t cnt[kSmallThreads / 32][kRadix];
    uint32_t first[kRadix];  // first slot of each digit
    uint32_t scan[33];
};

template <typename Key>
__global__ void __launch_bounds__(kSmallThreads, 1) small_sort_kernel(const Key *keys,
                                                                      const uint32_t *vals, uint32_t n,
                                                                      uint32_t nbits, uint32_t width, uint32_t rounds,
                                                                      Key *keys_out,
                                                                      uint32_t *vals_out)
{
    if (after_previous()) return;
    extern __shared__ __align__(16) unsigned char small_raw[];
    SmallSmem<Key> &S = *reinterpret_cast<SmallSmem<Key> *>(small_raw);
    const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5, at0 = w * rounds * 32 + lane;
    const uint32_t ltmask = lanemask_lt();
    Key k[kSmallRounds];
    uint32_t pl[kSmallRounds / 2], rk[kSmallRounds / 2];  // two 16-bit values each: places, ranks
#pragma unroll
    for (uint32_t r = 0; r < kSmallRounds; ++r) {
        const uint32_t at = at0 + r * 32;
        k[r] = r < rounds && at < n ? keys[at] : Key(0);
        pl[r / 2] = (r & 1) ? (pl[r / 2] | (at << 16)) : (at & 0xFFFFu);
    }
    const uint32_t mask = (1u << width) - 1u;
    for (uint32_t shift = 0; shift < nbits; shift += width) {
        uint32_t *zero = reinterpret_cast<uint32_t *>(S.cnt[w]);
#pragma unroll
        for (uint32_t i = 0; i < kRadix / 64; ++i) zero[lane + 32 * i] = 0u;
        __syncwarp();
#pragma unroll
        for (uint32_t r = 0; r < kSmallRounds; ++r) {
            if (r >= rounds) break;
            const bool ok = at0 + r * 32 < n;
            const uint32_t d = (uint32_t)(k[r] >> shift) & mask;
            const uint32_t peers = same_digit(d, ok, mask), before = __popc(peers & ltmask);
            const uint32_t base = S.cnt[w][d];
            __syncwarp();
            if (ok && before == 0) S.cnt[w][d] = (uint16_t)(base + __popc(peers));
            __syncwarp();
            rk[r / 2] = (r & 1) ? (rk[r / 2] | ((base + before) << 16)) : (base + before);
        }
        __syncthreads();
        // per digit: exclusive prefix over the warps, then the digits' first slots
        uint32_t run = 0;
        if (tid < kRadix) {
#pragma unroll
            for (uint32_t ww = 0; ww < kSmallThreads / 32; ++ww) {
                const uint32_t c = S.cnt[ww][tid];
                S.cnt[ww][tid] = (uint16_t)run;
                run += c;
            }
        }
        uint32_t tot;
        const uint32_t pre = block_exclusive_sum<uint32_t>(run, S.scan, &tot);
        if (tid < kRadix) S.first[tid] = pre;
        __syncthreads();
#pragma unroll
        for (uint32_t r = 0; r < kSmallRounds; ++r) {
            if (r < rounds && at0 + r * 32 < n) {
                const uint32_t d = (uint32_t)(k[r] >> shift) & mask;
                const uint32_t slot = S.first[d] + S.cnt[w][d] + ((rk[r / 2] >> (16 * (r & 1))) & 0xFFFFu);
                S.keys[slot] = k[r];
                S.place[slot] = (uint16_t)(pl[r / 2] >> (16 * (r & 1)));
            }
        }
        __syncthreads();
#pragma unroll
        for (uint32_t r = 0; r < kSmallRounds; ++r) {
            const uint32_t at = at0 + r * 32;
            if (r < rounds && at < n) {
                k[r] = S.keys[at];
                const uint32_t p = S.place[at];
                pl[r / 2] = (r & 1) ? ((pl[r / 2] & 0xFFFFu) | (p << 16)) : ((pl[r / 2] & 0xFFFF0000u) | p);
            }
        }
    }
#pragma unroll
    for (uint32_t r = 0; r < kSmallRounds; ++r) {
        const uint32_t at = at0 + r * 32;
        if (r < rounds && at < n) {
            keys_out[at] = k[r];
            vals_out[at] = vals[(pl[r / 2] >> (16 * (r & 1))) & 0xFFFFu];
        }
    }
}

template <typename Key>
void small_sort(const Key *keys, const uint32_t *vals, Key *keys_out, uint32_t *vals_out, uint32_t n, uint32_t nbits,
                cudaStream_t s)
{
    allow_shared<small_sort_kernel<Key>>();
    launch_after(small_sort_kernel<Key>, 1, kSmallThreads, sizeof(SmallSmem<Key>), s, 
        keys, vals, n, nbits, digit_width(nbits), (n + kSmallThreads - 1) / kSmallThreads, keys_out, vals_out);
    count_launch();
}

}  // namespace

uint64_t radix_sort_hist_words(uint64_t n, int num_sms, uint32_t segments)
{
    return (uint64_t)kRadix * (sort_ctas_bound(n, num_sms) + segments) + kRadix;
}

uint64_t radix_sort_max_ctas(uint64_t n, int num_sms) { return sort_ctas_bound(n, num_sms); }

uint32_t radix_sort_segment_table(const uint64_t *seg_lo, uint32_t segments, int num_sms, uint64_t *cta_lo,
                                  uint32_t *cta_seg)
{
    const uint64_t n = seg_lo[segments];
    const SortGeom g = sort_geom(n, num_sms);
    uint32_t P = 0;
    for (uint32_t f = 0; f < segments; ++f) {
        const uint64_t b = seg_lo[f], e = seg_lo[f + 1];
        const uint32_t p0 = P;
        for (uint64_t x = b; x < e; x += g.chunk) cta_lo[P++] = x;
        for (uint32_t p = p0; p < P; ++p) cta_seg[2 * p] = p0;
        for (uint32_t p = p0; p < P; ++p) cta_seg[2 * p + 1] = P;
    }
    cta_lo[P] = n;
    return P;
}

template <typename Key, typename Cfg>
static void launch_down(const Key *keys, const uint32_t *vals, uint64_t n, uint32_t shift, uint32_t mask, uint64_t chunk,
                        const uint32_t *hist, Key *keys_out, uint32_t *vals_out, const uint64_t *cta_lo,
                        const uint32_t *cta_seg, uint32_t P, cudaStream_t s)
{
    constexpr size_t smem = sizeof(DownSmem<Key, Cfg>);
    allow_shared<downsweep_kernel<Key, Cfg>>();
    launch_after(downsweep_kernel<Key, Cfg>, P, Cfg::threads, smem, s, keys, vals, n, shift, mask, chunk, hist, keys_out, vals_out,
                                                             cta_lo, cta_seg);
    count_launch();
}

template <typename Key>
static bool sort_passes(Key *keys, uint32_t *vals, Key *keys_alt, uint32_t *vals_alt, uint32_t *hist,
                        uint64_t n, uint32_t nbits, uint32_t P, uint64_t chunk, const uint64_t *cta_lo,
                        const uint32_t *cta_seg, int num_sms, cudaStream_t s)
{
    Key *ki = keys, *ko = keys_alt;
    uint32_t *vi = vals, *vo = vals_alt;
    bool flipped = false;
    const bool large = sort_large(n, num_sms);
    const uint32_t width = digit_width(nbits), mask = (1u << width) - 1u;
    for (uint32_t shift = 0; shift < nbits; shift += width) {
        if (large)
            launch_after(upsweep_kernel<Key, SortLarge::threads>, P, SortLarge::threads, 0, s, ki, n, shift, mask, chunk, hist, cta_lo);
        else
            launch_after(upsweep_kernel<Key, SortSmall::threads>, P, SortSmall::threads, 0, s, ki, n, shift, mask, chunk, hist, cta_lo);
        count_launch();
        launch_after(scan_cols_kernel, kRadix / 8, 256, 0, s, hist, P);
        count_launch();
        if (large)
            launch_down<Key, SortLarge>(ki, vi, n, shift, mask, chunk, hist, ko, vo, cta_lo, cta_seg, P, s);
        else
            launch_down<Key, SortSmall>(ki, vi, n, shift, mask, chunk, hist, ko, vo, cta_lo, cta_seg, P, s);
        Key *tk = ki;
        ki = ko;
        ko = tk;
        uint32_t *tv = vi;
        vi = vo;
        vo = tv;
        flipped = !flipped;
    }
    return flipped;
}

template <typename Key>
bool radix_sort(Key *keys, uint32_t *vals, Key *keys_alt, uint32_t *vals_alt, uint32_t *hist, uint64_t n,
                uint32_t nbits, int num_sms, cudaStream_t s)
{
    if (n <= 1 || nbits == 0) return false;
    if (n <= kSmallMax) {
        small_sort(keys, vals, keys_alt, vals_alt, (uint32_t)n, nbits, s);
        return true;
    }
    const SortGeom g = sort_geom(n, num_sms);
    return sort_passes(keys, vals, keys_alt, vals_alt, hist, n, nbits, g.P, g.chunk, nullptr, nullptr, num_sms, s);
}
template bool radix_sort<uint64_t>(uint64_t *, uint32_t *, uint64_t *, uint32_t *, uint32_t *, uint64_t, uint32_t, int,
                                   cudaStream_t);
template bool radix_sort<uint32_t>(uint32_t *, uint32_t *, uint32_t *, uint32_t *, uint32_t *, uint64_t, uint32_t, int,
                                   cudaStream_t);

bool radix_sort_segments(uint64_t *keys, uint32_t *vals, uint64_t *keys_alt, uint32_t *vals_alt, uint32_t *hist,
                         uint64_t n, uint32_t nbits, uint32_t ctas, const uint64_t *cta_lo, const uint32_t *cta_seg,
                         int num_sms, cudaStream_t s)
{
    if (n <= 1 || nbits == 0 || ctas == 0) return false;
    return sort_passes(keys, vals, keys_alt, vals_alt, hist, n, nbits, ctas, sort_geom(n, num_sms).chunk, cta_lo,
                       cta_seg, num_sms, s);
}

}  // namespace gsnfs
