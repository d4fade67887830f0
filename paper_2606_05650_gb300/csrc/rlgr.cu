// Quantisation and block RLGR entropy coding of RAHT coefficients
// (Sec. 3.4 "Quantization and Entropy Coding"; App. H, Table A.5).
//
// Each attribute channel is cut into blocks of B consecutive coefficients
// (Morton / in-place order of the transform output) and every block is one
// independent adaptive run-length Golomb-Rice stream coded by one thread
// (the paper's block parallelisation).  Threads of a CTA are the channels of
// one block of rows, so the row-major coefficient matrix is read row by row
// with coalesced loads; the quantiser (dead-zone / uniform, per group step)
// is applied on the fly.  RLGR constants (Malvar 2006 reading):
//   u = zigzag(q); k = K >> 4, kR = KR >> 4; K = 0, KR = 32 at block start.
//   k == 0: GR(u, kR); u == 0 -> K += 3 (cap 240), else K -= 3 (floor 0).
//   k >  0: a full run of 2^k zeros -> bit 0, K += 4; r < 2^k zeros then
//           u != 0 -> bit 1, r in k bits, GR(u - 1, kR), K -= 6; a run cut
//           by the block end -> bit 0 (the decoder clamps).
//   GR(v, k): p = v >> k; p < 24 -> p ones, a zero, the k low bits of v;
//            else 24 ones, 6-bit length n of v, the n bits of v.
//            p == 0 -> KR -= 2 (floor 0); p > 1 -> KR += p + 1 (cap 384).
//   Bits are packed least-significant first into 32-bit words; a block ends
//   on a word boundary.  At most 78 bits per coefficient.
#include <algorithm>

#include "kernels.cuh"

namespace gsnfs {

namespace {

constexpr int kUnaryEsc = 24;

// Bits are appended LSB first to a 64-bit accumulator holding nacc < 32 bits:
// one wide multiply-add by 2^nacc places a value (its bits are free there), a
// full low word is stored.  Words beyond `cap` are counted but not stored.
struct BitWriter {
    uint64_t acc;
    uint32_t nacc;
    uint32_t unit;  // 2^nacc
    uint32_t nw;
    uint32_t *out;
    uint32_t cap;
    __device__ __forceinline__ BitWriter(uint32_t *o, uint32_t c) : acc(0), nacc(0), unit(1), nw(0), out(o), cap(c) {}
    __device__ __forceinline__ void put(uint32_t v, uint32_t n)  // n <= 32, v < 2^n
    {
        acc += (uint64_t)v * unit;
        nacc += n;
        const bool full = nacc >= 32u;
        asm volatile("{\n.reg .pred f;\nsetp.ge.u32 f, %4, 32;\nsetp.lt.and.u32 f, %1, %2, f;\n@f st.global.u32 [%0], %3;\n}" ::"l"(
                         out + nw),
                     "r"(nw), "r"(cap), "r"((uint32_t)acc), "r"(nacc)
                     : "memory");  // one predicated store, no branch
        nw += full ? 1u : 0u;
        acc = full ? acc >> 32 : acc;
        nacc &= 31u;
        unit = 1u << nacc;
    }
    __device__ __forceinline__ void flush()
    {
        if (nacc) put(0u, 32u - nacc);
    }
};

// Golomb-Rice codewords by table.  The encoder's entry, for the mode, the
// parameter k (row) and column 2 t + s (magnitude t, sign s; zigzag index
// u = 2 t - s, or 0), is the codeword of u (of u - 1 in run mode; 16 bits),
// the change of KR (8 bits, signed) and the codeword's length n (8 bits); the
// decoder's, for k and the next 10 stream bits, is n, the changes of KR and K
// (signed) and the value + 128 that the codeword stands for in Golomb-Rice
// mode, 8 bits each.  Entry 0 sends the symbol to the general path: codewords
// longer than 16 (encoder) or 10 bits (decoder) and values that do not fit.
// One shared-memory load replaces the prefix and remainder arithmetic and the
// adaptation's comparisons.  The coders are bound by instruction issue, most
// of it on the half-rate integer pipe: one serial stream per thread, every
// stream slot of the SM filled.  With the tables 44 (encoder) and 51 (decoder)
// warp instructions per 32 symbols, 64 each before: 16 x 1M frames, encode 1.78
// -> 1.36 ms; a ladder of eight frames and five rungs 2.25 -> 1.69 ms; decode,
// at 32 warps per SM, 1.45 ms alone.  Large coefficients are past the tables, and
// so past their gain: what codes them without is chosen below.
constexpr uint32_t kEncRows = 8, kEncCols = 256;   // per mode: k 0 .. 7
constexpr uint32_t kEncMax = kEncCols / 2 - 1;     // magnitudes below; kEncMax stands for every larger one
constexpr uint32_t kEncMode = kEncRows * kEncCols;  // entries of one mode
constexpr uint32_t kDecRows = 8, kDecBits = 10;    // k 0 .. 7

struct EncTable {
    uint32_t e[2 * kEncMode];
};
struct DecTable {
    uint32_t e[kDecRows << kDecBits];
};

constexpr int kr_change(uint32_t p) { return p >= 2 ? (int)p + 1 : (p == 1 ? 0 : -2); }

constexpr EncTable make_enc_table()
{
    EncTable t{};
    for (uint32_t run = 0; run < 2; ++run)
        for (uint32_t k = 0; k < kEncRows; ++k)
            for (uint32_t i = 0; i < 2 * kEncMax; ++i) {
                const uint32_t m = i >> 1, u = (i & 1u) && m ? 2 * m - 1 : 2 * m;
                uint32_t &e = t.e[run * kEncMode + k * kEncCols + i];
                if (run && u == 0) {  // a zero of a run: no codeword (not an entry of the general path either)
                    e = 1u << 24;
                    continue;
                }
                const uint32_t v = u - run, p = v >> k, n = p + 1 + k, low = v & ((1u << k) - 1u);
                if (n > 16) continue;
                e = ((((low << 1) | 1u) << p) - 1u) | (((uint32_t)kr_change(p) & 0xFFu) << 16) | (n << 24);
            }
    return t;
}

constexpr DecTable make_dec_table()
{
    DecTable t{};
    for (uint32_t k = 0; k < kDecRows; ++k)
        for (uint32_t x = 0; x < (1u << kDecBits); ++x) {
            uint32_t p = 0;
            while (p < kDecBits && ((x >> p) & 1u)) ++p;
            const uint32_t n = p + 1 + k;
            if (n > kDecBits) continue;
            const uint32_t u = (p << k) | ((x >> (p + 1)) & ((1u << k) - 1u));
            const int q = (u & 1u) ? -(int)(u >> 1) - 1 : (int)(u >> 1);
            if (q < -128 || q > 127) continue;
            t.e[(k << kDecBits) | x] = n | (((uint32_t)kr_change(p) & 0xFFu) << 8) |
                                       (((uint32_t)(u == 0 ? 3 : -3) & 0xFFu) << 16) | ((uint32_t)(q + 128) << 24);
        }
    return t;
}

__device__ const EncTable g_enc_table = make_enc_table();
__device__ const DecTable g_dec_table = make_dec_table();

template <int BYTE>
__device__ __forceinline__ int signed_byte(uint32_t e)
{
    int r;
    asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(e), "n"(BYTE | (0x888 | (BYTE * 0x111)) << 4));
    return r;
}

template <typename Table>
__device__ __forceinline__ void stage_table(Table *dst, const Table *src)
{
    static_assert(sizeof(Table) % 16 == 0, "copied in 16-byte words");
    uint4 *d = reinterpret_cast<uint4 *>(dst);
    const uint4 *q = reinterpret_cast<const uint4 *>(src);
    for (uint32_t i = threadIdx.x; i < sizeof(Table) / 16; i += blockDim.x) d[i] = __ldg(q + i);
}

__device__ __forceinline__ uint32_t zz(int32_t q)
{
    return q >= 0 ? ((uint32_t)q << 1) : ((((uint32_t)(-(q + 1))) << 1) | 1u);
}

__device__ __forceinline__ int32_t unzz(uint32_t u)
{
    return (u & 1u) ? -(int32_t)(u >> 1) - 1 : (int32_t)(u >> 1);
}

__device__ __forceinline__ void adapt_kr(uint32_t p, int &KR)
{
    // p = 0: KR - 2, p = 1: unchanged, p > 1: KR + p + 1; within [0, 384]
    const int d = p >= 2u ? (int)(p > 384u ? 384u : p) + 1 : (p == 1u ? 0 : -2);
    KR = min(max(KR + d, 0), 384);
}

__device__ __forceinline__ void gr_put(BitWriter &bw, uint32_t v, uint32_t k, int &KR)
{
    const uint32_t p = v >> k;
    if (__builtin_expect(p + 1u + k <= 32u && p < (uint32_t)kUnaryEsc, 1)) {  // common case: one write
        // p ones, a zero, then the k low bits of v, least significant first:
        // ((2 low + 1) << p) - 1, where low = v mod 2^k (k <= 24)
        const uint32_t low = v & ((1u << k) - 1u);
        bw.put((((low << 1) | 1u) << p) - 1u, p + 1u + k);
    } else if (p < (uint32_t)kUnaryEsc) {
        bw.put((1u << p) - 1u, p + 1u);
        bw.put(v & ((1u << k) - 1u), k);
    } else {
        const uint32_t n = 32u - (uint32_t)__clz(v);
        bw.put((1u << kUnaryEsc) - 1u, kUnaryEsc);
        bw.put(n, 6);
        bw.put(v, n);
    }
    adapt_kr(p, KR);
}

// A value that is the same in every lane, in a register of each: left to
// itself the compiler reloads it for every symbol.
__device__ __forceinline__ uint32_t in_register(uint32_t x) { return __shfl_sync(0xFFFFFFFFu, x, 0); }
__device__ __forceinline__ float in_register(float x) { return __shfl_sync(0xFFFFFFFFu, x, 0); }

__device__ __forceinline__ uint32_t shared_address(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// from a table (not written after the CTA's first barrier)
__device__ __forceinline__ uint32_t table_load(uint32_t a)
{
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}

// Table column 2 t + s of a coefficient, t its magnitude by quantize_f32 up to
// kEncMax, plus kColBias: the floor by adding 2^23 rounded towards zero, the
// sign bit shifted in below it.
constexpr uint32_t kColBias = 2u * 0x4B000000u;

__device__ __forceinline__ uint32_t column_f32(float y, float inv_step, float tau)
{
    const float t = fminf(__fadd_rn(__fmul_rn(fabsf(y), inv_step), tau), (float)kEncMax);  // a NaN: kEncMax
    return __funnelshift_l(__float_as_uint(y), __float_as_uint(__fadd_rz(t, 8388608.0f)), 1);
}

__device__ __forceinline__ uint32_t column_i32(int32_t q)
{
    const uint32_t m = q < 0 ? 0u - (uint32_t)q : (uint32_t)q;
    return kColBias + 2u * min(m, kEncMax) + (q < 0 ? 1u : 0u);
}

// RLGR state of one block; code() takes any symbol, by its zigzag index, each lane on its own path.
struct RlgrState {
    int K, KR;
    uint32_t z;  // pending zeros of an open run
    __device__ __forceinline__ void code(BitWriter &bw, uint32_t u)
    {
        const uint32_t k = (uint32_t)K >> 4;
        if (__builtin_expect(k == 0, 1)) {  // Golomb-Rice mode
            gr_put(bw, u, (uint32_t)KR >> 4, KR);
            K = max(K + (u == 0 ? 3 : -3), 0);
        } else if (u == 0) {
            if (++z == (1u << k)) {
                bw.put(0, 1);
                K = min(K + 4, 240);
                z = 0;
            }
        } else {
            bw.put(1u | (z << 1), 1u + k);  // bit 1, then the run length in k bits (z < 2^k, k <= 15)
            gr_put(bw, u - 1u, (uint32_t)KR >> 4, KR);
            K = max(K - 6, 0);
            z = 0;
        }
    }
    __device__ __forceinline__ void finish(BitWriter &bw)
    {
        if (z) bw.put(0, 1);
        bw.flush();
    }
};

// RLGR coder of one block by table.
struct Rlgr : RlgrState {
    uint32_t tab;  // shared-memory address of the table, less the bias of its columns
    __device__ __forceinline__ void init(const EncTable &t)
    {
        K = 0;
        KR = 32;
        z = 0;
        tab = in_register(shared_address(t.e) - 4u * kColBias);
    }
    static __device__ __forceinline__ int next_kr(int kr, uint32_t e)
    {
        return __viaddmin_s32_relu(kr, signed_byte<2>(e), 384);
    }
    // Parameters at which so many symbols lie past the table that a warp is better off without it (deviations of some
    // 50 steps; 100k rows of 45 / 60 steps, with the line 8 lower: 95 / 100 us, here 71 / 95).
    __device__ __forceinline__ bool large() const { return KR >= 16 * (int)kEncRows - 16; }
    // Two symbols in Golomb-Rice mode (K < 16: no cap at 240), appended by one write; false, with nothing changed,
    // when the table does not hold one of the codewords.  Wants ready(): the first symbol raises K by 3 and KR by 16
    // at most, which leaves the second in Golomb-Rice mode and in the table's rows.
    __device__ __forceinline__ bool ready() const { return K < 13 && !large(); }
    __device__ __forceinline__ bool pair(BitWriter &bw, uint32_t a, uint32_t b)
    {
        const uint32_t e0 = table_load((uint32_t)(KR & 0x1F0) * (kEncCols / 4) + tab + 4u * a);
        const int kr1 = next_kr(KR, e0);
        const uint32_t e1 = table_load((uint32_t)(kr1 & 0x1F0) * (kEncCols / 4) + tab + 4u * b);
        if (e0 == 0u || e1 == 0u) return false;
        KR = next_kr(kr1, e1);
        K = __viaddmax_s32(K, a < kColBias + 2u ? 3 : -3, 0);
        K = __viaddmax_s32(K, b < kColBias + 2u ? 3 : -3, 0);
        const uint32_t n0 = e0 >> 24;
        bw.put((e0 & 0xFFFFu) + (e1 & 0xFFFFu) * (1u << n0), n0 + (e1 >> 24));
        return true;
    }
    // One symbol in either mode, without branches for the mode; false, with nothing changed, when the table does not
    // hold its codeword.  In run mode (k > 0) a nonzero is bit 1, the run length in k bits (z < 2^k, k <= 15), then
    // its codeword; in Golomb-Rice mode k and z are 0.  The 2^k-th zero of a run is bit 0.
    __device__ __forceinline__ bool one(BitWriter &bw, uint32_t a)
    {
        const uint32_t k = (uint32_t)K >> 4, run = min(k, 1u);
        const uint32_t e = table_load((uint32_t)(KR & 0x70) * (kEncCols / 4) + run * (4u * kEncMode) + tab + 4u * a);
        if (e == 0u || KR >= 16 * (int)kEncRows) return false;
        const bool zero = a < kColBias + 2u, more = zero && K >= 16;
        const uint32_t z1 = z + 1u, full = z1 >> k;  // used in a run only: z1 <= 2^k
        const uint32_t npre = k + run, c = ((e & 0xFFFFu) << npre) + (2u * z + run), n = npre + (e >> 24);
        const int dk = zero ? (more ? 4 * (int)full : 3) : -3 - 3 * (int)run;
        K = __viaddmin_s32_relu(K, dk, 240);
        KR = next_kr(KR, e);
        z = more && !full ? z1 : 0u;
        bw.put(more ? 0u : c, more ? full : n);
        return true;
    }
};

// ---- encoder: one CTA per rb row blocks; thread = (row block, rung, channel) --
// Each thread copies its channel's coefficients into a ring of its own in
// shared memory by cp.async (lanes of a warp are consecutive channels of a
// row, so a warp's copy of a row is one contiguous run), kRing - kPrefetch
// rows ahead of the one being coded: registers for that many rows would cost
// more resident warps than they hide.  Threads never wait for each other after
// the CTA's one barrier.  Threads of the other rungs of a row read the same
// words (served by L1).
struct EncJobs {
    RlgrJob j;
    const uint64_t *job_off;  // F + 1: first job (row block) of each frame
    uint32_t w0, ws;          // the launch codes streams w0 .. w0 + ws - 1 of each row block (kernel of a thread a stream)
    uint64_t least, most;     // and nothing unless the streams, known on the device only, number least .. most
    __device__ __forceinline__ bool concerned() const
    {
        const uint64_t n = job_off[j.F] * j.R * j.C;
        return n >= least && n <= most;
    }
};

constexpr uint32_t kPrefetch = 4;  // rows copied and coded at a time; even, for the rows are coded in pairs
constexpr uint32_t kRing = 16;     // rows of a ring

// Row blocks per CTA: enough that rb * W (W = rungs x channels threads per
// row block) fills whole warps (rb = 32 / gcd(W, 32)), at most 512 threads.
__host__ __device__ inline uint32_t row_blocks_per_cta(uint32_t W)
{
    uint32_t g = 32;
    while (W % g) g >>= 1;
    uint32_t rb = 32 / g;
    if (rb * W > 512) rb = W >= 512 ? 1 : 512 / W;
    return rb;
}

// asynchronous copy of the word p[r * step] to shared memory at dst + OFF; a load from at + OFF
template <uint32_t OFF>
__device__ __forceinline__ void copy_word(uint32_t dst, const uint32_t *p, uint32_t r, uint32_t step)
{
    asm volatile("{\n.reg .u64 a;\nmad.wide.u32 a, %1, %2, %3;\ncp.async.ca.shared.global [%0+%4], [a], 4;\n}" ::"r"(dst),
                 "r"(r), "r"(4u * step), "l"(p), "n"(OFF)
                 : "memory");
}
template <uint32_t OFF>
__device__ __forceinline__ uint32_t ring_load(uint32_t at)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(at), "n"(OFF) : "memory");
    return v;
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait()  // all but the latest N groups have arrived
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ uint32_t shared_load(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

struct EncBlock {  // one row block of a CTA
    uint64_t gbase;  // first coefficient (row-major) of the block
    uint32_t f, b, nb, len;
};

// row block `job` of the batch (length 0 past the last)
__device__ __forceinline__ EncBlock enc_block(const EncJobs &E, uint64_t job)
{
    const RlgrJob &j = E.j;
    EncBlock e{0, 0, 0, 0, 0};
    if (job < E.job_off[j.F]) {
        uint32_t lo = 0, hi = j.F;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (E.job_off[mid] <= job) lo = mid; else hi = mid;
        }
        const uint32_t vs = j.vstart[lo], nv = j.vstart[lo + 1] - vs;
        e.f = lo;
        e.b = (uint32_t)(job - E.job_off[lo]);
        e.nb = (nv + j.B - 1) / j.B;
        const uint32_t row0 = e.b * j.B;
        e.len = (nv - row0) < j.B ? (nv - row0) : j.B;
        e.gbase = ((uint64_t)vs + row0) * j.C;
    }
    return e;
}

// PITCH: threads of a CTA at most
template <bool FROM_INT, bool DIST, uint32_t PITCH>
__global__ void __launch_bounds__(PITCH, 1024 / PITCH) rlgr_encode_kernel(EncJobs E, const int32_t *qin, uint32_t rb)
{
    if (after_previous()) return;
    if (!E.concerned()) return;
    extern __shared__ uint32_t ring[];  // kRing x PITCH
    __shared__ EncBlock blk_info[32];
    __shared__ __align__(16) EncTable tab;
    stage_table(&tab, &g_enc_table);
    const RlgrJob &j = E.j;
    const uint32_t C = j.C, W = E.ws;
    const uint32_t t = threadIdx.x;
    if (t < rb) blk_info[t] = enc_block(E, (uint64_t)blockIdx.x * rb + t);
    __syncthreads();
    // lanes past the last stream do that stream's work once more and write nothing
    const bool spare = t >= rb * W;
    const uint32_t tt = spare ? rb * W - 1u : t, jl = tt / W, w = E.w0 + tt - jl * W;
    const EncBlock me = blk_info[jl];
    const uint32_t r = w / C, c = w - r * C;
    const uint64_t blk = j.blk_off[me.f] + ((uint64_t)r * me.nb + me.b) * C + c;
    BitWriter bw(j.slots + blk * j.slot_words, spare ? 0u : j.slot_words);
    Rlgr st;
    st.init(tab);
    const float inv = FROM_INT ? 0.f : j.inv_step[r * C + c];
    const float stp = DIST ? j.step[r * C + c] : 0.f;
    float sq = 0.f;
    double dc_err = 0.0;
    const uint32_t *src = FROM_INT ? reinterpret_cast<const uint32_t *>(qin) : reinterpret_cast<const uint32_t *>(j.Y);
    const uint32_t *col = src + me.gbase + c;  // row i of this channel at col[i * C]
    const uint32_t len = me.len;
    uint32_t i = 0;
    if (!FROM_INT && j.dc && me.b == 0 && me.len) {  // the frame's DC: quantised from its FP64 value
        const double y = j.dc[(uint64_t)me.f * C + c], st64 = j.steps_rg[r * j.G + j.groups[c]];
        const int32_t q = quantize_f64(y, st64, j.tau64);
        st.code(bw, zz(q));
        if (DIST) {
            const double e = __dsub_rn(y, __dmul_rn((double)q, st64));
            dc_err = __dmul_rn(e, e);
        }
        i = 1;
    }
    const float tau = in_register(j.tau);
    auto index_of = [&](uint32_t x) {
        return FROM_INT ? zz((int32_t)x) : quantize_zz_f32(__uint_as_float(x), inv, tau);
    };
    auto column_of = [&](uint32_t x) {
        return FROM_INT ? column_i32((int32_t)x) : column_f32(__uint_as_float(x), inv, tau);
    };
    auto distort = [&](uint32_t x) {  // squared error of the dequantised coefficient (Parseval: of the attributes)
        const float y = __uint_as_float(x);
        const float e = __fsub_rn(y, __fmul_rn((float)quantize_f32(y, inv, tau), stp));
        sq = __fadd_rn(sq, __fmul_rn(e, e));
    };
    // a lane's whole groups of kPrefetch rows; the warp stays together to the end of its longest block (a frame's
    // last block is shorter)
    const uint32_t groups = (len - i) / kPrefetch;
    const uint32_t common = __reduce_min_sync(0xFFFFFFFFu, groups), longest = __reduce_max_sync(0xFFFFFFFFu, groups);
    constexpr uint32_t kRow = 4u * PITCH, kGroup = kPrefetch * kRow, kBytes = kRing * kRow;  // bytes in the ring
    const uint32_t mine = in_register(shared_address(ring)) + 4u * t;
    uint32_t next = 0, slot = 0;  // group to copy, and its place
    auto copy_group = [&] {
        if (next < groups) {
            const uint32_t at = mine + slot, r = i + next * kPrefetch;
            copy_word<0>(at, col, r, C);
            copy_word<kRow>(at, col, r + 1, C);
            copy_word<2 * kRow>(at, col, r + 2, C);
            copy_word<3 * kRow>(at, col, r + 3, C);
        }
        static_assert(kPrefetch == 4, "copies of a group");
        copies_commit();
        ++next;
        slot = (slot + kGroup) % kBytes;
    };
    auto code_group = [&](bool live) {
        copies_wait<kRing / kPrefetch - 2>();
        const uint32_t from = mine + (slot + kGroup) % kBytes;
        const uint32_t x[kPrefetch] = {ring_load<0>(from), ring_load<kRow>(from), ring_load<2 * kRow>(from),
                                       ring_load<3 * kRow>(from)};
        copy_group();  // over the group before this one
        // One lane whose parameter is large takes its warp through the general path, one in run mode (or near it)
        // through the path for either mode; what the table does not hold is left to the general path too, by each lane.
        // (With the table tried again for every such symbol, a warp of large coefficients went through all the paths:
        // 100k rows of 56 channels of 120 steps 201 us, now 95; 1M rows of 100 steps 416 -> 221; a frame of 250k
        // Gaussians at the base steps 78 -> 57, the 8 x 5 ladder 1.78 -> 1.69 ms.)
        const bool large = __any_sync(0xFFFFFFFFu, live && st.large());
#pragma unroll
        for (uint32_t d = 0; d < kPrefetch; d += 2) {
            bool done = __all_sync(0xFFFFFFFFu, !live || st.ready());
            if (!live) continue;
            const uint32_t a = column_of(x[d]), b = column_of(x[d + 1]);
            if (done) done = st.pair(bw, a, b);
            if (!done) {
                const uint32_t coded = large ? 0u : st.one(bw, a) ? (st.one(bw, b) ? 2u : 1u) : 0u;
                if (coded == 0u) st.code(bw, index_of(x[d]));
                if (coded != 2u) st.code(bw, index_of(x[d + 1]));
            }
            if (DIST) {
                distort(x[d]);
                distort(x[d + 1]);
            }
        }
    };
#pragma unroll
    for (uint32_t g = 0; g + 1 < kRing / kPrefetch; ++g) copy_group();
    for (uint32_t g = 0; g < common; ++g) code_group(true);
    for (uint32_t g = common; g < longest; ++g) code_group(g < groups);
    copies_wait<0>();
    i += groups * kPrefetch;
    if (i < len) {  // fewer than kPrefetch rows
        uint32_t x[kPrefetch - 1];
#pragma unroll
        for (uint32_t d = 0; d + 1 < kPrefetch; ++d) x[d] = i + d < len ? *(col + (uint64_t)(i + d) * C) : 0u;
#pragma unroll 1
        for (uint32_t d = 0; i < len; ++i, ++d) {
            const uint32_t y = d == 0 ? x[0] : (d == 1 ? x[1] : x[2]);
            if (!st.one(bw, column_of(y))) st.code(bw, index_of(y));
            if (DIST) distort(y);
        }
    }
    if (len == 0 || spare) return;
    st.finish(bw);
    j.block_words[blk] = bw.nw;
    if (bw.nw > j.slot_words) atomicExch(j.overflow, 1u);
    if (DIST) atomicAdd(j.sq_err + ((uint64_t)me.f * j.R + r) * C + c, __dadd_rn((double)sq, dc_err));
}

// ---- encoder for few streams ----------------------------------------------------
// A launch takes as long as one stream does, and a thread that codes a symbol at
// a time spends some 200 cycles on each, one instruction after another.  Only
// the adaptation is serial, so here a CTA takes kSplitG streams in segments of
// kSplitSeg symbols and splits the work: one warp walks the adaptation, a lane
// per stream, and notes the state before each symbol (a fifth of the
// instructions while no stream is near run mode); a warp per stream then forms
// the segment's codewords, a lane per symbol, places them by a scan of their
// lengths and writes whole words, while the first walks the next segment and
// the one after it is loaded and quantised.  By the kernel above / by this one:
// 10k Gaussians (1.1k streams) 57 / 42 us, 30k 57 / 47, 40k 57 / 50; a cloud of 1M
// points (mostly runs) 84 / 47.  In all it takes more instructions, and where an
// SM has more than its four CTAs it loses: 45k Gaussians (4.9k streams) 57 / 80,
// 100k 57 / 130.  How many streams there are is known on the device (a cloud has
// far fewer voxels than points): up to kSplitBound times as many points as would
// make four CTAs an SM, both kernels are launched and the streams' number says
// which one works (encode of a cloud of 1.3M points 543 -> 482 us).
constexpr uint32_t kSplitCtas = 4, kSplitBound = 4;
constexpr uint32_t kSplitG = 8, kSplitSeg = 128, kSplitThreads = 32 * (1 + kSplitG);
constexpr uint32_t kSplitRow = kSplitG + 1;  // of a symbol's row in shared memory: no bank twice down a column

// state before a symbol: K (8 bits), KR (9 bits), pending zeros of an open run (15 bits)
__device__ __forceinline__ uint32_t split_state(uint32_t K, uint32_t KR, uint32_t z) { return K | KR << 8 | z << 17; }

// adapt_kr; p <= 2^31
__device__ __forceinline__ uint32_t adapted(uint32_t KR, uint32_t p)
{
    const uint32_t down = (uint32_t)max((int)KR - 2, 0), up = min(KR + p + 1u, 384u);
    return p == 0u ? down : (p == 1u ? KR : up);
}

// n <= 64 bits c at bit o of a zeroed buffer, least significant first (c < 2^n)
__device__ __forceinline__ void or_bits(uint32_t *buf, uint32_t o, uint64_t c)
{
    const uint32_t s = o & 31u;
    uint32_t *at = buf + (o >> 5);
    const uint64_t x = c << s;
    const uint32_t lo = (uint32_t)x, mid = (uint32_t)(x >> 32), hi = s ? (uint32_t)(c >> (64u - s)) : 0u;
    if (lo) atomicOr(at, lo);
    if (mid) atomicOr(at + 1, mid);
    if (hi) atomicOr(at + 2, hi);
}

__global__ void __launch_bounds__(kSplitThreads, 4) rlgr_encode_split_kernel(EncJobs E)
{
    if (after_previous()) return;
    if (!E.concerned()) return;
    __shared__ uint32_t sym[3][kSplitSeg * kSplitRow];  // zigzag indices of a segment
    __shared__ uint32_t pre[2][kSplitSeg * kSplitRow];  // states before its symbols
    __shared__ uint32_t bits[kSplitG][84];            // 32 codewords of up to 78 bits behind a part of a word
    __shared__ uint32_t s_len[kSplitG], s_open[kSplitG];
    const RlgrJob &j = E.j;
    const uint32_t C = j.C, W = j.R * C, lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    // a lane of the first warp and a whole later warp are a stream's; the loading threads, eight streams a row
    const uint32_t g = warp == 0 ? lane & (kSplitG - 1u) : warp - 1u, gl = threadIdx.x & (kSplitG - 1u);
    const auto block_of = [&](uint32_t gg, uint32_t &w) {
        const uint64_t stream = (uint64_t)blockIdx.x * kSplitG + gg, job = stream / W;
        w = (uint32_t)(stream - job * W);
        return enc_block(E, job);
    };
    uint32_t w, wl;
    const EncBlock me = block_of(g, w), ld = block_of(gl, wl);
    const uint32_t r = w / C, c = w - r * C, rl = wl / C, cl = wl - rl * C;
    if (warp == 0 && lane < kSplitG) s_len[lane] = me.len;
    __syncthreads();
    uint32_t longest = 0;
#pragma unroll
    for (uint32_t k = 0; k < kSplitG; ++k) longest = max(longest, s_len[k]);
    const uint32_t segs = (longest + kSplitSeg - 1) / kSplitSeg;
    // loading (warps 1 .. kSplitG): symbol at + kSplitSeg / kPer * h of the segment, of stream gl
    constexpr uint32_t kPer = kSplitSeg * kSplitG / (32 * kSplitG);
    const uint32_t at = (threadIdx.x - 32u) / kSplitG;
    const float inv = ld.len ? j.inv_step[rl * C + cl] : 0.f, tau = j.tau;
    const float *col = j.Y + ld.gbase + cl;
    float val[kPer];
    const auto load = [&](uint32_t seg) {
#pragma unroll
        for (uint32_t h = 0; h < kPer; ++h) {
            const uint32_t i = seg * kSplitSeg + at + kSplitSeg / kPer * h;
            val[h] = i < ld.len ? *(col + (uint64_t)i * C) : 0.f;
        }
    };
    const auto put_symbols = [&](uint32_t seg) {
        uint32_t *to = sym[seg % 3u];
#pragma unroll
        for (uint32_t h = 0; h < kPer; ++h)
            to[(at + kSplitSeg / kPer * h) * kSplitRow + gl] = quantize_zz_f32(val[h], inv, tau);
        if (seg == 0 && at == 0 && ld.len && j.dc && ld.b == 0)  // the frame's DC: quantised from its FP64 value
            to[gl] = zz(quantize_f64(j.dc[(uint64_t)ld.f * C + cl], j.steps_rg[rl * j.G + j.groups[cl]], j.tau64));
    };
    if (warp) {
        load(0);
        put_symbols(0);
    }
    __syncthreads();
    uint32_t K = 0, KR = 32, z = 0;                // the first warp's, a stream per lane
    uint32_t words = 0, part = 0, nbits = 0;       // a later warp's stream: whole words written, the bits after them
    const uint64_t blk = j.blk_off[me.f] + ((uint64_t)r * me.nb + me.b) * C + c;
    uint32_t *out = j.slots + blk * j.slot_words;
    for (uint32_t seg = 0; seg <= segs; ++seg) {
        if (warp == 0) {
            if (seg < segs && lane < kSplitG) {
                const uint32_t *u_at = sym[seg % 3u] + lane;
                uint32_t *pre_at = pre[seg & 1u] + lane;
                const uint32_t left = me.len > seg * kSplitSeg ? me.len - seg * kSplitSeg : 0u;
                for (uint32_t i = 0; i < kSplitSeg; i += 4) {
                    uint32_t u[4];
#pragma unroll
                    for (uint32_t h = 0; h < 4; ++h) u[h] = u_at[(i + h) * kSplitRow];
                    if (__all_sync((1u << kSplitG) - 1u, K < 4u && i + 4 <= left)) {  // four in Golomb-Rice mode: K + 3 each at most
#pragma unroll
                        for (uint32_t h = 0; h < 4; ++h) {
                            pre_at[(i + h) * kSplitRow] = split_state(K, KR, 0u);
                            const uint32_t p = u[h] >> (KR >> 4);
                            KR = adapted(KR, p);
                            K = (uint32_t)max((int)K + (u[h] == 0u ? 3 : -3), 0);
                        }
                        continue;
                    }
#pragma unroll
                    for (uint32_t h = 0; h < 4; ++h) {
                        pre_at[(i + h) * kSplitRow] = split_state(K, KR, z);
                        if (i + h >= left) continue;  // after the stream's end
                        const bool run = K >= 16u, zero = u[h] == 0u, quiet = run && zero;
                        const uint32_t k = K >> 4, z1 = z + 1u, full = z1 >> k;  // z1 <= 2^k in a run
                        const uint32_t p = (u[h] - (run ? 1u : 0u)) >> (KR >> 4);  // not used when quiet
                        if (!quiet) KR = adapted(KR, p);
                        const int dk = quiet ? (full ? 4 : 0) : (run ? -6 : (zero ? 3 : -3));
                        K = (uint32_t)min(max((int)K + dk, 0), 240);
                        z = quiet && !full ? z1 : 0u;
                    }
                }
                s_open[lane] = z;
            }
        } else {
            if (seg + 1 < segs) load(seg + 1);
            for (uint32_t q = 0; seg > 0 && q < kSplitSeg && (seg - 1) * kSplitSeg + q < me.len; q += 32) {
                const uint32_t i = q + lane;
                uint32_t n = 0, npre = 0, cpre = 0;
                uint64_t code = 0;
                if ((seg - 1) * kSplitSeg + i < me.len) {
                    const uint32_t u = sym[(seg - 1) % 3u][i * kSplitRow + g], st = pre[(seg - 1) & 1u][i * kSplitRow + g];
                    const uint32_t k = (st >> 4) & 15u, kr = (st >> 12) & 31u, zr = st >> 17;
                    if (k && u == 0u) {
                        n = zr + 1u == 1u << k ? 1u : 0u;  // the 2^k-th zero of a run is bit 0
                    } else {
                        if (k) {  // bit 1, then the run length in k bits
                            npre = 1u + k;
                            cpre = 1u | zr << 1;
                        }
                        const uint32_t v = u - (k ? 1u : 0u), p = v >> kr;
                        if (p < (uint32_t)kUnaryEsc) {  // as gr_put
                            n = p + 1u + kr;
                            code = (((uint64_t)(v & ((1u << kr) - 1u)) << 1 | 1u) << p) - 1u;
                        } else {
                            const uint32_t len = 32u - (uint32_t)__clz(v);
                            n = kUnaryEsc + 6u + len;
                            code = (uint64_t)v << (kUnaryEsc + 6) | (uint64_t)len << kUnaryEsc | ((1u << kUnaryEsc) - 1u);
                        }
                    }
                }
                const uint32_t end = nbits + warp_inclusive_sum(npre + n);
                const uint32_t total = __shfl_sync(0xFFFFFFFFu, end, 31), whole = total >> 5;
                uint32_t *buf = bits[g];
                for (uint32_t x = lane; x <= whole; x += 32) buf[x] = x ? 0u : part;
                __syncwarp();
                if (npre) or_bits(buf, end - n - npre, cpre);
                if (n) or_bits(buf, end - n, code);
                __syncwarp();
                for (uint32_t x = lane; x < whole; x += 32)
                    if (words + x < j.slot_words) out[words + x] = buf[x];
                part = buf[whole];
                words += whole;
                nbits = total & 31u;
                __syncwarp();
            }
            if (seg + 1 < segs) put_symbols(seg + 1);
        }
        __syncthreads();
    }
    if (warp && lane == 0 && me.len) {
        if (s_open[g]) ++nbits;  // an open run at the end: bit 0
        if (nbits) {
            if (words < j.slot_words) out[words] = part;
            ++words;
        }
        j.block_words[blk] = words;
        if (words > j.slot_words) atomicExch(j.overflow, 1u);
    }
}

// ---- decoder ------------------------------------------------------------------
// Bits are looked at through a 32-bit window over two consecutive words
// (cur, nxt) at bit offset pos; the word after them (ahead) is in a register
// too, so that no lane's refill makes the warp wait for a load.  The words
// come from a ring of four 16-byte pieces per thread in shared memory that the
// thread tops up by cp.async (top_up, every four symbols); a stream that drains
// it in between is read from global memory.  Words past the end of a stream
// read as zero, so a malformed stream cannot make the reader leave it; whether
// the stream was overrun is checked once, after its last coefficient, from the
// bits consumed.  Word numbers count from the 16-byte boundary at or below the
// stream's first word.
constexpr uint32_t kRingWords = 16, kPieces = kRingWords / 4;

struct WinReader {
    const uint32_t *base;  // the 16-byte boundary
    uint32_t ring;         // shared-memory address of the ring (aligned to its size)
    uint32_t lead, end;    // byte offsets of the stream's first word and of its end
    uint32_t cur, nxt, ahead, pos;
    uint32_t at;      // byte offset of the word after `ahead`
    uint32_t issued;  // pieces asked for; and as that was at the ends of the last three calls of top_up
    uint32_t issued1, issued2, issued3;
    uint32_t ready;   // bytes below have arrived

    __device__ __forceinline__ uint32_t ring_word(uint32_t o) const
    {
        return shared_load(ring | (o & (4u * kRingWords - 4u)));
    }
    __device__ __forceinline__ void issue()
    {
        const uint32_t bytes = (uint32_t)min(max((int)end - 16 * (int)issued, 0), 16);  // the rest: zeros
        const uint32_t dst = ring | (16u * (issued & (kPieces - 1u)));
        const uint32_t *src = base + 4 * (bytes ? issued : 0u);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
        ++issued;
    }
    __device__ __forceinline__ void init(const uint32_t *p, uint32_t n, const uint32_t *r)
    {
        lead = (uint32_t)((uintptr_t)p & 12u);
        base = p - lead / 4;
        ring = shared_address(r);
        end = lead + 4u * n;
        issued = 0;
#pragma unroll
        for (uint32_t k = 0; k < kPieces; ++k) issue();
        copies_commit();
        copies_wait<0>();
        issued1 = issued2 = issued3 = issued;
        ready = 16u * issued;
        cur = ring_word(lead);
        nxt = ring_word(lead + 4u);
        ahead = ring_word(lead + 8u);
        pos = 0;
        at = lead + 12u;
    }
    // Asks for the piece that the reader comes to next, once the one whose place it takes has been read; a piece is
    // taken to have arrived at the third call after.  True when the ring holds the two words that may be wanted
    // before the next call (skip_ready).
    __device__ __forceinline__ bool top_up()
    {
        copies_wait<2>();
        ready = 16u * issued3;
        issued3 = issued2;
        issued2 = issued1;
        issued = max(issued, at >> 4);
        if (at + 16u * (kPieces - 1u) >= 16u * issued) issue();
        issued1 = issued;
        copies_commit();
        return stocked();
    }
    __device__ __forceinline__ bool stocked() const { return at + 8u <= ready; }
    __device__ __forceinline__ uint32_t peek() const { return __funnelshift_r(cur, nxt, pos); }
    __device__ __forceinline__ void skip(uint32_t n)  // n <= 32
    {
        pos += n;
        if (pos >= 32u) {
            pos -= 32u;
            cur = nxt;
            nxt = ahead;
            ahead = at < ready ? ring_word(at) : (at < end ? base[at >> 2] : 0u);
            at += 4u;
        }
    }
    // the same when the ring holds the next word: no branch
    __device__ __forceinline__ void skip_ready(uint32_t n)
    {
        pos += n;
        asm volatile("{\n.reg .pred f;\n.reg .u32 a;\nsetp.ge.u32 f, %4, 32;\n"
                     "@f mov.u32 %0, %1;\n@f mov.u32 %1, %2;\n"
                     "lop3.b32 a, %3, %6, %5, 0xEA;\n@f ld.shared.u32 %2, [a];\n@f add.u32 %3, %3, 4;\n}"
                     : "+r"(cur), "+r"(nxt), "+r"(ahead), "+r"(at)
                     : "r"(pos), "r"(ring), "n"(4 * kRingWords - 4));
        pos &= 31u;
    }
    __device__ __forceinline__ bool overrun() const
    {
        return (uint64_t)(at - 12u - lead) * 8u + pos > (uint64_t)(end - lead) * 8u;
    }
};

// Rare path of gr_read: the remainder crosses the window, or the escape code.
__device__ __forceinline__ uint32_t gr_read_slow(WinReader &r, uint32_t k, uint32_t p, bool &bad)
{
    if (p < (uint32_t)kUnaryEsc) {
        r.skip(p + 1u);
        const uint32_t v = (p << k) | (r.peek() & ((1u << k) - 1u));
        r.skip(k);
        return v;
    }
    r.skip(kUnaryEsc);  // 24 ones, a 6-bit length n, n bits of value
    const uint32_t n = r.peek() & 63u;
    r.skip(6);
    if (n > 32u) {
        bad = true;
        return 0;
    }
    const uint32_t y = r.peek();
    const uint32_t v = n == 32u ? y : (y & ((1u << n) - 1u));
    r.skip(n);
    return v;
}

// Golomb-Rice value with parameter k (<= 24): p ones and a zero, then k low
// bits; p >= 24 is the escape (24 ones, a 6-bit length n, n bits of value).
__device__ __forceinline__ uint32_t gr_read(WinReader &r, uint32_t k, int &KR, bool &bad)
{
    const uint32_t x = r.peek();
    uint32_t p = (uint32_t)__ffs(~x) - 1u;  // leading ones (all ones: wraps to >= 32)
    const uint32_t n = p + 1u + k;
    uint32_t v;
    if (__builtin_expect(p < (uint32_t)kUnaryEsc && n <= 32u, 1)) {  // prefix and remainder inside the window
        v = (p << k) | ((x >> (p + 1u)) & ((1u << k) - 1u));
        r.skip(n);
    } else {
        v = gr_read_slow(r, k, p, bad);
        p = v >> k;
    }
    adapt_kr(p, KR);
    return v;
}

// Decodes one block stream (len coefficients of one channel) to out[i * C],
// i < len: dequantised (times sc) or as indices.  A Golomb-Rice symbol whose
// codeword the table holds (TABLE), or whose codeword lies in the window (else),
// takes the short path; run mode (runs are kept as pending zeros, and the nonzero
// that ends a partial run as a pending value) and longer codewords the general one.
constexpr uint32_t kDecThreads = 512, kDecSmall = 128;
constexpr int kRunLeft = 1 << 16;  // flags in K: zeros or a value of an earlier run are still to be written,
constexpr int kDrained = 1 << 17;  // the ring may not hold the next words: only the general path, which checks

template <bool TO_INT, bool TABLE>
__device__ __forceinline__ void decode_stream(const DecTable *tab, uint32_t *ring, const uint32_t *wp, uint32_t nw,
                                              uint32_t len, uint32_t C, float sc, float *yout, int32_t *qout,
                                              DevState *st)
{
    WinReader r;
    r.init(wp, nw, ring);
    int K = 0, KR = 32;
    uint32_t zeros = 0;
    bool bad = false;
    int32_t pending = 0;  // written after the zeros; 0: nothing (a pending value is a nonzero)
    auto general = [&](uint32_t left) -> int32_t {  // left: coefficients of the block from this one on
        if (K & kRunLeft) {
            int32_t q = 0;
            if (zeros) {
                --zeros;
            } else {
                q = pending;
                pending = 0;
            }
            if (!zeros && !pending) K &= ~kRunLeft;
            return q;
        }
        K &= ~kDrained;
        const uint32_t k = (uint32_t)K >> 4;
        if (k == 0) {
            const uint32_t u = gr_read(r, (uint32_t)KR >> 4, KR, bad);
            K = max(K + (u == 0 ? 3 : -3), 0);
            return unzz(u);
        }
        const uint32_t x = r.peek();
        if (!(x & 1u)) {  // a full run of 2^k zeros (clamped at the block end)
            r.skip(1);
            zeros = min(1u << k, left) - 1u;
            K = min(K + 4, 240);
            if (zeros) K |= kRunLeft;
            return 0;
        }
        const uint32_t rr = (x >> 1) & ((1u << k) - 1u);  // rr < 2^k zeros, then a nonzero
        r.skip(1u + k);
        const uint32_t v = gr_read(r, (uint32_t)KR >> 4, KR, bad);
        if (rr >= left || v == 0xFFFFFFFFu) bad = true;
        K = max(K - 6, 0);
        const int32_t q = unzz(v + 1u);
        if (rr == 0) return q;
        zeros = rr - 1;
        pending = q;
        if (zeros | (uint32_t)pending) K |= kRunLeft;
        return 0;
    };
    const uint32_t ta = TABLE ? shared_address(tab->e) : 0u;
    auto by_table = [&](uint32_t i) {
        const uint32_t e = table_load((uint32_t)(KR & 0x70) * (4u << (kDecBits - 4)) + ta +
                                      4u * (r.peek() & ((1u << kDecBits) - 1u)));
        int32_t q;
        float y;
        // Golomb-Rice mode (K < 16, no flag set), a row and a codeword of the table
        if (__builtin_expect(e != 0u && K < 16 && KR < 16 * (int)kDecRows, 1)) {
            q = (int32_t)(e >> 24) - 128;
            y = __fadd_rn(__uint_as_float(__byte_perm(e, 0x4B000000u, 0x7443)), -8388736.0f);  // 2^23 + (q + 128)
            KR = __viaddmin_s32_relu(KR, signed_byte<1>(e), 384);
            K = __viaddmax_s32(K, signed_byte<2>(e), 0);
            r.skip_ready(e & 0xFFu);
        } else {
            q = general(len - i);
            y = (float)q;
            if (!r.stocked()) K |= kDrained;
        }
        if (TO_INT)
            qout[(uint64_t)i * C] = q;
        else
            yout[(uint64_t)i * C] = __fmul_rn(y, sc);
    };
    auto by_arithmetic = [&](uint32_t i) {
        const uint32_t x = r.peek(), k = (uint32_t)KR >> 4;
        const uint32_t p = (uint32_t)__ffs(~x) - 1u, n = p + 1u + k;  // leading ones (all ones: wraps)
        int32_t q;
        // Golomb-Rice mode (K < 16, no flag set), a codeword inside the window
        if (__builtin_expect(K < 16 && p < (uint32_t)kUnaryEsc && n <= 32u, 1)) {
            const uint32_t u = (p << k) | ((x >> (p + 1u)) & ((1u << k) - 1u));
            q = unzz(u);
            adapt_kr(p, KR);
            K = max(K + (u == 0 ? 3 : -3), 0);
            r.skip_ready(n);
        } else {
            q = general(len - i);
        }
        if (!r.stocked()) K |= kDrained;  // up to 32 bits a symbol: looked after at each
        if (TO_INT)
            qout[(uint64_t)i * C] = q;
        else
            yout[(uint64_t)i * C] = __fmul_rn((float)q, sc);
    };
    auto symbol = [&](uint32_t i) {
        if constexpr (TABLE)
            by_table(i);
        else
            by_arithmetic(i);
    };
    uint32_t i = 0;
    for (; i + 4 <= len; i += 4) {
        K = r.top_up() ? K & ~kDrained : K | kDrained;
#pragma unroll
        for (uint32_t h = 0; h < 4; ++h) symbol(i + h);
    }
    K = r.top_up() ? K & ~kDrained : K | kDrained;
#pragma unroll 1
    for (; i < len; ++i) symbol(i);
    copies_wait<0>();
    if (bad || r.overrun()) set_error(&st->err, kErrCorrupt);
}

// whole CTA: the decoder's table in shared memory, or null
template <bool TABLE>
__device__ __forceinline__ const DecTable *dec_table()
{
    if constexpr (TABLE) {
        __shared__ __align__(16) DecTable tab;
        stage_table(&tab, &g_dec_table);
        __syncthreads();
        return &tab;
    }
    return nullptr;
}

// One frame: thread (local row block jl, channel c) of CTA x decodes block
// b = x * rb + jl of channel c.  Streams at block_off[b*C+c] (words) when
// block_off is given, else at (b*C+c) * stride.
template <bool TO_INT, bool TABLE>
__global__ void __launch_bounds__(kDecThreads, 2) rlgr_decode_kernel(const uint32_t *payload, uint64_t payload_words,
                                                          const uint32_t *block_words, const uint64_t *block_off,
                                                          uint32_t stride, uint32_t nv, uint32_t C, uint32_t B,
                                                          const float *step, float *Y, int32_t *qout,
                                                          DevState *st)
{
    if (after_previous()) return;
    extern __shared__ __align__(128) uint32_t ring[];  // kRingWords per thread
    const DecTable *tab = dec_table<TABLE>();
    const uint64_t stream = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, b = stream / C;
    const uint32_t c = (uint32_t)(stream - b * C);
    const uint64_t row0 = b * B;
    if (row0 >= nv) return;
    const uint32_t len = (nv - row0) < B ? (uint32_t)(nv - row0) : B;
    const uint64_t blk = b * C + c;
    uint64_t off = block_off ? block_off[blk] : blk * stride;
    uint32_t nw = block_words[blk];
    if (off + nw > payload_words) {
        set_error(&st->err, kErrCorrupt);
        nw = 0;
        off = 0;
    }
    decode_stream<TO_INT, TABLE>(tab, ring + threadIdx.x * kRingWords, payload + off, nw, len, C, TO_INT ? 0.f : step[c],
                          TO_INT ? nullptr : Y + row0 * C + c, TO_INT ? qout + row0 * C + c : nullptr, st);
}

// All frames of a batch: row blocks numbered across frames (job_off), rb per CTA.
template <bool TABLE>
__global__ void __launch_bounds__(kDecThreads, 2) rlgr_decode_batch_kernel(const DecFrame *fr, uint32_t F,
                                                                const uint64_t *job_off, const uint32_t *bw_all,
                                                                const uint64_t *boff_all, const float *steps_all,
                                                                uint32_t C, float *Y, DevState *st)
{
    if (after_previous()) return;
    extern __shared__ __align__(128) uint32_t ring[];  // kRingWords per thread
    const DecTable *tab = dec_table<TABLE>();
    const uint64_t stream = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, job = stream / C;
    const uint32_t c = (uint32_t)(stream - job * C);
    if (job >= job_off[F]) return;
    uint32_t lo = 0, hi = F;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (job_off[mid] <= job) lo = mid; else hi = mid;
    }
    const DecFrame &d = fr[lo];
    const uint32_t b = (uint32_t)(job - job_off[lo]);
    const uint32_t row0 = b * d.B;
    const uint32_t len = (d.nv - row0) < d.B ? (d.nv - row0) : d.B;
    const uint64_t base = boff_all[d.blk_off];
    const uint64_t blk = d.blk_off + (uint64_t)b * C + c;
    uint64_t off = boff_all[blk] - base;
    uint32_t nw = bw_all[blk];
    if (off + nw > d.payload_words) {
        set_error(&st->err, kErrCorrupt);
        nw = 0;
        off = 0;
    }
    decode_stream<false, TABLE>(tab, ring + threadIdx.x * kRingWords, d.payload + off, nw, len, C, steps_all[(uint64_t)lo * C + c],
                         Y + ((uint64_t)d.vstart + row0) * C + c, nullptr, st);
}

__global__ void __launch_bounds__(kMaxFrames) job_offsets_kernel(const uint32_t *vstart, uint32_t F, uint32_t B, uint32_t R,
                                                                 uint32_t C, uint64_t *job_off, uint64_t *blk_off)
{
    if (after_previous()) return;
    __shared__ uint64_t sh[33];
    const uint32_t f = threadIdx.x;
    const uint64_t nb = f < F ? ((uint64_t)(vstart[f + 1] - vstart[f]) + B - 1) / B : 0ull;
    uint64_t tot;
    const uint64_t jo = block_exclusive_sum<uint64_t>(nb, sh, &tot);
    if (f < F) {
        job_off[f] = jo;
        blk_off[f] = jo * R * C;
    }
    if (f == 0) {
        job_off[F] = tot;
        blk_off[F] = tot * R * C;
    }
}

}  // namespace

// launch(E, row blocks per CTA, CTAs, threads) for each slice of at most 512 of a row block's W streams
template <typename Launch>
static void launch_slices(EncJobs E, uint32_t W, uint64_t jobs, Launch launch)
{
    const uint32_t slices = (W + 511) / 512, most = (W + slices - 1) / slices;
    for (E.w0 = 0; E.w0 < W; E.w0 += most) {
        E.ws = std::min(most, W - E.w0);
        const uint32_t rb = row_blocks_per_cta(E.ws);
        launch(E, rb, (uint32_t)((jobs + rb - 1) / rb), (rb * E.ws + 31) / 32 * 32);
        count_launch();
    }
}

template <bool FROM_INT, bool DIST>
static void launch_encode(const EncJobs &E, const int32_t *q, uint32_t W, uint64_t jobs, cudaStream_t s)
{
    launch_slices(E, W, jobs, [&](const EncJobs &S, uint32_t rb, uint32_t grid, uint32_t threads) {
        if (threads <= 256) {
            allow_shared<rlgr_encode_kernel<FROM_INT, DIST, 256>>();
            launch_after(rlgr_encode_kernel<FROM_INT, DIST, 256>, grid, threads, 4 * (size_t)kRing * 256, s, S, q, rb);
        } else {
            allow_shared<rlgr_encode_kernel<FROM_INT, DIST, 512>>();
            launch_after(rlgr_encode_kernel<FROM_INT, DIST, 512>, grid, threads, 4 * (size_t)kRing * 512, s, S, q, rb);
        }
    });
}

// A slot holds 16 bits per coefficient on average (ample for quantised
// attribute coefficients); the worst case is 78 bits per coefficient.
uint32_t rlgr_slot_words(uint32_t B, bool worst_case)
{
    return worst_case ? (uint32_t)(((uint64_t)78 * B + 31) / 32 + 2) : (uint32_t)(B / 2 + 4);
}

void launch_rlgr_offsets(const uint32_t *vstart, uint32_t F, uint32_t B, uint32_t R, uint32_t C, uint64_t *job_off,
                         uint64_t *blk_off, cudaStream_t s)
{
    launch_after(job_offsets_kernel, 1, kMaxFrames, 0, s, vstart, F, B, R, C, job_off, blk_off);
    count_launch();
}

void launch_rlgr_encode(const RlgrJob &j, const uint64_t *job_off, uint64_t jobs_bound, int num_sms, cudaStream_t s)
{
    if (jobs_bound == 0 || j.C == 0) return;
    const uint32_t W = j.R * j.C;
    const uint64_t streams = jobs_bound * W;  // at most: the host knows the points, the device the voxels
    const uint64_t split = (uint64_t)kSplitG * kSplitCtas * num_sms;
    EncJobs E{j, job_off, 0, W, 0, ~0ull};
    if (!j.sq_err && streams <= kSplitBound * split) {
        E.most = split;
        launch_after(rlgr_encode_split_kernel, (uint32_t)((std::min(streams, split) + kSplitG - 1) / kSplitG), kSplitThreads, 0, s, E);
        count_launch();
        if (streams <= split) return;
        E.least = split + 1;
        E.most = ~0ull;
    }
    if (j.sq_err)
        launch_encode<false, true>(E, nullptr, W, jobs_bound, s);
    else
        launch_encode<false, false>(E, nullptr, W, jobs_bound, s);
}

void launch_rlgr_encode_indices(const int32_t *q, const uint32_t *vstart, uint32_t C, uint32_t B, uint32_t *slots,
                                uint32_t slot_words, uint32_t *bw, const uint64_t *job_off, const uint64_t *blk_off,
                                uint64_t jobs_bound, uint32_t *overflow, cudaStream_t s)
{
    if (jobs_bound == 0 || C == 0) return;
    RlgrJob j{};
    j.C = C;
    j.B = B;
    j.R = 1;
    j.vstart = vstart;
    j.F = 1;
    j.slots = slots;
    j.block_words = bw;
    j.blk_off = blk_off;
    j.slot_words = slot_words;
    j.overflow = overflow;
    launch_encode<true, false>(EncJobs{j, job_off, 0, C, 0, ~0ull}, q, C, jobs_bound, s);
}

// Threads per CTA: a CTA has a copy of the table (32 KB) beside 64 bytes a thread, and many streams are bound by the
// integer pipe once 32 warps are resident: 16 x 1M frames, beside the same geometry kernels, 2.14 ms with 224 threads
// (28 warps), 1.83 with 512 (32), 1.74 with 640 (40), which slows the geometry, the longer branch, by more.  Streams
// that do not fill every SM twice that way take smaller CTAs, for the sake of all SMs.
template <auto Kernel, typename... A>
static void launch_decode(uint64_t streams, int num_sms, cudaStream_t s, A... args)
{
    const uint32_t threads = streams < (uint64_t)num_sms * 2 * kDecThreads ? kDecSmall : kDecThreads;
    allow_shared<Kernel>();
    launch_after(Kernel, (uint32_t)((streams + threads - 1) / threads), threads, 4 * (size_t)kRingWords * threads, s, args...);
    count_launch();
}

// By table, or by arithmetic: the table's path takes fewer instructions while the codewords are short; a warp with a lane
// whose codeword is not in it goes through the general path too, which arithmetic seldom needs.  4 frames of 1M
// Gaussians (whole decode, ms, by table / by arithmetic): 4.3 bits of payload a coefficient 1.29 / 1.40, 5.6 1.34 /
// 1.40, 6.0 1.44 / 1.41, 6.6 1.57 / 1.41, 10.1 1.70 / 1.41.  And it takes many streams: with few the arithmetic kernel is
// done sooner, but holds up the geometry beside it, the longer branch (6.6 bits: 250k Gaussians 411 / 461 us, 550k 527 /
// 524, 700k 569 / 547).
static bool decode_by_table(uint64_t streams, uint64_t payload_words, uint64_t coefficients, int num_sms)
{
    return streams < (uint64_t)num_sms * 448 || 32 * payload_words < 5.9 * coefficients;
}

void launch_rlgr_decode(const uint32_t *payload, uint64_t payload_words, const uint32_t *block_words,
                        const uint64_t *block_off, uint64_t nv, uint32_t C, uint32_t B, const float *step, float *Y,
                        DevState *st, int num_sms, cudaStream_t s)
{
    if (nv == 0 || C == 0) return;
    const uint64_t streams = (nv + B - 1) / B * C;
    auto go = [&](auto launch) {
        launch(streams, num_sms, s, payload, payload_words, block_words, block_off, 0u, (uint32_t)nv, C, B, step, Y, nullptr, st);
    };
    if (decode_by_table(streams, payload_words, nv * C, num_sms))
        go([](auto... a) { launch_decode<rlgr_decode_kernel<false, true>>(a...); });
    else
        go([](auto... a) { launch_decode<rlgr_decode_kernel<false, false>>(a...); });
}

void launch_rlgr_decode_batch(const DecFrame *fr, uint32_t F, const uint64_t *job_off, uint64_t jobs_bound,
                              uint64_t payload_words, uint64_t nv_total, const uint32_t *bw_all, const uint64_t *boff_all,
                              const float *steps_all, uint32_t C, float *Y, DevState *st, int num_sms, cudaStream_t s)
{
    if (jobs_bound == 0 || C == 0) return;
    if (decode_by_table(jobs_bound * C, payload_words, nv_total * C, num_sms))
        launch_decode<rlgr_decode_batch_kernel<true>>(jobs_bound * C, num_sms, s, fr, F, job_off, bw_all, boff_all, steps_all, C, Y, st);
    else
        launch_decode<rlgr_decode_batch_kernel<false>>(jobs_bound * C, num_sms, s, fr, F, job_off, bw_all, boff_all, steps_all, C, Y, st);
}

// (how many bits the streams hold is known on the device only: by arithmetic, which is done sooner but for many short ones)
void launch_rlgr_decode_indices(const uint32_t *words, uint64_t total_words, const uint32_t *bw, uint32_t stride,
                                uint64_t nv, uint32_t C, uint32_t B, int32_t *q, DevState *st, int num_sms, cudaStream_t s)
{
    if (nv == 0 || C == 0) return;
    launch_decode<rlgr_decode_kernel<true, false>>((nv + B - 1) / B * C, num_sms, s, words, total_words, bw, nullptr, stride,
                                                   (uint32_t)nv, C, B, nullptr, nullptr, q, st);
}

}  // namespace gsnfs
