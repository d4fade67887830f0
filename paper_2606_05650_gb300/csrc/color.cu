// KLT of the SH colour decorrelation (Sec. 4): per frame, the covariance of
// each YUV channel's 15 AC values over the frame's first (up to 4096) input
// points, and its eigenvectors; rows of K = eigenvectors by decreasing
// eigenvalue, the largest component of each made positive.  Everything here
// is FP64: the YUV
// values of the sample, per-slice means and centred co-moments (64 slices of
// 64 rows), the slices combined in a fixed order by the
// pairwise update of Chan, Golub and LeVeque, and cyclic Jacobi rotations
// (seven disjoint rotations at a time).  K is rounded to
// FP32 once, for the header and the per-row transforms.  The frame's
// centring constants are then carried into the same domain.
#include "color.cuh"
#include "kernels.cuh"

namespace gsnfs {

namespace {

constexpr int kSample = 4096;
constexpr int kSlices = 64;                   // CTAs per frame for the sample sums
constexpr int kSliceRows = kSample / kSlices;  // 64
constexpr int kPairs = kKltN * (kKltN + 1) / 2;  // 120
constexpr int kPartWords = 3 * (kPairs + kKltN) + 1;  // per slice: co-moments, then means, per channel; row count

__device__ __forceinline__ void pair_of(int p, int &x, int &y)
{
    x = 0;
    while (x < kKltN && p >= kKltN - x) {
        p -= kKltN - x;
        ++x;
    }
    y = x + p;
}

// BT.601 analogue YUV of one SH function's RGB in FP64, each product and sum
// rounded separately (the order of the definition: m0 x + m1 y + m2 z)
__device__ __forceinline__ double yuv_f64(const float *row, int k, int ch)
{
    const double M[9] = {0.299, 0.587, 0.114, -0.14713, -0.28886, 0.436, 0.615, -0.51499, -0.10001};
    const double x = row[sh_chan(k, 0)], y = row[sh_chan(k, 1)], z = row[sh_chan(k, 2)];
    return __dadd_rn(__dadd_rn(__dmul_rn(M[3 * ch], x), __dmul_rn(M[3 * ch + 1], y)), __dmul_rn(M[3 * ch + 2], z));
}

// GB300 issues one FP64 warp instruction in some 16 cycles per SM, so the
// estimate is bound by the FP64 instructions that share an SM: every (slice,
// YUV channel) and every (frame, channel) has a CTA of its own, and the lanes
// of a warp are kept busy with independent elements (one warp per channel on
// one SM took 63 + 769 us for a frame).  The encoder runs it beside the
// voxelisation and the sort: encode and reconstruction of a 1M-Gaussian frame
// in colour mode 2.33 -> 1.83 ms.

// grid (slices, frames, 3 YUV channels), 4 warps: the mean and the centred
// co-moments (sums of products of deviations) of one slice of the frame's
// first 4096 input rows; a thread per pair of AC functions
__global__ void __launch_bounds__(128) klt_partials_kernel(const float *const *attr, const uint64_t *poff,
                                                           double *part)
{
    __shared__ double rows[kSliceRows][kKltN];  // the channel's AC values
    __shared__ double mean[kKltN];
    const uint32_t f = blockIdx.y, sl = blockIdx.x;
    const int t = threadIdx.x, ch = blockIdx.z;
    const uint64_t n = poff[f + 1] - poff[f];
    const int m = (int)(n < (uint64_t)kSample ? n : (uint64_t)kSample);
    const int rb = sl * kSliceRows, re = (rb + kSliceRows) < m ? (rb + kSliceRows) : m;
    const int cnt_rows = re > rb ? re - rb : 0;
    const float *a = attr[f];
    for (int e = t; e < cnt_rows * kKltN; e += blockDim.x) {
        const int r = e / kKltN, k = e - r * kKltN;
        rows[r][k] = yuv_f64(a + (uint64_t)(rb + r) * 56, k + 1, ch);
    }
    __syncthreads();
    if (t < kKltN) {
        double sum = 0.0;
        for (int r = 0; r < cnt_rows; ++r) sum = __dadd_rn(sum, rows[r][t]);
        mean[t] = cnt_rows ? __ddiv_rn(sum, (double)cnt_rows) : 0.0;
    }
    __syncthreads();
    double *ps = part + ((uint64_t)f * kSlices + sl) * kPartWords;
    double *o = ps + ch * (kPairs + kKltN);
    if (t < kPairs) {
        int px, py;
        pair_of(t, px, py);
        const double mx = mean[px], my = mean[py];
        double acc = 0.0;
        for (int r = 0; r < cnt_rows; ++r)
            acc = __dadd_rn(acc, __dmul_rn(__dsub_rn(rows[r][px], mx), __dsub_rn(rows[r][py], my)));
        o[t] = acc;
    }
    if (t < kKltN) o[kPairs + t] = mean[t];
    if (t == 0 && ch == 0) ps[kPartWords - 1] = (double)cnt_rows;
}

// grid (frames, 3 YUV channels), 4 warps: covariance from the slices (pairwise
// update, fixed order, FP64; a thread per pair), eigenvectors by cyclic Jacobi
// (FP64), ordering and signs; K rounded to FP32
__global__ void __launch_bounds__(128) klt_solve_kernel(const uint64_t *poff, const double *part, float *klt)
{
    __shared__ double S[kKltN * kKltN];
    __shared__ double V[kKltN * kKltN];
    __shared__ double mu[kKltN];
    __shared__ double cs[7][2];
    __shared__ int pq[7][2];
    __shared__ int order[kKltN];
    __shared__ int stop;
    const uint32_t f = blockIdx.x;
    const int t = threadIdx.x, lane = t & 31, ch = blockIdx.y;
    const uint64_t n = poff[f + 1] - poff[f];
    const int m = (int)(n < (uint64_t)kSample ? n : (uint64_t)kSample);
    const double *pf = part + (uint64_t)f * kSlices * kPartWords;
    // running combination over slices: count nA, mean muA (t < 15), co-moments CA (a pair per thread)
    double nA = 0.0, muA = 0.0, CA = 0.0;
    int px = 0, py = 0;
    if (t < kPairs) pair_of(t, px, py);
    for (int sl = 0; sl < kSlices; ++sl) {
        const double *ps = pf + (uint64_t)sl * kPartWords;
        const double nB = ps[kPartWords - 1];
        if (nB == 0.0) continue;
        const double *o = ps + ch * (kPairs + kKltN);
        const double nAB = __dadd_rn(nA, nB);
        const double w = __ddiv_rn(__dmul_rn(nA, nB), nAB);
        // delta of the means for both coordinates of each pair (read from this slice's and the running means)
        if (t < kKltN) mu[t] = __dsub_rn(o[kPairs + t], muA);  // delta_k = muB_k - muA_k
        __syncthreads();
        if (t < kPairs) CA = __dadd_rn(__dadd_rn(CA, o[t]), __dmul_rn(w, __dmul_rn(mu[px], mu[py])));
        if (t < kKltN) muA = __dadd_rn(muA, __dmul_rn(mu[t], __ddiv_rn(nB, nAB)));
        nA = nAB;
        __syncthreads();
    }
    const double inv_m = m ? 1.0 / (double)m : 0.0;
    if (t < kPairs) {
        const double c = __dmul_rn(CA, inv_m);
        S[px * kKltN + py] = c;
        S[py * kKltN + px] = c;
    }
    for (int e = t; e < kKltN * kKltN; e += blockDim.x) V[e] = (e / kKltN == e % kKltN) ? 1.0 : 0.0;
    __syncthreads();
    double tr2 = 0.0;
    for (int k = 0; k < kKltN; ++k) tr2 += S[k * kKltN + k] * S[k * kKltN + k];
    // Jacobi sweeps in parallel order: 15 rounds of 7 disjoint (p, q) pairs (a
    // round-robin over the 15 indices and one idle slot), the 7 rotations of a
    // round computed from the same S and applied together (they act on
    // disjoint rows and columns); every pair is met once per sweep.  Stop when
    // the off-diagonal mass is down to FP64 rounding of the diagonal.
    constexpr int kTasks = 7 * kKltN;  // (pair, row) of a round
    for (int sweep = 0; sweep < 20; ++sweep) {
        if (t < 32) {
            double off = 0.0;
            if (lane < kKltN)
                for (int q = lane + 1; q < kKltN; ++q) off += S[lane * kKltN + q] * S[lane * kKltN + q];
            for (int o = 16; o; o >>= 1) off += __shfl_xor_sync(0xFFFFFFFFu, off, o);
            if (t == 0) stop = !(off > 1e-28 * tr2);
        }
        __syncthreads();
        if (stop) break;
        for (int rd = 0; rd < kKltN; ++rd) {
            if (t < 7) {
                const int a = (rd + t + 1) % kKltN, b = (rd - t - 1 + kKltN) % kKltN;
                const int p = a < b ? a : b, q = a < b ? b : a;
                const double apq = S[p * kKltN + q];
                double c = 1.0, sn = 0.0;
                if (fabs(apq) > 1e-300) {
                    const double theta = (S[q * kKltN + q] - S[p * kKltN + p]) / (2.0 * apq);
                    const double tt = (theta >= 0.0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
                    c = 1.0 / sqrt(tt * tt + 1.0);
                    sn = tt * c;
                }
                cs[t][0] = c;
                cs[t][1] = sn;
                pq[t][0] = p;
                pq[t][1] = q;
            }
            __syncthreads();
            for (int e = t; e < 2 * kTasks; e += blockDim.x) {  // columns p, q of S and of V
                const int x = e < kTasks ? e : e - kTasks, i = x / kKltN, row = x - i * kKltN;
                const int p = pq[i][0], q = pq[i][1];
                const double c = cs[i][0], sn = cs[i][1];
                double *M = (e < kTasks ? S : V) + row * kKltN;
                const double kp = M[p], kq = M[q];
                M[p] = c * kp - sn * kq;
                M[q] = sn * kp + c * kq;
            }
            __syncthreads();
            for (int e = t; e < kTasks; e += blockDim.x) {  // rows p, q of S
                const int i = e / kKltN, col = e - i * kKltN;
                const int p = pq[i][0], q = pq[i][1];
                const double c = cs[i][0], sn = cs[i][1];
                const double spk = S[p * kKltN + col], sqk = S[q * kKltN + col];
                S[p * kKltN + col] = c * spk - sn * sqk;
                S[q * kKltN + col] = sn * spk + c * sqk;
            }
            __syncthreads();
        }
    }
    if (t == 0) {  // decreasing eigenvalue, stable
        for (int k = 0; k < kKltN; ++k) order[k] = k;
        for (int x = 0; x < kKltN; ++x)
            for (int y = x + 1; y < kKltN; ++y)
                if (S[order[y] * kKltN + order[y]] > S[order[x] * kKltN + order[x]]) {
                    const int tmp = order[x];
                    order[x] = order[y];
                    order[y] = tmp;
                }
    }
    __syncthreads();
    float *Kf = klt + (uint64_t)f * kKltFloats + ch * kKltN * kKltN;
    if (t < kKltN) {
        const int e = order[t];
        int big = 0;
        for (int k = 1; k < kKltN; ++k)
            if (fabs(V[k * kKltN + e]) > fabs(V[big * kKltN + e])) big = k;
        const double sg = V[big * kKltN + e] < 0.0 ? -1.0 : 1.0;
        for (int k = 0; k < kKltN; ++k) Kf[t * kKltN + k] = (float)(sg * V[k * kKltN + e]);
    }
}

// the frames' centres into the decorrelated domain, in the order of the row transforms
__global__ void __launch_bounds__(64) klt_centre_kernel(const float *klt, float *center)
{
    __shared__ float row[56];
    const int t = threadIdx.x;
    float *c = center + (uint64_t)blockIdx.x * 56;
    if (t < 56) row[t] = c[t];
    __syncthreads();
    if (t < 16) color_yuv_task(row, t, kYuvFwd);
    __syncthreads();
    float out = 0.f;
    const int ch = t / kKltN, r = t - ch * kKltN;
    if (t < 3 * kKltN) {
        const float *Kr = klt + (uint64_t)blockIdx.x * kKltFloats + (ch * kKltN + r) * kKltN;
        for (int k = 0; k < kKltN; ++k) out = __fadd_rn(out, __fmul_rn(Kr[k], row[11 + kKltN * ch + k]));
    }
    __syncthreads();
    if (t < 3 * kKltN) row[11 + t] = out;
    __syncthreads();
    if (t < 56) c[t] = row[t];
}

}  // namespace

YuvInv yuv_inverse()
{
    const double m[3][3] = {{0.299, 0.587, 0.114}, {-0.14713, -0.28886, 0.436}, {0.615, -0.51499, -0.10001}};
    const double det = m[0][0] * (m[1][1] * m[2][2] - m[1][2] * m[2][1]) -
                       m[0][1] * (m[1][0] * m[2][2] - m[1][2] * m[2][0]) +
                       m[0][2] * (m[1][0] * m[2][1] - m[1][1] * m[2][0]);
    const double inv[9] = {(m[1][1] * m[2][2] - m[1][2] * m[2][1]) / det, (m[0][2] * m[2][1] - m[0][1] * m[2][2]) / det,
                           (m[0][1] * m[1][2] - m[0][2] * m[1][1]) / det, (m[1][2] * m[2][0] - m[1][0] * m[2][2]) / det,
                           (m[0][0] * m[2][2] - m[0][2] * m[2][0]) / det, (m[0][2] * m[1][0] - m[0][0] * m[1][2]) / det,
                           (m[1][0] * m[2][1] - m[1][1] * m[2][0]) / det, (m[0][1] * m[2][0] - m[0][0] * m[2][1]) / det,
                           (m[0][0] * m[1][1] - m[0][1] * m[1][0]) / det};
    YuvInv r;
    for (int i = 0; i < 9; ++i) r.m[i] = (float)inv[i];
    return r;
}

uint64_t color_klt_partial_words(uint32_t F) { return (uint64_t)F * kSlices * kPartWords; }

void launch_color_klt(const float *const *attr, const uint64_t *poff, uint32_t F, float *klt, float *center,
                      double *partials, cudaStream_t s)
{
    if (F == 0) return;
    klt_partials_kernel<<<dim3(kSlices, F, 3), 128, 0, s>>>(attr, poff, partials);
    count_launch();
    klt_solve_kernel<<<dim3(F, 3), 128, 0, s>>>(poff, partials, klt);
    count_launch();
    if (center) {
        klt_centre_kernel<<<F, 64, 0, s>>>(klt, center);
        count_launch();
    }
}

}  // namespace gsnfs
