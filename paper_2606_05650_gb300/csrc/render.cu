// Splat rasteriser for rendered-view quality of decoded frames (the standard
// 3DGS forward pass, from its definition): per Gaussian, the projected mean,
// the EWA 2-D covariance J R S S^T R^T J^T + 0.3 I and its inverse (conic),
// a footprint square of radius ceil(3 sqrt(largest eigenvalue)), opacity
// sigmoid(logit) and a degree-3 real-SH colour at the viewing direction; the
// Gaussians are sorted by depth, each then lists the 16 x 16 tiles it overlaps
// and the list is sorted stably by tile (so a tile's list is by depth, then
// input index); a warp composites its tile's list front to back for 8 x 4
// pixels.  Attributes are the
// 56-channel 3DGS rows: log-scale 0-2, rotation (w, x, y, z) 3-6, opacity
// logit 7, SH DC RGB 8-10, SH AC 11-55 as R[15] G[15] B[15].
//
// Precision: everything per Gaussian (projection, covariance, conic, tile
// rectangle, opacity, colour) is evaluated in FP64, or in double-float where
// that certainly rounds to the same float, and rounded once to FP32 for the
// per-pixel loop, which runs in FP32.  The projected centre is kept as an unevaluated sum of two floats,
// so a pixel's offset from it is exact to FP32 rounding of the offset itself (a
// single float would carry an absolute error of its ulp at hundreds of pixels).  The conic enters the
// loop through its Cholesky factor, conic = L^T L with
// L = [[l1, l2], [0, l3]]: the exponent is -(|L d|^2) / 2, a sum of two
// squares, which FP32 evaluates without cancellation even for elongated
// footprints.
#include "kernels.cuh"

namespace gsnfs {

namespace {

constexpr int kTile = 16;

struct Splat {
    float u, v;            // projected centre, rounded
    uint32_t reach;        // pixels from the centre, in x (upper half) and in y, past which alpha stays below the cut: the
                           // upper halves of floats, rounded up, infinite where there is no such bound
    float opacity;
    float ulo, vlo;        // the centre's rest: u + ulo, v + vlo
    float l1, l2, l3;      // Cholesky factor of the conic
    float r, g, b;
};

// upper half of a float's bits, rounded up (x >= 0 or infinite)
__device__ __forceinline__ uint32_t upper_half(float x) { return (__float_as_uint(x) + 0xFFFFu) >> 16; }

// Double-float arithmetic (an unevaluated sum h + l of two floats, about 2^-46
// relative; the error-free sums of Knuth and products of Dekker, by FMA).  An
// SM issues an FP64 warp instruction in 16 cycles and four FP32 ones a cycle,
// and the projection was bound by its FP64 instructions (some 640 a Gaussian):
// what is rounded to FP32 next, and is not the difference of nearly equal
// numbers, is double-float (viewing direction, colour, opacity), evaluated in
// FP64 after all where double-float cannot tell which float FP64 rounds to; the
// rest stays in FP64 (camera coordinates, squared scales, covariance,
// determinant, footprint), some 240.  1M Gaussians at 960 x 540: this kernel
// 1,024 us all in FP64, 413 us now (332 us with the squared scales in
// double-float too, which kept 46 of their 53 bits).
struct Df {
    float h, l;
};
__device__ __forceinline__ Df df_quick(float a, float b)  // |a| >= |b|
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ Df df_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ Df operator+(Df a, Df b)
{
    Df s = df_sum(a.h, b.h);
    const Df t = df_sum(a.l, b.l);
    s = df_quick(s.h, __fadd_rn(s.l, t.h));
    return df_quick(s.h, __fadd_rn(s.l, t.l));
}
__device__ __forceinline__ Df operator-(Df a) { return {-a.h, -a.l}; }
__device__ __forceinline__ Df operator-(Df a, Df b) { return a + (-b); }
__device__ __forceinline__ Df operator*(Df a, Df b)
{
    const float p = __fmul_rn(a.h, b.h);
    const float e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p)));
    return df_quick(p, e);
}
__device__ __forceinline__ Df operator*(Df a, float b)
{
    const float p = __fmul_rn(a.h, b);
    return df_quick(p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p)));
}
// whether every number within err of h + l rounds to h (err counts some 2^-40 of h: its own rounding is nothing to it)
__device__ __forceinline__ bool rounds_to_high(Df a, float err)
{
    return __fadd_rn(a.h, __fadd_rn(a.l, err)) == a.h && __fadd_rn(a.h, __fsub_rn(a.l, err)) == a.h;
}
__device__ __forceinline__ Df df_of(double x)
{
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}
__host__ __device__ constexpr Df df_const(double x)
{
    return {(float)x, (float)(x - (double)(float)x)};
}

// e^x, |x| <= 80: x = k ln 2 + r (Cody and Waite), Taylor's series of e^r with
// its terms to r^5 in double-float (the rest is below 3e-6 of the sum)
__device__ __forceinline__ Df df_exp(float x, int &k)
{
    const float kf = rintf(__fmul_rn(x, 1.44269504f));
    k = (int)kf;
    constexpr float kLn2Hi = 2839.f / 4096.f;  // the first 12 bits of ln 2: kf * kLn2Hi is exact
    constexpr Df kLn2Lo = df_const(0.693147180559945309417 - 2839.0 / 4096.0);
    const Df r = Df{__fmaf_rn(-kf, kLn2Hi, x), 0.f} + kLn2Lo * -kf;
    float t = 1.f / 479001600.f;
    t = __fmaf_rn(t, r.h, 1.f / 39916800.f);
    t = __fmaf_rn(t, r.h, 1.f / 3628800.f);
    t = __fmaf_rn(t, r.h, 1.f / 362880.f);
    t = __fmaf_rn(t, r.h, 1.f / 40320.f);
    t = __fmaf_rn(t, r.h, 1.f / 5040.f);
    t = __fmaf_rn(t, r.h, 1.f / 720.f);
    Df s = r * t + df_const(1.0 / 120.0);
    s = s * r + df_const(1.0 / 24.0);
    s = s * r + df_const(1.0 / 6.0);
    s = s * r + Df{0.5f, 0.f};
    s = s * r + Df{1.f, 0.f};
    return s * r + Df{1.f, 0.f};
}

// 1 / (1 + e^-a), rounded once: in double-float (within 2^-40) unless that is too near the middle of two floats to
// tell, one in some 30,000
__device__ __forceinline__ float sigmoid(float a)
{
    if (fabsf(a) <= 60.f) {
        int k;
        Df e = df_exp(-a, k);
        const float sc = __int_as_float((127 + k) << 23);  // |k| <= 87
        e = Df{1.f, 0.f} + Df{__fmul_rn(e.h, sc), __fmul_rn(e.l, sc)};
        const float q = __frcp_rn(e.h);
        const Df r = Df{1.f, 0.f} - e * q;  // 1 / e = q + q r + ...
        const Df s = df_quick(q, __fmul_rn(q, r.h));
        if (rounds_to_high(s, __fmul_rn(s.h, 0x1p-40f))) return s.h;
    }
    return (float)(1.0 / (1.0 + exp(-(double)a)));
}

constexpr double kPi = 3.14159265358979323846;
__host__ __device__ constexpr double csqrt_(double x)
{
    double r = x > 1 ? x : 1;
    for (int i = 0; i < 60; ++i) r = 0.5 * (r + x / r);
    return r;
}

// Degree-3 real SH basis at the unit direction (x, y, z), times the three colours' coefficients (DC at a[8 + c], AC at
// a[11 + 15 c]), plus 0.5, cut off below at 0.  False where a sum is too near the middle of two floats to be rounded, or
// not finite: colour_f64.  The direction is within 41 2^-48, the basis functions are within 2^-41, a sum is within 2^-40
// times 0.5 and its coefficients' magnitudes: one Gaussian in some 4,000.
__device__ __forceinline__ bool sh_colour(Df x, Df y, Df z, const float *a, float col[3])
{
    constexpr Df c0 = df_const(0.5 / csqrt_(kPi)), c1 = df_const(csqrt_(3.0 / (4.0 * kPi)));
    constexpr Df c2a = df_const(0.5 * csqrt_(15.0 / kPi)), c2b = df_const(0.25 * csqrt_(5.0 / kPi)),
                 c2c = df_const(0.25 * csqrt_(15.0 / kPi));
    constexpr Df c3a = df_const(0.25 * csqrt_(35.0 / (2.0 * kPi))), c3b = df_const(0.5 * csqrt_(105.0 / kPi)),
                 c3c = df_const(0.25 * csqrt_(21.0 / (2.0 * kPi))), c3d = df_const(0.25 * csqrt_(7.0 / kPi)),
                 c3e = df_const(0.25 * csqrt_(105.0 / kPi));
    const Df xx = x * x, yy = y * y, zz = z * z, xy = x * y;
    const Df dm = xx - yy, dz = zz * 4.f - xx - yy;
    Df sum[3];
    float mag[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        sum[c] = c0 * a[8 + c] + Df{0.5f, 0.f};
        mag[c] = 0.5f + fabsf(a[8 + c]);
    }
    auto add = [&](int k, Df Y) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float v = a[11 + 15 * c + (k - 1)], p = __fmul_rn(Y.h, v);
            const Df s = df_sum(sum[c].h, p);
            sum[c] = df_quick(s.h, __fadd_rn(__fadd_rn(s.l, sum[c].l), __fmaf_rn(Y.l, v, __fmaf_rn(Y.h, v, -p))));
            mag[c] += fabsf(v);
        }
    };
    add(1, -(c1 * y));
    add(2, c1 * z);
    add(3, -(c1 * x));
    add(4, c2a * xy);
    add(5, -(c2a * (y * z)));
    add(6, c2b * (zz * 2.f - xx - yy));
    add(7, -(c2a * (x * z)));
    add(8, c2c * dm);
    add(9, -(c3a * (y * (xx * 3.f - yy))));
    add(10, c3b * (xy * z));
    add(11, -(c3c * (y * dz)));
    add(12, c3d * (z * (zz * 2.f - (xx + yy) * 3.f)));
    add(13, -(c3c * (x * dz)));
    add(14, c3e * (z * dm));
    add(15, -(c3a * (x * (xx - yy * 3.f))));
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        ok = ok && rounds_to_high(sum[c], __fmul_rn(mag[c], 0x1p-40f));
        col[c] = sum[c].h > 0.f ? sum[c].h : 0.f;
    }
    return ok;
}

// the same in FP64, from the Gaussian's position
__device__ __noinline__ void colour_f64(const float *p, const float *a, double cam0, double cam1, double cam2,
                                        float col[3])
{
    const double d[3] = {(double)p[0] - cam0, (double)p[1] - cam1, (double)p[2] - cam2};
    const double dn = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]), id = dn > 0.0 ? 1.0 / dn : 1.0;
    const double x = d[0] * id, y = d[1] * id, z = d[2] * id;
    const double c0 = 0.5 / sqrt(kPi), c1 = sqrt(3.0 / (4.0 * kPi)), c2a = 0.5 * sqrt(15.0 / kPi),
                 c2b = 0.25 * sqrt(5.0 / kPi), c2c = 0.25 * sqrt(15.0 / kPi), c3a = 0.25 * sqrt(35.0 / (2.0 * kPi)),
                 c3b = 0.5 * sqrt(105.0 / kPi), c3c = 0.25 * sqrt(21.0 / (2.0 * kPi)), c3d = 0.25 * sqrt(7.0 / kPi),
                 c3e = 0.25 * sqrt(105.0 / kPi);
    const double Y[16] = {c0, -c1 * y, c1 * z, -c1 * x, c2a * x * y, -c2a * y * z, c2b * (2.0 * z * z - x * x - y * y),
                          -c2a * x * z, c2c * (x * x - y * y), -c3a * y * (3.0 * x * x - y * y), c3b * x * y * z,
                          -c3c * y * (4.0 * z * z - x * x - y * y), c3d * z * (2.0 * z * z - 3.0 * x * x - 3.0 * y * y),
                          -c3c * x * (4.0 * z * z - x * x - y * y), c3e * z * (x * x - y * y),
                          -c3a * x * (x * x - 3.0 * y * y)};
    for (int c = 0; c < 3; ++c) {
        double v = Y[0] * (double)a[8 + c];
#pragma unroll
        for (int k = 1; k < 16; ++k) v += Y[k] * (double)a[11 + 15 * c + (k - 1)];
        v += 0.5;
        col[c] = v > 0.0 ? (float)v : 0.f;
    }
}

// (p - camera) / |p - camera|, the camera's position as a sum of three floats;
// zero when they coincide
__device__ __forceinline__ void view_direction(const float *p, const RenderCam &cam, Df dir[3])
{
    Df d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
        d[c] = (Df{p[c], 0.f} - Df{cam.campos3[c][0], cam.campos3[c][1]}) - Df{cam.campos3[c][2], 0.f};
    const Df d2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    if (!(d2.h > 1e-24f && d2.h < 1e24f)) {  // products outside the range of floats
        double e[3];
        for (int c = 0; c < 3; ++c) e[c] = (double)p[c] - cam.campos[c];
        const double e2 = e[0] * e[0] + e[1] * e[1] + e[2] * e[2], ie = e2 > 0.0 ? rsqrt(e2) : 1.0;
        for (int c = 0; c < 3; ++c) dir[c] = df_of(e[c] * ie);
        return;
    }
    // r (1 + e / 2 + 3 e^2 / 8) with e = 1 - d2 r^2, r within a few units in the last place
    const float r = rsqrtf(d2.h), r2 = __fmul_rn(r, r);
    const Df t = d2 * df_quick(r2, __fmaf_rn(r, r, -r2));
    const float e = __fsub_rn(__fsub_rn(1.f, t.h), t.l);
    const Df id = df_quick(r, __fmul_rn(__fmul_rn(r, e), __fmaf_rn(0.375f, e, 0.5f)));
#pragma unroll
    for (int c = 0; c < 3; ++c) dir[c] = d[c] * id;
}

__global__ void __launch_bounds__(256) preprocess_kernel(const float *pos,
                                                         const float *attr, uint64_t n, RenderCam cam,
                                                         Splat *sp, uint32_t *depth, uint32_t *idx,
                                                         ushort4 *rect, uint32_t *count)
{
    if (after_previous()) return;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        count[i] = 0;
        depth[i] = 0xFFFFFFFFu;
        idx[i] = (uint32_t)i;
        const float *p = pos + 3 * i, *a = attr + 56 * i;
        double pc[3];
        for (int r = 0; r < 3; ++r)
            pc[r] = cam.R[3 * r] * (double)p[0] + cam.R[3 * r + 1] * (double)p[1] + cam.R[3 * r + 2] * (double)p[2] +
                    cam.t[r];
        const double z = pc[2];
        if (!(z > cam.znear)) continue;
        // rotation of the normalised quaternion: I - (2 / |q|^2) (...)
        double qw = a[3], qx = a[4], qy = a[5], qz = a[6];
        double q2 = qw * qw + qx * qx + qy * qy + qz * qz;
        if (!(q2 > 0.0)) {
            qw = q2 = 1.0;
            qx = qy = qz = 0.0;
        }
        const double s2 = 2.0 / q2;
        const double sx = s2 * qx, sy = s2 * qy, sz = s2 * qz;
        const double xx = sx * qx, yy = sy * qy, zz = sz * qz, xy = sx * qy, xz = sx * qz, yz = sy * qz, wx = sx * qw,
                     wy = sy * qw, wz = sz * qw;
        const double Rq[9] = {1 - (yy + zz), xy - wz, xz + wy, xy + wz, 1 - (xx + zz), yz - wx, xz - wy, yz + wx,
                              1 - (xx + yy)};
        const double v2[3] = {exp(2.0 * a[0]), exp(2.0 * a[1]), exp(2.0 * a[2])};  // squared scales
        // 2-D covariance N diag(v2) N^T, N = J W Rq
        const double iz = 1.0 / z, jx = cam.fx * iz, jy = cam.fy * iz;
        const double ux = jx * pc[0], vy = jy * pc[1], jxz = -ux * iz, jyz = -vy * iz;
        double N0[3], N1[3], T0[3], T1[3];
        for (int c = 0; c < 3; ++c) {
            T0[c] = jx * cam.R[c] + jxz * cam.R[6 + c];
            T1[c] = jy * cam.R[3 + c] + jyz * cam.R[6 + c];
        }
        for (int c = 0; c < 3; ++c) {
            N0[c] = T0[0] * Rq[c] + T0[1] * Rq[3 + c] + T0[2] * Rq[6 + c];
            N1[c] = T1[0] * Rq[c] + T1[1] * Rq[3 + c] + T1[2] * Rq[6 + c];
        }
        double ca = 0.3, cb = 0.0, cc = 0.3;
        for (int c = 0; c < 3; ++c) {
            const double w0 = v2[c] * N0[c], w1 = v2[c] * N1[c];
            ca += w0 * N0[c];
            cb += w0 * N1[c];
            cc += w1 * N1[c];
        }
        const double det = ca * cc - cb * cb;
        if (!(det > 0.0)) continue;
        // conic Q = [[cc, -cb], [-cb, ca]] / det; Q = L^T L with L = [[l1, l2], [0, l3]]
        const double l3 = rsqrt(cc), g = l3 * rsqrt(det);
        const double l1 = cc * g, l2 = -cb * g;
        // footprint radius ceil(3 sqrt(largest eigenvalue)): in FP32 unless that is too near an integer to tell
        const float caf = (float)ca, ccf = (float)cc, cbf = (float)cb, half = 0.5f * (caf - ccf);
        const float r3 = 3.f * sqrtf(0.5f * (caf + ccf) + sqrtf(fmaxf(half * half + cbf * cbf, 0.1f)));
        double rad = ceil((double)r3);
        if (!(fabsf(r3 - rintf(r3)) > 4e-6f * r3 + 1e-6f)) {
            const double mid = 0.5 * (ca + cc), disc = mid * mid - det;
            rad = ceil(3.0 * sqrt(mid + sqrt(disc > 0.1 ? disc : 0.1)));
        }
        const double u = ux + cam.cx, v = vy + cam.cy;
        const float opacity = sigmoid(a[7]);
        // Past |d_x| = sqrt(c cov_xx) the exponent d^T conic d is above c whatever d_y is, so with
        // c = 2 ln(255 opacity) alpha stays below 1/255 there and the splat changes no pixel; likewise in y.  The
        // margins cover the FP32 rounding of the per-pixel exponent, whose relative error grows with
        // cov_xx cov_yy / det (1e-7 sqrt(of it)): very elongated footprints keep the square of radius rad alone.
        double rx = rad, ry = rad;
        float reach_x = INFINITY, reach_y = INFINITY;
        if (ca * cc < 1e8 * det && opacity >= 0.f) {  // a NaN opacity draws 0.99 wherever its tiles lie
            if (opacity * 255.f < 0.9999f) continue;
            const float c = 2.04f * fmaxf(logf(opacity * 255.f), 0.f) + 0.1f;
            reach_x = sqrtf(c * caf) * 1.0001f;
            reach_y = sqrtf(c * ccf) * 1.0001f;
            rx = fmin(rad, (double)reach_x);
            ry = fmin(rad, (double)reach_y);
        }
        static_assert(kTile == 16, "tile of a pixel coordinate by a shift");
        int tx0 = __double2int_rd(u - rx) >> 4, tx1 = __double2int_rd(u + rx) >> 4;
        int ty0 = __double2int_rd(v - ry) >> 4, ty1 = __double2int_rd(v + ry) >> 4;
        tx0 = max(tx0, 0);
        ty0 = max(ty0, 0);
        tx1 = min(tx1, cam.TX - 1);
        ty1 = min(ty1, cam.TY - 1);
        if (tx0 > tx1 || ty0 > ty1) continue;
        Splat s;
        s.u = (float)u;
        s.ulo = (float)(u - (double)s.u);
        s.v = (float)v;
        s.vlo = (float)(v - (double)s.v);
        s.l1 = (float)l1;
        s.l2 = (float)l2;
        s.l3 = (float)l3;
        s.opacity = opacity;
        Df dir[3];
        view_direction(p, cam, dir);
        float col[3];
        if (!sh_colour(dir[0], dir[1], dir[2], a, col)) colour_f64(p, a, cam.campos[0], cam.campos[1], cam.campos[2], col);
        s.r = col[0];
        s.g = col[1];
        s.b = col[2];
        s.reach = upper_half(ceilf(reach_x) + 1.f) << 16 | upper_half(ceilf(reach_y) + 1.f);
        sp[i] = s;
        depth[i] = __float_as_uint((float)z);  // positive: integer order = float order
        rect[i] = make_ushort4((unsigned short)tx0, (unsigned short)tx1, (unsigned short)ty0, (unsigned short)ty1);
        count[i] = (uint32_t)((tx1 - tx0 + 1) * (ty1 - ty0 + 1));
    }
}

__global__ void gather_counts_kernel(const uint32_t *order, const uint32_t *count, uint64_t n, uint32_t *out)
{
    if (after_previous()) return;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
        out[i] = count[order[i]];
}

// The tile lists, in depth order: a warp writes the tiles of 32 consecutive
// Gaussians, whose entries are contiguous, one entry per lane (a thread per
// Gaussian would scatter its stores over the others' ranges).
__global__ void __launch_bounds__(256) emit_kernel(uint64_t n, const uint32_t *order, const ushort4 *rect,
                                                   const uint64_t *offs, int TX, uint32_t *tiles, uint32_t *vals)
{
    if (after_previous()) return;
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t w = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); w * 32 < n; w += warps) {
        const uint64_t k = w * 32 + lane, last = w * 32 + 32 < n ? w * 32 + 32 : n;
        const uint64_t base = offs[w * 32], total = offs[last] - base;
        if (total == 0) continue;
        const uint32_t i = k < n ? order[k] : 0u;
        const uint64_t off = (k < n ? offs[k] : offs[n]) - base;
        const ushort4 r = k < n ? rect[i] : make_ushort4(0, 0, 0, 0);
        const uint32_t xs = r.x | ((uint32_t)r.y << 16), y0 = r.z;
        for (uint64_t e0 = 0; e0 < total; e0 += 32) {
            const uint64_t e = e0 + lane;
            uint32_t g = 0;  // the last Gaussian that starts at or before entry e
#pragma unroll
            for (uint32_t st = 16; st; st >>= 1) {
                const uint64_t o = __shfl_sync(0xFFFFFFFFu, off, g + st);  // g + st < 32
                if (o <= e) g += st;
            }
            const uint32_t rel = (uint32_t)(e - __shfl_sync(0xFFFFFFFFu, off, g));
            const uint32_t gxs = __shfl_sync(0xFFFFFFFFu, xs, g), gy = __shfl_sync(0xFFFFFFFFu, y0, g);
            const uint32_t gi = __shfl_sync(0xFFFFFFFFu, i, g);
            const uint32_t x0 = gxs & 0xFFFFu, width = (gxs >> 16) - x0 + 1u, row = rel / width;
            if (e < total) {
                tiles[base + e] = (gy + row) * (uint32_t)TX + x0 + (rel - row * width);
                vals[base + e] = gi;
            }
        }
    }
}

// Entries [x, y) of the sorted list per tile, by binary search: a thread per
// tile and some twenty-five dependent loads, against a pass over the whole list
// (1M Gaussians at 960 x 540: 85 -> 17 us).
__global__ void ranges_kernel(const uint32_t *tiles, uint64_t total, uint32_t ntiles, uint2 *ranges)
{
    if (after_previous()) return;
    const uint32_t tile = blockIdx.x * blockDim.x + threadIdx.x;
    if (tile >= ntiles) return;
    auto first = [&](uint32_t key) {  // the first entry with a tile of at least key
        uint64_t lo = 0, hi = total;
        while (lo < hi) {
            const uint64_t mid = (lo + hi) >> 1;
            if (tiles[mid] < key) lo = mid + 1; else hi = mid;
        }
        return (uint32_t)lo;
    };
    ranges[tile] = make_uint2(first(tile), first(tile + 1));
}

__device__ __forceinline__ void copy16(void *smem, const void *gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}

// A warp per 8 x 4 pixels, a pixel per lane, each on its own: of its tile's
// list it takes 32 splats at a time, a splat per lane, finds which of them reach
// its pixels (Splat::reach) and copies those, in order and without gaps, to its
// own shared memory while the 32 before are composited.  Most of a tile's list
// does not reach a given block, and what is skipped would have failed the alpha
// cut at every pixel, so the image is the same.  Bound by instruction issue, some
// 30 a splat.  1M Gaussians at 960 x 540: 806 us with a CTA per tile that
// staged batches of 256 splats for its eight warps (a barrier per batch, so
// that all waited for the slowest, and half the issue slots empty) -> 547 us.
constexpr int kWarpsPerCta = 4;  // the blocks of half a tile

__global__ void __launch_bounds__(32 * kWarpsPerCta) render_kernel(const uint2 *ranges, const uint32_t *vals,
                                                                   const Splat *sp, RenderCam cam, float *image)
{
    if (after_previous()) return;
    static_assert(sizeof(Splat) == 48 && kTile == 16, "copied in 16-byte words; two halves of 16 x 8 pixels");
    __shared__ __align__(16) Splat batch[kWarpsPerCta][2][32];
    const int tx = blockIdx.x, ty = blockIdx.y >> 1;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5, ltmask = lanemask_lt();
    const int bx = tx * kTile + (int)(w & 1) * 8, by = (int)blockIdx.y * (kTile / 2) + (int)(w >> 1) * 4;
    const int px = bx + (int)(lane & 7), py = by + (int)(lane >> 3);
    const float mx = bx + 4.f, my = by + 2.f;  // the block's centre
    const bool inside = px < cam.W && py < cam.H;
    const uint2 rg = ranges[ty * cam.TX + tx];
    const uint32_t *list = vals + rg.x;
    const uint32_t n = rg.y - rg.x;
    const float fxp = px + 0.5f, fyp = py + 0.5f;
    float T = 1.f, col[3] = {0.f, 0.f, 0.f};
    bool done = !inside;
    // entry g + lane of the list (g a multiple of 32), and the first 16 bytes of its splat
    auto val_at = [&](uint32_t g) { return g < n && lane < n - g ? list[g + lane] : 0u; };
    auto head_at = [&](uint32_t g, uint32_t val) {
        return g < n && lane < n - g ? *reinterpret_cast<const uint4 *>(sp + val) : make_uint4(0u, 0u, 0u, 0u);
    };
    auto stage = [&](uint32_t g, uint32_t val, uint4 head, Splat *to) {  // returns how many reach the block
        const bool hit = g < n && lane < n - g &&
                         fabsf(__uint_as_float(head.x) - mx) <= __uint_as_float(head.z & 0xFFFF0000u) + 4.f &&
                         fabsf(__uint_as_float(head.y) - my) <= __uint_as_float(head.z << 16) + 2.f;
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, hit);
        if (hit) {
            char *d = reinterpret_cast<char *>(to + __popc(m & ltmask));
            const char *q = reinterpret_cast<const char *>(sp + val);
            *reinterpret_cast<uint4 *>(d) = head;
            copy16(d + 16, q + 16);
            copy16(d + 32, q + 32);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        return (uint32_t)__popc(m);
    };
    uint32_t v1 = val_at(0), v2 = val_at(32);
    uint4 h1 = head_at(0, v1);
    uint32_t cnt = stage(0, v1, h1, batch[w][0]);
    v1 = v2;
    h1 = head_at(32, v1);
    v2 = val_at(64);
    for (uint32_t g = 0, k = 0; g < n; g += 32, k ^= 1u) {
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncwarp();  // this group has landed for every lane, and all have left the one before
        if (__all_sync(0xFFFFFFFFu, done)) break;
        const uint32_t next = stage(g + 32, v1, h1, batch[w][k ^ 1u]);
        v1 = v2;
        h1 = head_at(g + 64, v1);
        v2 = val_at(g + 96);
        const Splat *B = batch[w][k];
#pragma unroll 2
        for (uint32_t j = 0; j < cnt; ++j) {
            const Splat s = B[j];
            const float dx = (s.u - fxp) + s.ulo, dy = (s.v - fyp) + s.vlo;
            const float e0 = fmaf(s.l1, dx, s.l2 * dy), e1 = s.l3 * dy;
            const float power = -0.5f * fmaf(e0, e0, e1 * e1);
            const float alpha = fminf(0.99f, s.opacity * expf(power));
            const float tn = T * (1.f - alpha);
            const bool on = !done && !(alpha < 1.f / 255.f), stop = tn < 1e-4f;
            if (on && !stop) {
                col[0] += s.r * alpha * T;
                col[1] += s.g * alpha * T;
                col[2] += s.b * alpha * T;
                T = tn;
            }
            done = done || (on && stop);
        }
        cnt = next;
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (inside)
        for (int c = 0; c < 3; ++c) image[((uint64_t)py * cam.W + px) * 3 + c] = col[c] + T * cam.bg[c];
}

uint32_t rgrid(uint64_t n, int num_sms)
{
    uint64_t b = (n + 255) / 256;
    const uint64_t cap = (uint64_t)num_sms * 8;
    return (uint32_t)(b < 1 ? 1 : (b < cap ? b : cap));
}

}  // namespace

size_t render_splat_bytes() { return sizeof(Splat); }

void launch_render_prepare(const float *pos, const float *attr, uint64_t n, const RenderCam &cam,
                           const RenderBuffers &b, const uint32_t **order, int num_sms, cudaStream_t s)
{
    launch_after(preprocess_kernel, rgrid(n, num_sms), 256, 0, s, pos, attr, n, cam, (Splat *)b.splats, b.depth, b.idx, b.rect,
                                                        b.count);
    count_launch();
    // Depth first, over the Gaussians; then only the tile bits over the many times longer list of their tiles.
    // Sorting that list by (tile, depth) at once took six passes of 12-byte pairs, 3.3 ms of 6.6 with the emission at
    // 1M Gaussians and 960 x 540 (24M entries); the whole call was 4.6 ms this way.
    const bool alt = radix_sort(b.depth, b.idx, b.depth_alt, b.idx_alt, b.hist, n, 32u, num_sms, s);
    *order = alt ? b.idx_alt : b.idx;
    launch_after(gather_counts_kernel, rgrid(n, num_sms), 256, 0, s, *order, b.count, n, b.count_sorted);
    count_launch();
    launch_scan_u32_to_u64(b.count_sorted, n, b.offs, b.partials, num_sms, s);
}

void launch_render_tiles(uint64_t n, const RenderBuffers &b, const uint32_t *order, uint64_t total,
                         const RenderCam &cam, uint32_t *tiles, uint32_t *vals, uint32_t *tiles_alt,
                         uint32_t *vals_alt, uint32_t *hist, uint2 *ranges, float *image, int num_sms, cudaStream_t s)
{
    const uint32_t ntiles = (uint32_t)(cam.TX * cam.TY);
    const uint32_t *sv = vals;
    if (total) {
        launch_after(emit_kernel, rgrid(n, num_sms), 256, 0, s, n, order, b.rect, b.offs, cam.TX, tiles, vals);
        count_launch();
        uint32_t tb = 0;
        while ((1u << tb) < ntiles) ++tb;
        const bool alt = radix_sort(tiles, vals, tiles_alt, vals_alt, hist, total, tb, num_sms, s);
        if (alt) sv = vals_alt;
        launch_after(ranges_kernel, (ntiles + 63) / 64, 64, 0, s, alt ? tiles_alt : tiles, total, ntiles, ranges);
        count_launch();
    } else {
        dev_memset(ranges, 0, sizeof(uint2) * ntiles, s);
    }
    launch_after(render_kernel, dim3(cam.TX, 2 * cam.TY), 32 * kWarpsPerCta, 0, s, ranges, sv, (const Splat *)b.splats, cam, image);
    count_launch();
}

}  // namespace gsnfs
