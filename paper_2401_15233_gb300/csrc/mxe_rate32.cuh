// mxe_rate32.cuh -- the CFL rate of one cell in FP32 with correctly rounded
// divisions and roots and a log2 and exp2 of full FP32 precision.
//
// The time step is cfl / max over the cells of the rate, so the rounding of
// one cell's rate goes into every step: from the FP32 primitives W and with
// approximate reciprocals, roots and exponentials it is off by about 7e-7.
// Those serve as a screen: a cell whose approximate rate may be the largest
// is evaluated again, from the primitives of its FP64 state and with the
// functions below (2.5e-7), so that the maximum is over such values whatever the
// order of the blocks.  Few cells are.  Kept out of line: rare, and long.
#pragma once
#include "mxe_planar.cuh"

namespace mxe {
namespace rn {

__device__ __forceinline__ float rcp(float x) { return __frcp_rn(x); }
__device__ __forceinline__ float div(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float sqrt_(float x) { return __fsqrt_rn(x); }
// log2 of a positive normal number: exponent + (2 / ln 2) atanh(s), s = (m - 1) /
// (m + 1), m in [3/4, 3/2), the series to s^9 (remainder below 1e-8)
__device__ __forceinline__ float log2_(float x) {
    const int b = __float_as_int(x);
    const int e = (b - 0x3f400000) >> 23;
    const float m = __int_as_float(b - (e << 23));
    const float s = div(m - 1.0f, m + 1.0f), z = s * s;
    float p = 0.32059890f;
    p = fmaf(p, z, 0.41219858f);
    p = fmaf(p, z, 0.57707802f);
    p = fmaf(p, z, 0.96179669f);
    p = fmaf(p, z, 2.88539008f);
    return fmaf(s, p, (float)e);
}
// 2^x for |x| < 100: n + f, |f| <= 1/2, Taylor series of 2^f to f^7
__device__ __forceinline__ float exp2_(float x) {
    const float n = rintf(x), f = x - n;
    float p = 1.52527338e-5f;
    p = fmaf(p, f, 1.54035304e-4f);
    p = fmaf(p, f, 1.33335581e-3f);
    p = fmaf(p, f, 9.61812911e-3f);
    p = fmaf(p, f, 5.55041087e-2f);
    p = fmaf(p, f, 2.40226507e-1f);
    p = fmaf(p, f, 6.93147181e-1f);
    p = fmaf(p, f, 1.0f);
    return fabsf(x) < 100.0f ? p * __int_as_float(((int)n + 127) << 23) : exp2f(x);
}

__device__ __forceinline__ float hyp(float z, float D0) {
    const float D = fmaf(z, z, D0), s = sqrt_(fmaxf(D, 0.0f)) + fabsf(z);
    return z >= 0.0f ? s : D > 0.0f ? div(D0, s) : z;
}
// max(|lambda_min|, |lambda_max|) along one direction (lam_core_x2's formulas)
__device__ __forceinline__ float speed(float P, float qd, float qperp, float sb, float u,
                                       float ks) {
    constexpr float LOG2E = 1.4426950408889634f;
    const float l = log2_(P), ssb = sqrt_(sb);
    const float a = exp2_(fmaf(1.1f, l, -LOG2E * (P * P)));
    const float b = exp2_((-0.5f * LOG2E) * exp2_(1.4f * l));
    const float pre = fmaf(0.7f, a, div(0.45f * P * b, sb));
    const float E = 0.8f * sqrt_(fmaf(-3.0f, sb, 3.0f) * P);
    const float B = fmaf(-4.0f, ssb, 5.0f) + sqrt_(fmaf(-6.0f, ssb, 10.0f) * (1.0f - ssb));
    const float sd = (sqrt_(B) - E) * sb;
    const float al = qperp * fmaf(P, fmaf(0.6f, P, -0.38f), 0.35f);
    const float base = fmaf(4.0f * sd, sd, 0.1f * qperp * qperp), sE = sb * E;
    const float zp = qd + al, zm = al - qd;
    const float lp = fmaf(pre, hyp(zp, fmaf(-zp, sE, base)), E);
    const float lm = fmaf(pre, hyp(zm, fmaf(-zm, sE, base)), E);
    return fmaxf(fabsf(fmaf(lp, ks, u)), fabsf(fmaf(-lm, ks, u)));
}
// sigma of A, X and tr P*^2, clamped
__device__ __forceinline__ float sigma(float A, float X, float T2, float sigma_lim) {
    const float s = sqrt_(fmaf(A, A, X)) + fabsf(A), f = 4.0f * T2;
    return clamp_sigma(A >= 0.0f ? div(s, f) : div(X, f * s), sigma_lim);
}

template <int NF>
struct Cell {
    float w[NF];
};

// rate in x times idx plus rate in y times idy
static __device__ __noinline__ float rate_p(Cell<NP> c, float sigma_lim, float k_ws, float idx,
                                            float idy) {
    const float* Q = c.w;
    const float p = (Q[3] + Q[5] + Q[6]) * (1.0f / 3.0f), ip = rcp(p);
    const float sq = sqrt_(div(p, Q[0])), isc3 = div(ip, sq);
    const float a = Q[3] * ip, b = Q[4] * ip, d = Q[5] * ip, f = Q[6] * ip;
    const float qx = Q[7] * isc3, qy = Q[8] * isc3, Rs = (Q[9] * Q[0]) * (ip * ip);
    const float t = a + d + f, T2 = fmaf(a, a, fmaf(d, d, fmaf(f, f, 2.0f * b * b)));
    const float det = fmaf(a, d, -b * b);
    const float qPq = div(fmaf(qx, fmaf(d, qx, -b * qy), qy * fmaf(a, qy, -b * qx)), det);
    const float sb = sigma(fmaf(t, t, fmaf(2.0f, T2, -Rs)), 8.0f * T2 * qPq, T2, sigma_lim);
    const float ks = k_ws * sq;
    return fmaf(speed(a, qx, fabsf(qy), sb, Q[1], ks), idx,
                speed(d, qy, fabsf(qx), sb, Q[2], ks) * idy);
}
static __device__ __noinline__ float rate_14(Cell<14> c, float sigma_lim, float k_ws, float idx,
                                             float idy) {
    const float* Q = c.w;
    const float p = (Q[4] + Q[7] + Q[9]) * (1.0f / 3.0f), ip = rcp(p);
    const float sq = sqrt_(div(p, Q[0])), isc3 = div(ip, sq);
    float P[6], q[3];
#pragma unroll
    for (int n = 0; n < 6; ++n) P[n] = Q[4 + n] * ip;
#pragma unroll
    for (int n = 0; n < 3; ++n) q[n] = Q[10 + n] * isc3;
    const float Rs = (Q[13] * Q[0]) * (ip * ip), t = P[0] + P[3] + P[5];
    const float off = fmaf(P[1], P[1], fmaf(P[2], P[2], P[4] * P[4]));
    const float T2 = fmaf(P[0], P[0], fmaf(P[3], P[3], fmaf(P[5], P[5], 2.0f * off)));
    const float c0 = fmaf(P[3], P[5], -P[4] * P[4]), c1 = fmaf(P[2], P[4], -P[1] * P[5]);
    const float c2 = fmaf(P[1], P[4], -P[2] * P[3]), c3 = fmaf(P[0], P[5], -P[2] * P[2]);
    const float c4 = fmaf(P[1], P[2], -P[0] * P[4]), c5 = fmaf(P[0], P[3], -P[1] * P[1]);
    const float det = fmaf(P[0], c0, fmaf(P[1], c1, P[2] * c2));
    const float y0 = fmaf(c0, q[0], fmaf(c1, q[1], c2 * q[2]));
    const float y1 = fmaf(c1, q[0], fmaf(c3, q[1], c4 * q[2]));
    const float y2 = fmaf(c2, q[0], fmaf(c4, q[1], c5 * q[2]));
    const float qPq = div(fmaf(q[0], y0, fmaf(q[1], y1, q[2] * y2)), det);
    const float sb = sigma(fmaf(t, t, fmaf(2.0f, T2, -Rs)), 8.0f * T2 * qPq, T2, sigma_lim);
    const float ks = k_ws * sq, z2 = q[2] * q[2];
    return fmaf(speed(P[0], q[0], sqrt_(fmaf(q[1], q[1], z2)), sb, Q[1], ks), idx,
                speed(P[3], q[1], sqrt_(fmaf(q[0], q[0], z2)), sb, Q[2], ks) * idy);
}
template <int NF>
__device__ __forceinline__ float rate(const float* Q, float sigma_lim, float k_ws, float idx,
                                      float idy) {
    Cell<NF> c;
#pragma unroll
    for (int k = 0; k < NF; ++k) c.w[k] = Q[k];
    if constexpr (NF == NP) return rate_p(c, sigma_lim, k_ws, idx, idy);
    else return rate_14(c, sigma_lim, k_ws, idx, idy);
}

}  // namespace rn
}  // namespace mxe
