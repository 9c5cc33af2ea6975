// mxe_fast64.cuh -- FP64 arithmetic for a GPU whose FP64 pipe is the bound.
//
// GB300 retires 2 FP64 operations per clock and SM: a warp holds one SM
// sub-partition's FP64 pipe for 64 clocks per instruction (measured: 64.4
// clocks alone, 76 with all four sub-partitions busy), whatever its active
// lanes, while 32 FP32 or integer instructions beside it cost nothing.  Every
// FP64-pipe operation that can be spared counts, comparisons, conversions and
// the iterations inside a division or a transcendental included:
//   * reciprocal and reciprocal square root: an FP32 seed of the mantissa,
//     scaled by exponent arithmetic on the integer pipe, and one cubically
//     convergent Newton-type step (Householder's method of order 2): 3 and 5
//     FP64 operations;
//   * exp2 and log2: table-driven (P. T. P. Tang, ACM TOMS 15, 1989 and 16,
//     1990), 64 entries, Taylor remainders on |f| <= 2^-7: 7 and 9 operations;
//   * comparisons, clamps, signs and float <-> double conversions of seeds by
//     integer operations.
// Accurate for every normal argument to about one unit in the last place (measured over 2^21
// arguments each: reciprocal, roots and their reciprocals 1.05, exp2 1.27, log2 1.17, the
// latter in units of 1 below 1); arguments outside that range (zero, subnormal, infinite,
// NaN, negative where undefined) take the CUDA functions.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace mxe {
namespace f64 {

// ---------------------------------------------------------------- bits
__device__ __forceinline__ unsigned hi32(double x) { return (unsigned)__double2hiint(x); }
__device__ __forceinline__ unsigned lo32(double x) { return (unsigned)__double2loint(x); }
// x < 0 (false for -0, subnormal and NaN-free reading of the sign otherwise)
__device__ __forceinline__ bool is_neg(double x) { return hi32(x) > 0x80000000u; }
__device__ __forceinline__ double sel(bool c, double a, double b) { return c ? a : b; }
__device__ __forceinline__ double abs_(double x) {
    return __hiloint2double((int)(hi32(x) & 0x7fffffffu), (int)lo32(x));
}
// order-preserving integer image of a non-NaN double
__device__ __forceinline__ long long key(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ (long long)((unsigned long long)(b >> 63) >> 1);
}
__device__ __forceinline__ bool lt(double a, double b) { return key(a) < key(b); }
__device__ __forceinline__ bool is_nan(double x) {
    return (unsigned long long)(__double_as_longlong(x) & 0x7fffffffffffffffll) >
           0x7ff0000000000000ull;
}
__device__ __forceinline__ bool is_finite(double x) { return (hi32(x) & 0x7ff00000u) != 0x7ff00000u; }
// x >= 0 and x <= 0 without the FP64 pipe (false for NaN, as the comparisons)
__device__ __forceinline__ bool ge0(double x) {
    return hi32(x) <= 0x7ff00000u || __double_as_longlong(x) == (long long)0x8000000000000000ull;
}
__device__ __forceinline__ bool le0(double x) {
    const long long b = __double_as_longlong(x);
    return b <= 0 && (unsigned)(b >> 32) <= 0xfff00000u ? true : b == 0;
}
__device__ __forceinline__ double max_(double a, double b) { return sel(lt(a, b), b, a); }
// a FP32 value (normal, or zero mapped to zero) as double bits
__device__ __forceinline__ double widen(float f) {
    const unsigned b = __float_as_uint(f), em = b & 0x7fffffffu;
    const unsigned hi = em ? (b & 0x80000000u) | ((em >> 3) + (896u << 20)) : 0u;
    return __hiloint2double((int)hi, (int)(em << 29));
}
// the nearest float towards zero of a double whose magnitude lies in FP32's
// normal range; smaller magnitudes give 0, larger ones the largest float
__device__ __forceinline__ float narrow(double x) {
    const unsigned h = hi32(x), e = (h >> 20) & 0x7ffu;
    const unsigned m = ((h & 0xfffffu) << 3) | (lo32(x) >> 29);
    unsigned f = ((e - 896u) << 23) | m;
    if (e <= 896u) f = 0u;
    if (e >= 1151u) f = 0x7f7fffffu;
    return __uint_as_float((h & 0x80000000u) | f);
}

// (float)x, rounded to nearest, by integer operations in FP32's normal range
__device__ __forceinline__ float to_f32(double x) {
    const unsigned e = (hi32(x) >> 20) & 0x7ffu;
    if (e - 898u > 250u) return (float)x;
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return narrow(__longlong_as_double((long long)(b + 0x0fffffffull + ((b >> 29) & 1ull))));
}

// ---------------------------------------------------------------- 1/x, 1/sqrt(x)
__device__ __forceinline__ float rcp32(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt32(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

static __device__ __noinline__ double rcp_slow(double x) { return 1.0 / x; }
static __device__ __noinline__ double rsqrt_slow(double x) { return 1.0 / ::sqrt(x); }

// 1/x: seed r0 = 2^-e / m with the FP32 reciprocal of the mantissa m in
// [1, 2) (|1 - x r0| < 2^-21), then r0 (1 + d + d^2), d = 1 - x r0: the
// truncated geometric series leaves d^3 < 2^-63.
__device__ __forceinline__ double rcp(double x) {
    const unsigned h = hi32(x), e = (h >> 20) & 0x7ffu;
    const unsigned m = 0x3f800000u | ((h & 0xfffffu) << 3) | (lo32(x) >> 29);
    const unsigned f = __float_as_uint(rcp32(__uint_as_float(m)));
    const unsigned rh = ((h & 0x80000000u) | (f >> 3)) + ((1919u - e) << 20);
    const double r0 = __hiloint2double((int)rh, (int)(f << 29));
    const double d = ::fma(-x, r0, 1.0);
    double r = ::fma(r0, ::fma(d, d, d), r0);
    if (e - 1u > 2043u) r = rcp_slow(x);            // zero, subnormal, huge, inf, NaN
    return r;
}

// a/b with one residual correction of a * rcp(b) (rb = rcp(b)): within a unit in the last
// place, the rounded quotient in almost all cases.  Rounding it always costs four operations
// more on the chain of a recovery (61 x 47 cells: 457 -> 490 us for three steps) and
// changed no run's error against a 64-bit evaluation.
__device__ __forceinline__ double div_by(double a, double b, double rb) {
    const double q = a * rb;
    const double v = ::fma(::fma(-b, q, a), rb, q);
    return is_finite(q) && is_finite(v) ? v : a / b;
}

// y0 = 2^(-e/2) / sqrt(m), m in [1, 4); with h = 1 - x y0^2 (|h| < 2^-20) the
// series 1/sqrt(1 - h) = 1 + h/2 + 3h^2/8 + ... is cut after the square term.
// t = x y0 is kept: sqrt(x) = t (1 + h/2 + 3h^2/8).
__device__ __forceinline__ bool rsqrt_parts(double x, double& y0, double& t, double& p) {
    const unsigned h = hi32(x), e = (h >> 20);       // sign bit makes e > 2046
    const unsigned odd = (e + 1u) & 1u;              // exponent e - 1023 odd
    const unsigned m = ((127u + odd) << 23) | ((h & 0xfffffu) << 3) | (lo32(x) >> 29);
    const unsigned f = __float_as_uint(rsqrt32(__uint_as_float(m)));
    const int half = ((int)e - 1023 - (int)odd) >> 1;
    y0 = __hiloint2double((int)((f >> 3) + ((unsigned)(896 - half) << 20)), (int)(f << 29));
    t = x * y0;
    const double r = ::fma(-t, y0, 1.0);
    p = ::fma(0.375, r, 0.5) * r;
    return e - 1u <= 2045u;                          // positive normal
}
__device__ __forceinline__ double rsqrt(double x) {
    double y0, t, p;
    const bool ok = rsqrt_parts(x, y0, t, p);
    double y = ::fma(y0, p, y0);
    if (!ok) y = rsqrt_slow(x);
    return y;
}
__device__ __forceinline__ double sqrt_(double x) {
    double y0, t, p;
    const bool ok = rsqrt_parts(x, y0, t, p);
    double s = ::fma(t, p, t);
    if (!ok) s = ::sqrt(x);
    return s;
}
// sqrt(x) and 1/sqrt(x) together
__device__ __forceinline__ void sqrt_rsqrt(double x, double& s, double& y) {
    double y0, t, p;
    const bool ok = rsqrt_parts(x, y0, t, p);
    s = ::fma(t, p, t);
    y = ::fma(y0, p, y0);
    if (!ok) {
        s = ::sqrt(x);
        y = 1.0 / s;
    }
}

// ---------------------------------------------------------------- exp2, log2
// 2^(j/64)
static __device__ const double EXP2_TAB[64] = {
    0x1.0000000000000p+0, 0x1.02c9a3e778061p+0, 0x1.059b0d3158574p+0, 0x1.0874518759bc8p+0,
    0x1.0b5586cf9890fp+0, 0x1.0e3ec32d3d1a2p+0, 0x1.11301d0125b51p+0, 0x1.1429aaea92de0p+0,
    0x1.172b83c7d517bp+0, 0x1.1a35beb6fcb75p+0, 0x1.1d4873168b9aap+0, 0x1.2063b88628cd6p+0,
    0x1.2387a6e756238p+0, 0x1.26b4565e27cddp+0, 0x1.29e9df51fdee1p+0, 0x1.2d285a6e4030bp+0,
    0x1.306fe0a31b715p+0, 0x1.33c08b26416ffp+0, 0x1.371a7373aa9cbp+0, 0x1.3a7db34e59ff7p+0,
    0x1.3dea64c123422p+0, 0x1.4160a21f72e2ap+0, 0x1.44e086061892dp+0, 0x1.486a2b5c13cd0p+0,
    0x1.4bfdad5362a27p+0, 0x1.4f9b2769d2ca7p+0, 0x1.5342b569d4f82p+0, 0x1.56f4736b527dap+0,
    0x1.5ab07dd485429p+0, 0x1.5e76f15ad2148p+0, 0x1.6247eb03a5585p+0, 0x1.6623882552225p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6dfb23c651a2fp+0, 0x1.71f75e8ec5f74p+0, 0x1.75feb564267c9p+0,
    0x1.7a11473eb0187p+0, 0x1.7e2f336cf4e62p+0, 0x1.82589994cce13p+0, 0x1.868d99b4492edp+0,
    0x1.8ace5422aa0dbp+0, 0x1.8f1ae99157736p+0, 0x1.93737b0cdc5e5p+0, 0x1.97d829fde4e50p+0,
    0x1.9c49182a3f090p+0, 0x1.a0c667b5de565p+0, 0x1.a5503b23e255dp+0, 0x1.a9e6b5579fdbfp+0,
    0x1.ae89f995ad3adp+0, 0x1.b33a2b84f15fbp+0, 0x1.b7f76f2fb5e47p+0, 0x1.bcc1e904bc1d2p+0,
    0x1.c199bdd85529cp+0, 0x1.c67f12e57d14bp+0, 0x1.cb720dcef9069p+0, 0x1.d072d4a07897cp+0,
    0x1.d5818dcfba487p+0, 0x1.da9e603db3285p+0, 0x1.dfc97337b9b5fp+0, 0x1.e502ee78b3ff6p+0,
    0x1.ea4afa2a490dap+0, 0x1.efa1bee615a27p+0, 0x1.f50765b6e4540p+0, 0x1.fa7c1819e90d8p+0};
// per mantissa interval j of [1, 2): c ~ 1/midpoint (12 bits), -log2(c)
static __device__ const double2 LOG2_TAB[64] = {
    0x1.fc00000000000p-1, 0x1.72c7ba20f7327p-7, 0x1.f440000000000p-1, 0x1.1263289517ae7p-5,
    0x1.ecc0000000000p-1, 0x1.c4eb3635cea06p-5, 0x1.e580000000000p-1, 0x1.3a0cf56a06c4bp-4,
    0x1.de60000000000p-1, 0x1.916a59b80a235p-4, 0x1.d780000000000p-1, 0x1.e6f50c2d9f754p-4,
    0x1.d0c0000000000p-1, 0x1.1e153cd5de584p-3, 0x1.ca40000000000p-1, 0x1.47b2c2f8cb155p-3,
    0x1.c400000000000p-1, 0x1.7046031c79f85p-3, 0x1.bde0000000000p-1, 0x1.9895d0a732f96p-3,
    0x1.b7e0000000000p-1, 0x1.c09d64546b554p-3, 0x1.b200000000000p-1, 0x1.e857d3d361368p-3,
    0x1.ac60000000000p-1, 0x1.0771a9766e3bcp-2, 0x1.a6e0000000000p-1, 0x1.1a88d1009acc9p-2,
    0x1.a160000000000p-1, 0x1.2ddff3bc5e4aep-2, 0x1.9c20000000000p-1, 0x1.409347a934e48p-2,
    0x1.9700000000000p-1, 0x1.530fd08f29fa7p-2, 0x1.9200000000000p-1, 0x1.6552b49986277p-2,
    0x1.8d40000000000p-1, 0x1.76e2065019d0ap-2, 0x1.8860000000000p-1, 0x1.891fe20affb86p-2,
    0x1.83c0000000000p-1, 0x1.9aa4354228033p-2, 0x1.7f40000000000p-1, 0x1.abe2f8ec9671ep-2,
    0x1.7ae0000000000p-1, 0x1.bcd915bcb6fb2p-2, 0x1.7680000000000p-1, 0x1.ce01a12f5d8d1p-2,
    0x1.7240000000000p-1, 0x1.dede169c35d77p-2, 0x1.6e20000000000p-1, 0x1.ef6b3d344485ap-2,
    0x1.6a20000000000p-1, 0x1.ffa5d49cee602p-2, 0x1.6620000000000p-1, 0x1.080748d542b72p-1,
    0x1.6240000000000p-1, 0x1.1010826b187a9p-1, 0x1.5e80000000000p-1, 0x1.17ece9555fd72p-1,
    0x1.5ac0000000000p-1, 0x1.1fdef5db3a511p-1, 0x1.5720000000000p-1, 0x1.27a23a05a872cp-1,
    0x1.53a0000000000p-1, 0x1.2f34fd35e682ap-1, 0x1.5020000000000p-1, 0x1.36dbd5d549ffep-1,
    0x1.4ca0000000000p-1, 0x1.3e972f86d05edp-1, 0x1.4960000000000p-1, 0x1.45d7e475de565p-1,
    0x1.4600000000000p-1, 0x1.4d7380dcc422dp-1, 0x1.42e0000000000p-1, 0x1.5490e8d62733cp-1,
    0x1.3fc0000000000p-1, 0x1.5bc007cc076f2p-1, 0x1.3ca0000000000p-1, 0x1.630136d308a22p-1,
    0x1.39a0000000000p-1, 0x1.6a096fbcd380ep-1, 0x1.36a0000000000p-1, 0x1.7122f642b3601p-1,
    0x1.33a0000000000p-1, 0x1.784e205f4c276p-1, 0x1.30e0000000000p-1, 0x1.7ef026ac0a2e7p-1,
    0x1.2e00000000000p-1, 0x1.85efd062c656dp-1, 0x1.2b40000000000p-1, 0x1.8cb19c5f05fa8p-1,
    0x1.2880000000000p-1, 0x1.938360a10a160p-1, 0x1.25e0000000000p-1, 0x1.9a14f63cdc2e7p-1,
    0x1.2340000000000p-1, 0x1.a0b5a267b28d6p-1, 0x1.20c0000000000p-1, 0x1.a713ca57071afp-1,
    0x1.1e20000000000p-1, 0x1.add2b706984f0p-1, 0x1.1bc0000000000p-1, 0x1.b3fae09ea5173p-1,
    0x1.1940000000000p-1, 0x1.ba844ffcd610ep-1, 0x1.16e0000000000p-1, 0x1.c0c7e947528b3p-1,
    0x1.1480000000000p-1, 0x1.c71939b5d8856p-1, 0x1.1240000000000p-1, 0x1.cd2248a6c7354p-1,
    0x1.0fe0000000000p-1, 0x1.d38efdd9e36cap-1, 0x1.0dc0000000000p-1, 0x1.d95acc02d690ap-1,
    0x1.0b80000000000p-1, 0x1.df8aae0e46f56p-1, 0x1.0960000000000p-1, 0x1.e56ed99fb4bd2p-1,
    0x1.0740000000000p-1, 0x1.eb5f254ba8bf0p-1, 0x1.0520000000000p-1, 0x1.f15bc3637397cp-1,
    0x1.0300000000000p-1, 0x1.f764e7742b428p-1, 0x1.0100000000000p-1, 0x1.fd1ec77250aa7p-1};

static __device__ __noinline__ double exp2_slow(double x) { return ::exp2(x); }
static __device__ __noinline__ double log2_slow(double x) { return ::log2(x); }

// 2^x = 2^k T_j 2^f with n = 64 k + j = rint(64 x) (formed in FP32: any
// integer within 0.51 of 64 x serves) and f = x - n/64, |f| < 2^-6.9:
// 2^f - 1 by its Taylor series to f^5 (remainder < 2^-54)
__device__ __forceinline__ double exp2_(double x) {
    const float xf = narrow(x);
    const int n = __float2int_rn(xf * 64.0f);
    const double f = x - widen((float)n * 0.015625f);
    const double T = EXP2_TAB[n & 63];
    double p = 0x1.5d87fe78a6731p-10;
    p = ::fma(p, f, 0x1.3b2ab6fba4e77p-7);
    p = ::fma(p, f, 0x1.c6b08d704a0c0p-5);
    p = ::fma(p, f, 0x1.ebfbdff82c58fp-3);
    p = ::fma(p, f, 0x1.62e42fefa39efp-1);
    const double r = ::fma(T, f * p, T);
    const double v = __hiloint2double((int)(hi32(r) + ((unsigned)(n >> 6) << 20)), (int)lo32(r));
    return fabsf(xf) < 1000.0f ? v : exp2_slow(x);
}

// log2(x) = e - log2(c) + log2(1 + r), r = m c - 1, |r| <= 2^-7: Taylor
// series to r^7 (remainder < 2^-57, absolute)
__device__ __forceinline__ double log2_(double x) {
    const unsigned h = hi32(x), e = h >> 20;
    const double m = __hiloint2double((int)((h & 0xfffffu) | 0x3ff00000u), (int)lo32(x));
    const double2 cl = LOG2_TAB[(h >> 14) & 63u];
    const double r = ::fma(m, cl.x, -1.0);
    double p = 0x1.a61762a7aded9p-3;
    p = ::fma(p, r, -0x1.ec709dc3a03fdp-3);
    p = ::fma(p, r, 0x1.2776c50ef9bfep-2);
    p = ::fma(p, r, -0x1.71547652b82fep-2);
    p = ::fma(p, r, 0x1.ec709dc3a03fdp-2);
    p = ::fma(p, r, -0x1.71547652b82fep-1);
    p = ::fma(p, r, 0x1.71547652b82fep+0);
    const double v = ::fma(p, r, widen((float)((int)e - 1023)) + cl.y);
    return e - 1u <= 2045u ? v : log2_slow(x);       // positive normal
}

// min(max(s, lo), 1), NaN kept (the clamp of sigma, Appendix A)
__device__ __forceinline__ double clamp_sigma(double s, double lo) {
    const long long b = __double_as_longlong(s);
    const long long one = 0x3ff0000000000000ll;
    long long r = b < __double_as_longlong(lo) ? __double_as_longlong(lo) : b;   // also s < 0
    r = r > one ? one : r;
    return is_nan(s) ? s : __longlong_as_double(r);
}

}  // namespace f64
}  // namespace mxe
