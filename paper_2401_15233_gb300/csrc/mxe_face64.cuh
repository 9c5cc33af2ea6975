// mxe_face64.cuh -- FP64 face states: conserved state, flux and wave speeds
// of the 5-moment, the general 14-moment and the planar 14-moment system
// (Sec. 2.3, 2.4 closures, Sec. 5 / Appendix B wave speeds), arranged for the
// fewest FP64-pipe operations (see mxe_fast64.cuh for why that is the
// measure).  The formulas are those of mxe_physics.cuh / mxe_planar.cuh:
//   * one reciprocal per denominator, shared by all its quotients; 1/sigma
//     and sqrt(sigma) from one reciprocal square root;
//   * sigma and the wave-speed bracket choose numerator and denominator of
//     their rationalised form first and divide once: at most one of
//     zeta+ = q + al, zeta- = -q + al (al >= 0) is negative;
//   * B = 2 T2 P + 4 P^3 enters as B/4;
//   * the wave-speed fit in base 2: P^1.1 exp(-P^2) = 2^(1.1 l - P^2 log2 e),
//     l = log2 P; Y = (sqrt B - E)^2 and 10 - 16 r + 6 r^2 =
//     2 (5 - 3 r)(1 - r), r = sqrt(sigma), which cannot round below zero.
#pragma once
#include "mxe_fast64.cuh"
#include "mxe_planar.cuh"

namespace mxe {
namespace f64 {

constexpr double LOG2E = 0x1.71547652b82fep+0;

// raw sigma = [A + sqrt(A^2 + X)] / T4, T4 = 4 T2; X / (T4 (sqrt - A)) for A < 0
__device__ __forceinline__ double sigma_raw(double A, double X, double T4) {
    const double s = sqrt_(::fma(A, A, X)) + abs_(A);
    const bool neg = is_neg(A);
    return sel(neg, X, s) * rcp(sel(neg, T4 * s, T4));
}

// zeta + sqrt(D), D = zeta^2 + D0, given s = sqrt(D) + |zeta| and, for
// zeta < 0, the quotient q = D0 / s; zeta alone where D <= 0
struct Bracket {
    double D0, s;
    bool none, neg;
};
__device__ __forceinline__ Bracket bracket(double z, double D0) {
    Bracket b;
    const double D = ::fma(z, z, D0);
    b.D0 = D0;
    b.none = __double_as_longlong(D) <= 0 && !is_nan(D);
    b.neg = is_neg(z);
    b.s = sqrt_(b.none ? 1.0 : D) + abs_(z);
    return b;
}

// sigma_bar with its roots
struct SigRoots {
    double sb, ssb, isb;         // sigma, sqrt(sigma), 1/sigma
};
__device__ __forceinline__ SigRoots sig_roots(double sig, double slim) {
    SigRoots g;
    double y;
    g.sb = clamp_sigma(sig, slim);
    sqrt_rsqrt(g.sb, g.ssb, y);
    g.isb = y * y;
    return g;
}

// magnitudes of lambda*_max (lp) and -lambda*_min (lm) from the bracket
// arguments zp, zm, pre = (a sigma + b) / (2 sigma), E and base
__device__ __forceinline__ void two_speeds(double zp, double zm, double sbE, double base,
                                           double pre, double E, double& lp, double& lm) {
    const Bracket P = bracket(zp, ::fma(-zp, sbE, base)), N = bracket(zm, ::fma(-zm, sbE, base));
    double q = 0.0;
    if (P.neg || N.neg) q = sel(P.neg, P.D0, N.D0) * rcp(sel(P.neg, P.s, N.s));
    const double hp = P.none ? zp : sel(P.neg, q, P.s), hm = N.none ? zm : sel(N.neg, q, N.s);
    lp = ::fma(pre, hp, E);
    lm = ::fma(pre, hm, E);
}

// E = 0.8 sqrt((3 - 3 sigma) P) and sqrt(B) - E
__device__ __forceinline__ void speed_terms(const SigRoots& g, double three_P, double& E,
                                            double& dd) {
    E = 0.8 * sqrt_(::fma(-g.sb, three_P, three_P));
    const double R = sqrt_(::fma(-6.0, g.ssb, 10.0) * (1.0 - g.ssb));
    dd = sqrt_(::fma(-4.0, g.ssb, 5.0) + R) - E;
}

// Eq. (14mom-approx-ws-equations) for P*_kk, q*_k and q*_perp = qp, qp2 = qp^2
__device__ __forceinline__ void lam(double Pkk, double qd, double qp, double qp2,
                                    const SigRoots& g, double& lp, double& lm) {
    const double l = log2_(Pkk);
    const double a = exp2_(::fma(1.1, l, -LOG2E * (Pkk * Pkk)));
    const double b = exp2_((-0.5 * LOG2E) * exp2_(1.4 * l));
    const double pre = ::fma(0.45 * Pkk * b, g.isb, 0.7 * a);
    double E, dd;
    speed_terms(g, 3.0 * Pkk, E, dd);
    const double al = qp * ::fma(Pkk, ::fma(0.6, Pkk, -0.38), 0.35);
    const double sd = g.sb * dd;
    two_speeds(qd + al, al - qd, g.sb * E, ::fma(4.0 * sd, sd, 0.1 * qp2), pre, E, lp, lm);
}

// =========================================================================
// planar 14-moment state (ten fields)
// =========================================================================
struct DimP {
    double tr, p, th, sq;        // tr P, p, theta, sqrt(theta)
    double a, b, d, f, bb;       // P* = [[a b 0][b d 0][0 0 f]], b^2
    double qx, qy, t, T2, yx, yy;
    SigRoots g;
};
__device__ __forceinline__ void dimless(const double* Q, double slim, DimP& g) {
    const double rho = Q[0];
    g.tr = Q[3] + Q[5] + Q[6];
    g.p = g.tr * (1.0 / 3.0);
    const double ip = rcp(g.p);
    g.th = g.p * rcp(rho);
    double rsq;
    sqrt_rsqrt(g.th, g.sq, rsq);
    const double isc3 = ip * rsq;                    // 1 / (rho theta^{3/2})
    g.a = Q[3] * ip; g.b = Q[4] * ip; g.d = Q[5] * ip; g.f = Q[6] * ip;
    g.qx = Q[7] * isc3; g.qy = Q[8] * isc3;
    const double Rs = Q[9] * rho * ip * ip;
    g.t = g.a + g.d + g.f;
    g.bb = g.b * g.b;
    g.T2 = ::fma(g.a, g.a, ::fma(g.d, g.d, ::fma(g.f, g.f, g.bb + g.bb)));
    const double i2 = rcp(::fma(g.a, g.d, -g.bb));
    g.yx = ::fma(g.d, g.qx, -g.b * g.qy) * i2;
    g.yy = ::fma(g.a, g.qy, -g.b * g.qx) * i2;
    const double T4 = 4.0 * g.T2;
    const double A = ::fma(g.t, g.t, ::fma(2.0, g.T2, -Rs));
    const double X = (T4 + T4) * ::fma(g.qx, g.yx, g.qy * g.yy);
    g.g = sig_roots(sigma_raw(A, X, T4), slim);
}

template <int K>
__device__ __forceinline__ void speeds(const double* Q, const DimP& g, double kw, double& lo,
                                       double& hi) {
    const double qo = K == 0 ? g.qy : g.qx;
    double lp, lm;
    lam(K == 0 ? g.a : g.d, K == 0 ? g.qx : g.qy, abs_(qo), qo * qo, g.g, lp, lm);
    const double ks = kw * g.sq;
    hi = ::fma(lp, ks, Q[1 + K]);
    lo = ::fma(-lm, ks, Q[1 + K]);
}

// conserved state and K-flux (closure_p, prim2cons_p, flux_p in fused form)
template <int K>
__device__ __forceinline__ void state_flux(const double* Q, const DimP& g, double* U, double* F) {
    const double a = g.a, b = g.b, d = g.d, f = g.f, t = g.t, T2 = g.T2;
    const double sb = g.g.sb, ssb = g.g.ssb, isb = g.g.isb;
    const double P2xx = ::fma(a, a, g.bb), P2xy = b * (a + d), P2yy = ::fma(d, d, g.bb);
    const double P2zz = f * f;
    const double P3xx = ::fma(P2xx, a, P2xy * b), P3xy = ::fma(P2xx, b, P2xy * d);
    const double P3yy = ::fma(P2xy, b, P2yy * d);
    const double trP3 = ::fma(P2zz, f, P3xx + P3yy);
    // v = B^-1 q*, B/4 = (T2/2) P* + P*^3 (in-plane block)
    const double h2 = 0.5 * T2;
    const double Bxx = ::fma(h2, a, P3xx), Bxy = ::fma(h2, b, P3xy), Byy = ::fma(h2, d, P3yy);
    const double iB = 0.25 * rcp(::fma(Bxx, Byy, -Bxy * Bxy));
    const double vx = ::fma(Byy, g.qx, -Bxy * g.qy) * iB;
    const double vy = ::fma(Bxx, g.qy, -Bxy * g.qx) * iB;
    const double wx = ::fma(a, vx, b * vy), wy = ::fma(b, vx, d * vy);
    const double wK = K == 0 ? wx : wy, wO = K == 0 ? wy : wx;
    const double vK = K == 0 ? vx : vy, vO = K == 0 ? vy : vx;
    const double yK = K == 0 ? g.yx : g.yy, yO = K == 0 ? g.yy : g.yx;
    const double P2KK = K == 0 ? P2xx : P2yy, P2OO = K == 0 ? P2yy : P2xx;
    const double P3KK = K == 0 ? P3xx : P3yy;
    const double PKK = K == 0 ? a : d;
    const double w2K = wK + wK, w2O = wO + wO;
    double QK[4];
    QK[0] = 3.0 * w2K * P2KK;
    QK[1] = ::fma(w2K + w2K, P2xy, w2O * P2KK);
    QK[2] = ::fma(w2K, P2OO, (w2O + w2O) * P2xy);
    QK[3] = w2K * P2zz;
    const double omsb2 = ::fma(-2.0, sb, 2.0);
    const double t1 = ::fma(QK[0], yK, QK[1] * yO), t2 = ::fma(QK[1], yK, QK[2] * yO);
    double RKK = ::fma(t1, isb, ::fma(omsb2, P2KK, PKK * t));
    double ROK = ::fma(t2, isb, ::fma(omsb2, P2xy, b * t));
    const double yQy = ::fma(yK, t1, yO * t2);
    // row K of the W bracket against v
    const double tt = t * t;
    const double c1 = ::fma(t + t, tt - T2, 12.0 * trP3), c2 = ::fma(14.0, T2, -6.0 * tt);
    const double c3 = 20.0 * t;
    const double P4KK = ::fma(P2KK, P2KK, P2xy * P2xy), P4KO = P2xy * (P2xx + P2yy);
    const double mKK = ::fma(c1, PKK, ::fma(c2, P2KK, ::fma(c3, P3KK, 20.0 * P4KK)));
    const double mKO = ::fma(c1, b, ::fma(c2, P2xy, ::fma(c3, P3xy, 20.0 * P4KO)));
    const double Wq = ::fma(mKK, vK, mKO * vO);
    const double qs = K == 0 ? g.qx : g.qy;
    const double Ss = ::fma(yQy * isb, isb, ::fma(ssb + ssb, t * qs, (1.0 - ssb) * Wq));
    const double sc3 = g.p * g.sq, sc4 = g.p * g.th;
    QK[0] *= sc3; QK[1] *= sc3; QK[2] *= sc3; QK[3] *= sc3;
    RKK *= sc4; ROK *= sc4;
    const double SK = Ss * (sc4 * g.sq);
    // conserved state
    const double rho = Q[0], ux = Q[1], uy = Q[2], Pxx = Q[3], Pxy = Q[4], Pyy = Q[5];
    const double u2 = ::fma(ux, ux, uy * uy);
    const double Pux = ::fma(Pxx, ux, Pxy * uy), Puy = ::fma(Pxy, ux, Pyy * uy);
    const double uPuq = ::fma(ux, Pux + Q[7], uy * (Puy + Q[8]));
    const double ru2 = rho * u2, e = ru2 + g.tr;
    U[0] = rho;
    U[1] = rho * ux; U[2] = rho * uy;
    U[3] = ::fma(U[1], ux, Pxx); U[4] = ::fma(U[1], uy, Pxy); U[5] = ::fma(U[2], uy, Pyy);
    U[6] = Q[6];
    U[7] = ::fma(ux, e, ::fma(2.0, Pux, Q[7]));
    U[8] = ::fma(uy, e, ::fma(2.0, Puy, Q[8]));
    U[9] = ::fma(u2, ::fma(2.0, g.tr, ru2), ::fma(4.0, uPuq, Q[9]));
    // flux u_K U + central part
    const double uK = K == 0 ? ux : uy, uO = K == 0 ? uy : ux;
    const double PxK = K == 0 ? Pxx : Pxy, PyK = K == 0 ? Pxy : Pyy;
    const double qK = Q[7 + K], PuK = K == 0 ? Pux : Puy;
    const double QuK = ::fma(QK[0], uK, QK[1] * uO), QuO = ::fma(QK[1], uK, QK[2] * uO);
    const double gK = ::fma(2.0, PuK, qK);
    F[0] = U[1 + K];
    F[1] = ::fma(uK, U[1], PxK);
    F[2] = ::fma(uK, U[2], PyK);
    F[3] = ::fma(uK, U[3], ::fma(ux + ux, PxK, K == 0 ? QK[0] : QK[2]));
    F[4] = ::fma(uK, U[4], ::fma(ux, PyK, ::fma(uy, PxK, QK[1])));
    F[5] = ::fma(uK, U[5], ::fma(uy + uy, PyK, K == 0 ? QK[2] : QK[0]));
    F[6] = ::fma(uK, U[6], QK[3]);
    F[7] = ::fma(uK, U[7], ::fma(ux, gK, ::fma(u2, PxK, ::fma(2.0, K == 0 ? QuK : QuO,
                                                              K == 0 ? RKK : ROK))));
    F[8] = ::fma(uK, U[8], ::fma(uy, gK, ::fma(u2, PyK, ::fma(2.0, K == 0 ? QuO : QuK,
                                                              K == 0 ? ROK : RKK))));
    const double uQR = ::fma(uK, QuK + RKK, uO * (QuO + ROK));
    F[9] = ::fma(uK, U[9], ::fma(u2 + u2, gK, ::fma(4.0, uQR, SK)));
}

template <int K>
__device__ __forceinline__ void face_p(const double* Q, double slim, double kw, double* U,
                                       double* F, double& lo, double& hi) {
    DimP g;
    dimless(Q, slim, g);
    state_flux<K>(Q, g, U, F);
    speeds<K>(Q, g, kw, lo, hi);
}

// CFL rates max(|lambda_min|, |lambda_max|) in x and y
__device__ __forceinline__ double abs_max_bits(double a, double b) {   // NaN in b alone is dropped,
    const double x = abs_(a), y = abs_(b);                             // as in x > y ? x : y
    return sel(lt(y, x) || is_nan(x), x, y);
}
__device__ __forceinline__ void rates_p(const double* Q, double slim, double kw, double& ax,
                                        double& ay) {
    DimP g;
    dimless(Q, slim, g);
    double lo, hi;
    speeds<0>(Q, g, kw, lo, hi);
    ax = abs_max_bits(lo, hi);
    speeds<1>(Q, g, kw, lo, hi);
    ay = abs_max_bits(lo, hi);
}
__device__ __forceinline__ double rate_x_p(const double* Q, double slim, double kw) {
    DimP g;
    dimless(Q, slim, g);
    double lo, hi;
    speeds<0>(Q, g, kw, lo, hi);
    return abs_max_bits(lo, hi);
}

// =========================================================================
// general 14-moment state
// =========================================================================
struct Dim14 {
    double p, th, sq, P[6], q[3], t, T2, y[3];
    SigRoots g;
};
// cofactors of a symmetric 3 x 3 matrix (xx, xy, xz, yy, yz, zz); returns det
__device__ __forceinline__ double cofactors(const double* A, double* c) {
    c[0] = ::fma(A[3], A[5], -A[4] * A[4]);
    c[1] = ::fma(A[2], A[4], -A[1] * A[5]);
    c[2] = ::fma(A[1], A[4], -A[2] * A[3]);
    c[3] = ::fma(A[0], A[5], -A[2] * A[2]);
    c[4] = ::fma(A[1], A[2], -A[0] * A[4]);
    c[5] = ::fma(A[0], A[3], -A[1] * A[1]);
    return ::fma(A[0], c[0], ::fma(A[1], c[1], A[2] * c[2]));
}
__device__ __forceinline__ double dot3(double a0, double a1, double a2, const double* v) {
    return ::fma(a0, v[0], ::fma(a1, v[1], a2 * v[2]));
}
__device__ __forceinline__ void symv(const double* A, const double* v, double* o) {
    o[0] = dot3(A[0], A[1], A[2], v);
    o[1] = dot3(A[1], A[3], A[4], v);
    o[2] = dot3(A[2], A[4], A[5], v);
}

__device__ __forceinline__ void dimless(const double* Q, double slim, Dim14& g) {
    const double rho = Q[0];
    g.p = (Q[4] + Q[7] + Q[9]) * (1.0 / 3.0);
    const double ip = rcp(g.p);
    g.th = g.p * rcp(rho);
    double rsq;
    sqrt_rsqrt(g.th, g.sq, rsq);
    const double isc3 = ip * rsq;
#pragma unroll
    for (int n = 0; n < 6; ++n) g.P[n] = Q[4 + n] * ip;
#pragma unroll
    for (int n = 0; n < 3; ++n) g.q[n] = Q[10 + n] * isc3;
    const double Rs = Q[13] * rho * ip * ip;
    const double* P = g.P;
    g.t = P[0] + P[3] + P[5];
    const double off = ::fma(P[1], P[1], ::fma(P[2], P[2], P[4] * P[4]));
    g.T2 = ::fma(P[0], P[0], ::fma(P[3], P[3], ::fma(P[5], P[5], off + off)));
    double c[6];
    const double id = rcp(cofactors(P, c));
    symv(c, g.q, g.y);
#pragma unroll
    for (int n = 0; n < 3; ++n) g.y[n] *= id;
    const double T4 = 4.0 * g.T2;
    const double A = ::fma(g.t, g.t, ::fma(2.0, g.T2, -Rs));
    const double X = (T4 + T4) * dot3(g.q[0], g.q[1], g.q[2], g.y);
    g.g = sig_roots(sigma_raw(A, X, T4), slim);
}

template <int K>
__device__ __forceinline__ void speeds(const double* Q, const Dim14& g, double kw, double& lo,
                                       double& hi) {
    constexpr int E1 = (K + 1) % 3, E2 = (K + 2) % 3;
    const double qp2 = ::fma(g.q[E1], g.q[E1], g.q[E2] * g.q[E2]);
    double lp, lm;
    lam(g.P[sidx(K, K)], g.q[K], sqrt_(qp2), qp2, g.g, lp, lm);
    const double ks = kw * g.sq;
    hi = ::fma(lp, ks, Q[1 + K]);
    lo = ::fma(-lm, ks, Q[1 + K]);
}

// closing slice along K (closure14_slice)
template <int K>
__device__ __forceinline__ void closure(const Dim14& g, double* Qk, double* Rk, double& Sk) {
    const double* P = g.P;
    const double sb = g.g.sb, ssb = g.g.ssb, isb = g.g.isb, t = g.t, T2 = g.T2;
    double P2[6], P3[6], B[6], c[6], v[3], w[3];
    sym_mul(P, P, P2);
    sym_mul(P2, P, P3);
    const double trP3 = P3[0] + P3[3] + P3[5];
    const double h2 = 0.5 * T2;
#pragma unroll
    for (int n = 0; n < 6; ++n) B[n] = ::fma(h2, P[n], P3[n]);      // B / 4
    const double iB = 0.25 * rcp(cofactors(B, c));
    symv(c, g.q, v);
#pragma unroll
    for (int n = 0; n < 3; ++n) v[n] *= iB;
    symv(P, v, w);
#pragma unroll
    for (int n = 0; n < 3; ++n) w[n] += w[n];
    double Qs[6], T[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = a; b < 3; ++b) {
            if (a == K && b == K) Qs[sidx(a, b)] = 3.0 * w[K] * P2[sidx(K, K)];
            else if (a == K || b == K) {
                const int o = a == K ? b : a;
                Qs[sidx(a, b)] = ::fma(w[K] + w[K], P2[sidx(K, o)], w[o] * P2[sidx(K, K)]);
            } else
                Qs[sidx(a, b)] = ::fma(w[K], P2[sidx(a, b)],
                                       ::fma(w[a], P2[sidx(K, b)], w[b] * P2[sidx(K, a)]));
        }
    symv(Qs, g.y, T);
    const double omsb2 = ::fma(-2.0, sb, 2.0);
    const double sc3 = g.p * g.sq, sc4 = g.p * g.th;
#pragma unroll
    for (int a = 0; a < 3; ++a)
        Rk[a] = sc4 * ::fma(T[a], isb, ::fma(omsb2, P2[sidx(a, K)], P[sidx(a, K)] * t));
    const double yQy = dot3(g.y[0], g.y[1], g.y[2], T);
    const double tt = t * t;
    const double c1 = ::fma(t + t, tt - T2, 12.0 * trP3), c2 = ::fma(14.0, T2, -6.0 * tt);
    const double c3 = 20.0 * t;
    double Wq = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double P4 = ::fma(P2[sidx(K, 0)], P2[sidx(0, a)],
                                ::fma(P2[sidx(K, 1)], P2[sidx(1, a)],
                                      P2[sidx(K, 2)] * P2[sidx(2, a)]));
        const double m = ::fma(c1, P[sidx(K, a)], ::fma(c2, P2[sidx(K, a)],
                               ::fma(c3, P3[sidx(K, a)], 20.0 * P4)));
        Wq = a == 0 ? m * v[a] : ::fma(m, v[a], Wq);
    }
    Sk = (sc4 * g.sq) * ::fma(yQy * isb, isb, ::fma(ssb + ssb, t * g.q[K], (1.0 - ssb) * Wq));
#pragma unroll
    for (int n = 0; n < 6; ++n) Qk[n] = Qs[n] * sc3;
}

template <int K>
__device__ __forceinline__ void face_14(const double* Q, double slim, double kw, double* U,
                                        double* F, double& lo, double& hi) {
    Dim14 g;
    dimless(Q, slim, g);
    double Qk[6], Rk[3], Sk;
    closure<K>(g, Qk, Rk, Sk);
    prim2cons14(Q, U);
    flux14<double, K>(Q, U, Qk, Rk, Sk, F);
    speeds<K>(Q, g, kw, lo, hi);
}
__device__ __forceinline__ void rates_14(const double* Q, double slim, double kw, double& ax,
                                         double& ay) {
    Dim14 g;
    dimless(Q, slim, g);
    double lo, hi;
    speeds<0>(Q, g, kw, lo, hi);
    ax = abs_max_bits(lo, hi);
    speeds<1>(Q, g, kw, lo, hi);
    ay = abs_max_bits(lo, hi);
}
__device__ __forceinline__ double rate_x_14(const double* Q, double slim, double kw) {
    Dim14 g;
    dimless(Q, slim, g);
    double lo, hi;
    speeds<0>(Q, g, kw, lo, hi);
    return abs_max_bits(lo, hi);
}

// =========================================================================
// 5-moment system
// =========================================================================
struct Dim5 {
    double th, sq, qs;
    SigRoots g;
};
__device__ __forceinline__ void dimless(const double* Q, double slim, Dim5& g) {
    const double rho = Q[0], P = Q[2];
    const double ip = rcp(P);
    g.th = P * rcp(rho);
    double rsq;
    sqrt_rsqrt(g.th, g.sq, rsq);
    g.qs = Q[3] * (ip * rsq);
    const double A = ::fma(-Q[4] * rho, ip * ip, 3.0);
    g.g = sig_roots(sigma_raw(A, 8.0 * g.qs * g.qs, 4.0), slim);
}
// Baradaran's fit, Eq. (ws-max-baradaran-orig)
__device__ __forceinline__ void speeds(const double* Q, const Dim5& g, double kw, double& lo,
                                       double& hi) {
    double E, dd, lp, lm;
    speed_terms(g.g, 3.0, E, dd);
    const double sd = g.g.sb * dd;
    two_speeds(g.qs, -g.qs, g.g.sb * E, 4.0 * sd * sd, 0.5 * g.g.isb, E, lp, lm);
    const double ks = kw * g.sq;
    hi = ::fma(lp, ks, Q[1]);
    lo = ::fma(-lm, ks, Q[1]);
}
__device__ __forceinline__ void face_5(const double* Q, double slim, double kw, double* U,
                                       double* F, double& lo, double& hi) {
    Dim5 g;
    dimless(Q, slim, g);
    const double rho = Q[0], u = Q[1], P = Q[2], q = Q[3], r = Q[4], qs = g.qs;
    const double c = qs * g.g.isb;
    const double ss = qs * ::fma(c, c, ::fma(-8.0, g.g.ssb, 10.0));
    const double s = ss * (P * g.th * g.sq);
    U[0] = rho;
    U[1] = rho * u;
    U[2] = ::fma(U[1], u, P);
    const double Pu = P * u, m2 = U[1] * u;           // rho u^2
    U[3] = ::fma(m2, u, ::fma(3.0, Pu, q));
    const double qu = q * u, Pu2 = Pu * u, m3 = m2 * u;
    U[4] = ::fma(m3, u, ::fma(6.0, Pu2, ::fma(4.0, qu, r)));
    F[0] = U[1]; F[1] = U[2]; F[2] = U[3]; F[3] = U[4];
    F[4] = ::fma(u, ::fma(m3, u, ::fma(10.0, Pu2, ::fma(10.0, qu, 5.0 * r))), s);
    speeds(Q, g, kw, lo, hi);
}
__device__ __forceinline__ double rate_5(const double* Q, double slim, double kw) {
    Dim5 g;
    dimless(Q, slim, g);
    double lo, hi;
    speeds(Q, g, kw, lo, hi);
    return abs_max_bits(lo, hi);
}

// =========================================================================
// BGK source and relaxation rate
// =========================================================================
// 1/tau = rho sqrt(theta) k, k = 1 / (tau_ref rho_ref sqrt(T_ref)) (hard
// spheres), or k = 1 / tau_ref: the cell-independent factor
__device__ __forceinline__ double tau_factor(int model, double tau_ref, double rho_ref,
                                             double T_ref) {
    if (model == 0) return 0.0;
    return model == 1 ? 1.0 / tau_ref : 1.0 / (tau_ref * rho_ref * ::sqrt(T_ref));
}
// sqrt(rho p) = rho sqrt(theta)
__device__ __forceinline__ double inv_tau(int model, double k, double rho, double p) {
    return model == 1 ? k : k * sqrt_(rho * p);
}

__device__ __forceinline__ void source_5(const double* Q, double it, double* C) {
    const double P = Q[2];
    C[0] = C[1] = C[2] = 0.0;
    C[3] = -Q[3] * it;
    C[4] = it * ::fma(3.0 * P, P * rcp(Q[0]), -::fma(4.0 * Q[1], Q[3], Q[4]));
}
__device__ __forceinline__ void source_p(const double* Q, double p, double it, double* C) {
    const double ux = Q[1], uy = Q[2], Pxy = Q[4];
    const double dx = p - Q[3], dy = p - Q[5];
    C[0] = C[1] = C[2] = 0.0;
    C[3] = dx * it; C[4] = -Pxy * it; C[5] = dy * it; C[6] = (p - Q[6]) * it;
    // (P - p I) u, the parts of 2 P u - 2 p u and u.P.u - |u|^2 p
    const double ax = ::fma(dx, ux, -Pxy * uy), ay = ::fma(dy, uy, -Pxy * ux);
    C[7] = it * ::fma(2.0, ax, -Q[7]);
    C[8] = it * ::fma(2.0, ay, -Q[8]);
    const double v = ::fma(ux, ax - Q[7], uy * (ay - Q[8]));
    C[9] = it * ::fma(4.0, v, ::fma(15.0 * p, p * rcp(Q[0]), -Q[9]));
}
__device__ __forceinline__ void source_14(const double* Q, double p, double it, double* C) {
    const double* u = Q + 1;
    const double D[6] = {p - Q[4], -Q[5], -Q[6], p - Q[7], -Q[8], p - Q[9]};
    double a[3];
    symv(D, u, a);
    C[0] = C[1] = C[2] = C[3] = 0.0;
#pragma unroll
    for (int n = 0; n < 6; ++n) C[4 + n] = D[n] * it;
#pragma unroll
    for (int n = 0; n < 3; ++n) C[10 + n] = it * ::fma(2.0, a[n], -Q[10 + n]);
    const double v = ::fma(u[0], a[0] - Q[10], ::fma(u[1], a[1] - Q[11], u[2] * (a[2] - Q[12])));
    C[13] = it * ::fma(4.0, v, ::fma(15.0 * p, p * rcp(Q[0]), -Q[13]));
}

// =========================================================================
// shared limiter (Sec. 3.2) and reconstruction
// =========================================================================
// phi = min_k phi_k over the fields that are not flat.  The
// fields that cannot set phi are ruled out in FP32: r_k = min / max of
// |dm|, |dp| (their common exponent removed first, so that no magnitude is out
// of range) orders the fields as phi_k does, and a field clearly inside or
// outside its flat tolerance is decided there too.  FP64 then evaluates only
// the fields within 2^-18 of the smallest ratio (usually one) and those whose
// flat test is close: 2 NF differences and about 12 operations a candidate
// instead of about 17 a field.
struct PhiScreen {
    float r;               // ratio, 0 for opposite signs
    float mx;              // max(|dm|, |dp|) in FP32
    bool exact0;           // phi_k (not flat) is 0 for certain
};
__device__ __forceinline__ PhiScreen phi_screen(double dm, double dp) {
    PhiScreen o;
    const unsigned hm = hi32(dm) & 0x7fffffffu, hp = hi32(dp) & 0x7fffffffu;
    const unsigned hx = hm > hp ? hm : hp, hn = hm > hp ? hp : hm;
    const unsigned lx = hm > hp ? lo32(dm) : lo32(dp), ln = hm > hp ? lo32(dp) : lo32(dm);
    const unsigned ex = hx >> 20, en = hn >> 20;
    const float fx = __uint_as_float(0x3f800000u | ((hx & 0xfffffu) << 3) | (lx >> 29));
    const unsigned sh = ex - en;                         // the smaller one relative to it
    const float fn = sh > 100u ? 0.0f
        : __uint_as_float(((127u - sh) << 23) | ((hn & 0xfffffu) << 3) | (ln >> 29));
    const bool opp = ((hi32(dm) ^ hi32(dp)) >> 31) != 0u;
    const bool tiny = en == 0u || ex + en < 1060u;       // subnormal factor or product
    o.r = opp || tiny ? 0.0f : fn * rcp32(fx);
    o.exact0 = (opp && !tiny) || ((hn | ln) == 0u && ex != 0u);   // opposite, or one is zero
    o.mx = __uint_as_float(ex <= 896u ? 0u : ex >= 1151u ? 0x7f7fffffu
                           : ((ex - 896u) << 23) | ((hx & 0xfffffu) << 3) | (lx >> 29));
    return o;
}

// at(m, k): field k of the stencil cell m = -1, 0, 1; ks: the field that sets
// phi where its derivative there is not zero (else -1).
template <int NF, class At>
__device__ __forceinline__ double limiter_at(const At& at, int lim, int& ks) {
    ks = -1;
    FlatRef<double> fr;
    {
        constexpr int p1 = NF == 5 ? 2 : NF == 10 ? 3 : 4, p2 = NF == 10 ? 5 : 7,
                      p3 = NF == 10 ? 6 : 9;
        fr.rho = at(0, 0);
        fr.s = at(0, p1);
        if (NF != 5) fr.s = add_rn(add_rn(fr.s, at(0, p2)), at(0, p3));
    }
    // flat tolerances T x natural scale in FP32 (p = s or s / 3); a class whose
    // tolerance leaves FP32's range is left to the exact test (thr = -1)
    float thr[5];
    {
        const float rho = narrow(fr.rho), p = narrow(fr.s) * (NF == 5 ? 1.0f : 1.0f / 3.0f);
        const float th = p * rcp32(rho), v = th * rsqrt32(th);
        const float sc[5] = {rho, v, p, p * v, p * th};
#pragma unroll
        for (int n = 0; n < 5; ++n) {
            const float t = 1e-10f * sc[n];
            thr[n] = t > 1e-35f && t < 1e30f ? t : -1.0f;
        }
    }
    float r[NF], rc = 1.0f;
    unsigned maybe = 0u;                                 // fields not certainly flat
    bool zero = false;
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        const PhiScreen s = phi_screen(at(0, k) - at(-1, k), at(1, k) - at(0, k));
        const float t = thr[flat_class<NF>(k)];
        const bool known = t > 0.0f && s.mx < 1e37f;
        const bool flat = known && s.mx < 0.9999f * t, rough = known && s.mx > 1.0001f * t;
        r[k] = s.r;
        if (rough) {
            rc = fminf(rc, s.r);
            zero |= s.exact0;
        }
        if (!flat) maybe |= 1u << k;
    }
    if (zero) return 0.0;
    rc = rc * 1.000004f;
    unsigned cand = 0u;
#pragma unroll
    for (int k = 0; k < NF; ++k)
        if (((maybe >> k) & 1u) && r[k] <= rc) cand |= 1u << k;
    double phi = 1.0;
    while (cand) {
        const int k = __ffs((int)cand) - 1;
        cand &= cand - 1u;
        const double dm = at(0, k) - at(-1, k), dp = at(1, k) - at(0, k);
        const double pk = phi_field(dm, dp, lim);
        if (lt(pk, phi) && !field_flat_at<NF>(fr, k, max_(abs_(dm), abs_(dp)))) {
            phi = pk;
            ks = k;
        }
    }
    if (phi == 0.0) ks = -1;
    return phi;
}
// the cell c of fields fs apart, neighbours at +- stride
template <int NF>
__device__ __forceinline__ double limiter(const double* W, int c, int stride, int fs, int lim) {
    int ks;
    const double* w = W + c;
    return limiter_at<NF>([=](int m, int k) { return w[k * fs + m * stride]; }, lim, ks);
}

// MUSCL face value Q0 + sgn/2 phi (Qp - Qm)/2, h = sgn phi / 4
__device__ __forceinline__ double face_value(double qm, double q0, double qp, double h) {
    return ::fma(h, qp - qm, q0);
}

// =========================================================================
// numerical flux of a face (Sec. 3.1): HLL with Davis speeds, or Rusanov
// =========================================================================
template <int NF>
__device__ __forceinline__ void riemann(const double* UL, const double* FL, double l0, double l1,
                                        const double* UR, const double* FR, double r0, double r1,
                                        int flux, double* F) {
    if (flux == 1) {
        double s = abs_(l0), v = abs_(l1);
        s = sel(lt(s, v), v, s);
        v = abs_(r0);
        s = sel(lt(s, v), v, s);
        v = abs_(r1);
        s = 0.5 * sel(lt(s, v), v, s);
#pragma unroll
        for (int k = 0; k < NF; ++k) F[k] = ::fma(0.5, FL[k] + FR[k], -s * (UR[k] - UL[k]));
        return;
    }
    const double SL = sel(lt(l0, r0), l0, r0), SR = sel(lt(r1, l1), l1, r1);
    if (ge0(SL)) {
#pragma unroll
        for (int k = 0; k < NF; ++k) F[k] = FL[k];
    } else if (le0(SR)) {
#pragma unroll
        for (int k = 0; k < NF; ++k) F[k] = FR[k];
    } else {
        // [SR FL - SL FR + SL SR (UR - UL)] / (SR - SL)
        const double inv = rcp(SR - SL);
        const double cl = SR * inv, cr = -SL * inv, cu = SL * cl;
#pragma unroll
        for (int k = 0; k < NF; ++k)
            F[k] = ::fma(cl, FL[k], ::fma(cr, FR[k], cu * (UR[k] - UL[k])));
    }
}

// Face flux from the two states of a face held by adjacent lanes (left in the
// even lane): the lanes exchange half of their conserved states and fluxes,
// and each forms half of the fields, the even lane [0, H), the odd lane [H, NF).
template <int NF>
__device__ __forceinline__ void pair_flux(const double* U, const double* F, double lo, double hi,
                                          bool right, int flux, double* Fo) {
    constexpr int H = (NF + 1) / 2;
    const double plo = __shfl_xor_sync(0xffffffffu, lo, 1);
    const double phi = __shfl_xor_sync(0xffffffffu, hi, 1);
    double UL[H], FL[H], UR[H], FR[H];
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const int k1 = H + k < NF ? H + k : NF - 1;
        const double pu = __shfl_xor_sync(0xffffffffu, right ? U[k] : U[k1], 1);
        const double pf = __shfl_xor_sync(0xffffffffu, right ? F[k] : F[k1], 1);
        const double ou = right ? U[k1] : U[k], of = right ? F[k1] : F[k];
        UL[k] = right ? pu : ou;
        FL[k] = right ? pf : of;
        UR[k] = right ? ou : pu;
        FR[k] = right ? of : pf;
    }
    riemann<H>(UL, FL, right ? plo : lo, right ? phi : hi, UR, FR, right ? lo : plo,
                    right ? hi : phi, flux, Fo);
}

}  // namespace f64
}  // namespace mxe
