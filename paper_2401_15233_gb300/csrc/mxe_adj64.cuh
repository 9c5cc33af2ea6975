// mxe_adj64.cuh -- FP64 reverse mode of one planar face state, of the BGK
// source and of the primitive recovery, arranged for the fewest FP64-pipe
// operations (see mxe_fast64.cuh for why that is the measure).  The derivatives
// are those of mxe_adjoint.cuh:
//   * the face state is evaluated as in mxe_face64.cuh, with the reciprocals
//     and roots it forms kept for the reverse, which then divides nowhere but
//     by P*_kk;
//   * HLL and Rusanov give each state the adjoints U-bar = beta F-bar and
//     F-bar' = alpha F-bar: two scalars, found from the two lanes' dot products
//     of F-bar with U and F;
//   * the scalings by p, theta and sqrt(theta) are reversed through their
//     logarithms (one sum of products each);
//   * tr P* = 3 identically: its adjoint has no effect on P and is not formed.
// The state vectors are indexed in the flux frame: K = flux direction, O the
// other one.
//
// 128 x 128, three recorded RK2 steps and their reverse sweep on GB300: 3.6 ms
// with the derivatives of mxe_adjoint.cuh in FP64 (about 45 divisions a face
// state, 20 values exchanged with the partner lane, each limiter in FP64 field by
// field, blocks of 64 faces of one line), 1.84 ms with these.
#pragma once
#include "mxe_adjoint.cuh"
#include "mxe_face64.cuh"

namespace mxe {
namespace f64 {

// x > 0 without the FP64 pipe (false for NaN)
__device__ __forceinline__ bool gt0(double x) { return __double_as_longlong(x) > 0 && !is_nan(x); }
// x 2^e: exponent arithmetic while argument and result are normal
__device__ __forceinline__ double scale2(double x, int e) {
    const unsigned h = hi32(x), ex = (h >> 20) & 0x7ffu;
    const int ne = (int)ex + e;
    if (ex - 1u < 2046u && ne > 0 && ne < 2047)
        return __hiloint2double((int)(h + ((unsigned)e << 20)), (int)lo32(x));
    return ((h & 0x7fffffffu) | lo32(x)) == 0u ? x : ::ldexp(x, e);
}

// zeta bracket h = zeta + sqrt(D), D = zeta^2 + D0, with what its reverse needs
struct BracketAdj {
    double z, h, irt, is;        // 1 / sqrt(D); 1 / (sqrt(D) + |zeta|) for zeta < 0
    bool none, neg;
};
__device__ __forceinline__ BracketAdj bracket_fwd(double z, double D0) {
    BracketAdj b;
    const double D = ::fma(z, z, D0);
    b.z = z;
    b.none = __double_as_longlong(D) <= 0 && !is_nan(D);
    b.neg = is_neg(z);
    double rt;
    sqrt_rsqrt(b.none ? 1.0 : D, rt, b.irt);
    const double s = rt + abs_(z);
    b.is = 0.0;
    b.h = s;
    if (b.neg) {
        b.is = rcp(s);
        b.h = D0 * b.is;
    }
    if (b.none) b.h = z;
    return b;
}
// adjoint hb of h -> zb (returned), D0b
__device__ __forceinline__ double bracket_rev(const BracketAdj& b, double hb, double& D0b) {
    D0b = 0.0;
    if (b.none) return hb;
    double zb = hb, rtb = hb;
    if (b.neg) {                 // h = D0 / (rt - z)
        D0b = hb * b.is;
        rtb = -D0b * b.h;
        zb = -rtb;
    }
    const double Db = 0.5 * rtb * b.irt;
    D0b += Db;
    return ::fma(b.z + b.z, Db, zb);
}

// Weights alpha, beta of the numerical flux's adjoint for the own state of a
// face, and the adjoints of its wave speeds, from the dot products of F-bar
// with U and F of both states.  HLL: with dU = U_R - U_L, dF = F_R - F_L,
//   d F / d S_R = S_L (dF - S_L dU) / (S_R - S_L)^2,
//   d F / d S_L = S_R (S_R dU - dF) / (S_R - S_L)^2.
struct FluxAdj {
    double alpha, beta, lob, hib;
};
__device__ __forceinline__ FluxAdj riemann_rev(bool isL, int flux, double lo, double hi,
                                               double dotU, double dotF) {
    const double plo = __shfl_xor_sync(0xffffffffu, lo, 1);
    const double phi = __shfl_xor_sync(0xffffffffu, hi, 1);
    const double pU = __shfl_xor_sync(0xffffffffu, dotU, 1);
    const double pF = __shfl_xor_sync(0xffffffffu, dotF, 1);
    const double l0 = isL ? lo : plo, l1 = isL ? hi : phi, r0 = isL ? plo : lo, r1 = isL ? phi : hi;
    FluxAdj w{0.0, 0.0, 0.0, 0.0};
    const double dU = isL ? pU - dotU : dotU - pU;
    if (flux == 1) {
        double s = abs_(l0);
        int sel_ = 0;
        double v = abs_(l1);
        if (lt(s, v)) { s = v; sel_ = 1; }
        v = abs_(r0);
        if (lt(s, v)) { s = v; sel_ = 2; }
        v = abs_(r1);
        if (lt(s, v)) { s = v; sel_ = 3; }
        w.alpha = 0.5;
        w.beta = isL ? 0.5 * s : -0.5 * s;
        const double lam = sel_ == 0 ? l0 : sel_ == 1 ? l1 : sel_ == 2 ? r0 : r1;
        const double sb = -0.5 * dU;
        const double g = gt0(lam) ? sb : is_neg(lam) ? -sb : 0.0;
        if ((sel_ < 2) == isL) {
            if (sel_ & 1) w.hib = g;
            else w.lob = g;
        }
        return w;
    }
    const bool Lmin = lt(l0, r0), Lmax = lt(r1, l1);
    const double SL = sel(Lmin, l0, r0), SR = sel(Lmax, l1, r1);
    if (ge0(SL)) {
        w.alpha = isL ? 1.0 : 0.0;
    } else if (le0(SR)) {
        w.alpha = isL ? 0.0 : 1.0;
    } else {
        const double dF = isL ? pF - dotF : dotF - pF;
        const double inv = rcp(SR - SL), cl = SR * inv, cr = -SL * inv;
        w.alpha = isL ? cl : cr;
        w.beta = isL ? cr * SR : -cr * SR;
        // S_L inv = -cr, S_R inv = cl
        const double SRb = -cr * inv * ::fma(-SL, dU, dF), SLb = cl * inv * ::fma(SR, dU, -dF);
        if (isL == Lmin) w.lob = SLb;
        if (isL == Lmax) w.hib = SRb;
    }
    return w;
}

// One face state (left state in the even lane, right in the odd): evaluates
// it, reverses the numerical flux with the partner lane's scalars, then the
// state itself.  Fb: adjoint of the face flux (the same in both lanes); Qb:
// adjoint of the state's primitives.  Lanes with !live take part in the
// exchange and return zeros.
template <int K>
__device__ __forceinline__ void face_adj_p(const double* Q, double slim, double kw, int flux,
                                           const double* Fb, bool live, double* Qb) {
    constexpr int iK = 1 + K, iO = 2 - K;                    // velocities
    constexpr int kKK = K == 0 ? 3 : 5, kOO = K == 0 ? 5 : 3;    // second moments, Pxy = 4
    constexpr int qK = 7 + K, qO = 8 - K;                    // heat fluxes
    // ---- dimensionless state
    const double rho = Q[0];
    const double tr = Q[3] + Q[5] + Q[6], p = tr * (1.0 / 3.0);
    const double ip = rcp(p), ir = rcp(rho), th = p * ir;
    double sq, rsq;
    sqrt_rsqrt(th, sq, rsq);
    const double isc3 = ip * rsq, rip2 = rho * ip * ip;
    const double a = Q[kKK] * ip, b = Q[4] * ip, d = Q[kOO] * ip, f = Q[6] * ip;
    const double qs = Q[qK] * isc3, qo = Q[qO] * isc3;
    const double Rs = Q[9] * rip2;
    const double t = a + d + f, bb = b * b;
    const double T2 = ::fma(a, a, ::fma(d, d, ::fma(f, f, bb + bb)));
    const double i2 = rcp(::fma(a, d, -bb));
    const double yK = ::fma(d, qs, -b * qo) * i2, yO = ::fma(a, qo, -b * qs) * i2;
    const double T4 = 4.0 * T2, qPq = ::fma(qs, yK, qo * yO);
    const double A = ::fma(t, t, ::fma(2.0, T2, -Rs)), X = (T4 + T4) * qPq;
    double rt, irt;
    sqrt_rsqrt(::fma(A, A, X), rt, irt);
    const bool Aneg = is_neg(A);
    const double srt = rt + abs_(A);
    const double rden = rcp(sel(Aneg, T4 * srt, T4));
    const double sig = sel(Aneg, X, srt) * rden;
    const double sb = clamp_sigma(sig, slim);
    double ssb, rssb;
    sqrt_rsqrt(sb, ssb, rssb);
    const double isb = rssb * rssb;
    // ---- wave speeds
    const double l2 = log2_(a);
    const double ea = exp2_(::fma(1.1, l2, -LOG2E * (a * a))), e1 = exp2_(1.4 * l2);
    const double eb = exp2_((-0.5 * LOG2E) * e1);
    const double pb45 = 0.45 * a * eb, pre = ::fma(pb45, isb, 0.7 * ea);
    const double a3 = 3.0 * a;
    double C, iC, sR, isR, sB, isB;
    sqrt_rsqrt(::fma(-sb, a3, a3), C, iC);
    const double E = 0.8 * C;
    sqrt_rsqrt(::fma(-6.0, ssb, 10.0) * (1.0 - ssb), sR, isR);
    sqrt_rsqrt(::fma(-4.0, ssb, 5.0) + sR, sB, isB);
    const double dd = sB - E, sd = sb * dd, sbE = sb * E;
    const double qp = abs_(qo), poly = ::fma(a, ::fma(0.6, a, -0.38), 0.35), al = qp * poly;
    const double base = ::fma(4.0 * sd, sd, 0.1 * qo * qo);
    const double zp = qs + al, zm = al - qs;
    const BracketAdj Bp = bracket_fwd(zp, ::fma(-zp, sbE, base));
    const BracketAdj Bm = bracket_fwd(zm, ::fma(-zm, sbE, base));
    const double lp = ::fma(pre, Bp.h, E), lm = ::fma(pre, Bm.h, E), ks = kw * sq;
    const double uK = Q[iK], uO = Q[iO];
    const double hi = ::fma(lp, ks, uK), lo = ::fma(-lm, ks, uK);
    // ---- closure along K
    const double P2KK = ::fma(a, a, bb), apd = a + d, P2KO = b * apd, P2OO = ::fma(d, d, bb);
    const double P2zz = f * f;
    const double P3KK = ::fma(P2KK, a, P2KO * b), P3KO = ::fma(P2KK, b, P2KO * d);
    const double P3OO = ::fma(P2KO, b, P2OO * d);
    const double trP3 = ::fma(P2zz, f, P3KK + P3OO);
    const double h2 = 0.5 * T2;
    const double BKK = ::fma(h2, a, P3KK), BKO = ::fma(h2, b, P3KO), BOO = ::fma(h2, d, P3OO);
    const double iB = 0.25 * rcp(::fma(BKK, BOO, -BKO * BKO));
    const double vK = ::fma(BOO, qs, -BKO * qo) * iB, vO = ::fma(BKK, qo, -BKO * qs) * iB;
    double w2K = ::fma(a, vK, b * vO), w2O = ::fma(b, vK, d * vO);
    w2K += w2K;
    w2O += w2O;
    const double tP2KK = 3.0 * P2KK, dP2KO = P2KO + P2KO;
    const double q0 = w2K * tP2KK, q1 = ::fma(w2K, dP2KO, w2O * P2KK);
    const double q2 = ::fma(w2K, P2OO, w2O * dP2KO), q3 = w2K * P2zz;
    const double om2 = ::fma(-2.0, sb, 2.0), om1 = 1.0 - ssb;
    const double t1 = ::fma(q0, yK, q1 * yO), t2 = ::fma(q1, yK, q2 * yO);
    const double yQy = ::fma(yK, t1, yO * t2);
    const double c1 = ::fma(t + t, ::fma(t, t, -T2), 12.0 * trP3);
    const double c2 = ::fma(14.0, T2, -6.0 * (t * t)), c3 = 20.0 * t;
    const double P2s = P2KK + P2OO, P4KK = ::fma(P2KK, P2KK, P2KO * P2KO), P4KO = P2KO * P2s;
    const double mKK = ::fma(c1, a, ::fma(c2, P2KK, ::fma(c3, P3KK, 20.0 * P4KK)));
    const double mKO = ::fma(c1, b, ::fma(c2, P2KO, ::fma(c3, P3KO, 20.0 * P4KO)));
    const double Wq = ::fma(mKK, vK, mKO * vO);
    const double isb2 = isb * isb, tq = t * qs;
    const double Ss = ::fma(yQy, isb2, ::fma(ssb + ssb, tq, om1 * Wq));
    const double sc3 = p * sq, sc4 = p * th, sc5 = sc4 * sq;
    const double QK0 = q0 * sc3, QK1 = q1 * sc3, QK2 = q2 * sc3, QK3 = q3 * sc3;
    const double RKK = sc4 * ::fma(t1, isb, ::fma(om2, P2KK, a * t));
    const double ROK = sc4 * ::fma(t2, isb, ::fma(om2, P2KO, b * t)), SK = Ss * sc5;
    // ---- conserved state and flux, against F-bar
    const double PKK = Q[kKK], PKO = Q[4], POO = Q[kOO];
    const double mK = rho * uK, mO = rho * uO;
    const double u2 = ::fma(uK, uK, uO * uO), ru2 = rho * u2, e = ru2 + tr;
    const double PuK = ::fma(PKK, uK, PKO * uO), PuO = ::fma(PKO, uK, POO * uO);
    const double PqK = PuK + Q[qK], PqO = PuO + Q[qO];
    const double e2 = ::fma(2.0, tr, ru2);
    const double QuK = ::fma(QK0, uK, QK1 * uO), QuO = ::fma(QK1, uK, QK2 * uO);
    const double gK = ::fma(2.0, PuK, Q[qK]), QRK = QuK + RKK, QRO = QuO + ROK;
    double dotU, cen;            // F-bar . U and F-bar . (F - u_K U)
    {
        double s = Fb[0] * rho;
        s = ::fma(Fb[iK], mK, s);
        s = ::fma(Fb[iO], mO, s);
        s = ::fma(Fb[kKK], ::fma(mK, uK, PKK), s);
        s = ::fma(Fb[4], ::fma(mK, uO, PKO), s);
        s = ::fma(Fb[kOO], ::fma(mO, uO, POO), s);
        s = ::fma(Fb[6], Q[6], s);
        s = ::fma(Fb[qK], ::fma(uK, e, ::fma(2.0, PuK, Q[qK])), s);
        s = ::fma(Fb[qO], ::fma(uO, e, ::fma(2.0, PuO, Q[qO])), s);
        dotU = ::fma(Fb[9], ::fma(u2, e2, ::fma(4.0, ::fma(uK, PqK, uO * PqO), Q[9])), s);
        double c = Fb[iK] * PKK;
        c = ::fma(Fb[iO], PKO, c);
        c = ::fma(Fb[kKK], ::fma(uK + uK, PKK, QK0), c);
        c = ::fma(Fb[4], ::fma(uK, PKO, ::fma(uO, PKK, QK1)), c);
        c = ::fma(Fb[kOO], ::fma(uO + uO, PKO, QK2), c);
        c = ::fma(Fb[6], QK3, c);
        c = ::fma(Fb[qK], ::fma(uK, gK, ::fma(u2, PKK, ::fma(2.0, QuK, RKK))), c);
        c = ::fma(Fb[qO], ::fma(uO, gK, ::fma(u2, PKO, ::fma(2.0, QuO, ROK))), c);
        cen = ::fma(Fb[9], ::fma(u2 + u2, gK, ::fma(4.0, ::fma(uK, QRK, uO * QRO), SK)), c);
    }
    const FluxAdj w = riemann_rev((threadIdx.x & 1) == 0, flux, lo, hi, dotU,
                                  ::fma(uK, dotU, cen));
#pragma unroll
    for (int k = 0; k < NP; ++k) Qb[k] = 0.0;
    if (!live) return;

    // ---- reverse of the flux's central part, f = alpha F-bar
    double uKb, uOb, u2b, PKKb, PKOb, POOb, qKb, qOb;
    double Q0b, Q1b, Q2b, Q3b, R1, R2;       // adjoints of Q_K.., R_KK, R_OK
    const double f9 = w.alpha * Fb[9];
    {
        const double fmK = w.alpha * Fb[iK], fmO = w.alpha * Fb[iO], fKK = w.alpha * Fb[kKK];
        const double fKO = w.alpha * Fb[4], fOO = w.alpha * Fb[kOO];
        const double fqK = w.alpha * Fb[qK], fqO = w.alpha * Fb[qO];
        Q3b = w.alpha * Fb[6];
        const double k4 = 4.0 * f9, k4K = k4 * uK, k4O = k4 * uO;
        const double gKb = ::fma(u2 + u2, f9, ::fma(uK, fqK, uO * fqO));
        u2b = ::fma(gK + gK, f9, ::fma(PKK, fqK, PKO * fqO));
        const double QuKb = ::fma(2.0, fqK, k4K), QuOb = ::fma(2.0, fqO, k4O);
        R1 = k4K + fqK;
        R2 = k4O + fqO;
        qKb = gKb;
        const double PuKb = gKb + gKb;
        PKKb = ::fma(u2, fqK, ::fma(uK + uK, fKK, ::fma(uO, fKO, ::fma(PuKb, uK, fmK))));
        PKOb = ::fma(u2, fqO, ::fma(uO + uO, fOO, ::fma(uK, fKO, ::fma(PuKb, uO, fmO))));
        uKb = w.alpha * dotU;
        uKb = ::fma(k4, QRK, uKb);
        uKb = ::fma(gK, fqK, uKb);
        uKb = ::fma(PuKb, PKK, uKb);
        uKb = ::fma(PKK + PKK, fKK, uKb);
        uKb = ::fma(PKO, fKO, uKb);
        uKb = ::fma(QuKb, QK0, ::fma(QuOb, QK1, uKb));
        uOb = k4 * QRO;
        uOb = ::fma(gK, fqO, uOb);
        uOb = ::fma(PuKb, PKO, uOb);
        uOb = ::fma(PKK, fKO, uOb);
        uOb = ::fma(PKO + PKO, fOO, uOb);
        uOb = ::fma(QuKb, QK1, ::fma(QuOb, QK2, uOb));
        Q0b = ::fma(QuKb, uK, fKK);
        Q1b = ::fma(QuKb, uO, ::fma(QuOb, uK, fKO));
        Q2b = ::fma(QuOb, uO, fOO);
    }
    // ---- reverse of the conserved state, U-bar = gamma F-bar
    double rhob, trb;
    {
        const double gam = ::fma(uK, w.alpha, w.beta);
        const double h9 = gam * Fb[9], k4 = 4.0 * h9, hqK = gam * Fb[qK], hqO = gam * Fb[qO];
        const double hKK = gam * Fb[kKK], hKO = gam * Fb[4], hOO = gam * Fb[kOO];
        Qb[9] = h9;
        Qb[6] = gam * Fb[6];
        u2b = ::fma(h9, e2, u2b);
        const double xK = k4 * uK, xO = k4 * uO;
        qKb += xK + hqK;
        qOb = xO + hqO;
        const double PuKb = ::fma(2.0, hqK, xK), PuOb = ::fma(2.0, hqO, xO);
        const double eb = ::fma(uK, hqK, uO * hqO);
        const double ru2b = ::fma(u2, h9, eb);
        trb = ::fma(u2 + u2, h9, eb);
        u2b = ::fma(rho, ru2b, u2b);
        const double mKb = ::fma(uK, hKK, ::fma(uO, hKO, gam * Fb[iK]));
        const double mOb = ::fma(uO, hOO, gam * Fb[iO]);
        rhob = ::fma(u2, ru2b, ::fma(uK, mKb, ::fma(uO, mOb, gam * Fb[0])));
        uKb = ::fma(k4, PqK, uKb);
        uKb = ::fma(e, hqK, uKb);
        uKb = ::fma(PKK, PuKb, ::fma(PKO, PuOb, uKb));
        uKb = ::fma(mK, hKK, ::fma(rho, mKb, uKb));
        uOb = ::fma(k4, PqO, uOb);
        uOb = ::fma(e, hqO, uOb);
        uOb = ::fma(PKO, PuKb, ::fma(POO, PuOb, uOb));
        uOb = ::fma(mK, hKO, ::fma(mO, hOO, ::fma(rho, mOb, uOb)));
        PKKb = ::fma(PuKb, uK, PKKb + hKK);
        PKOb = ::fma(PuKb, uO, ::fma(PuOb, uK, PKOb + hKO));
        POOb = ::fma(PuOb, uO, hOO);
        const double u2b2 = u2b + u2b;
        uKb = ::fma(u2b2, uK, uKb);
        uOb = ::fma(u2b2, uO, uOb);
    }
    // ---- reverse of the closure
    double ab, bbar, db, fb, qsb, qob, T2b, yKb, yOb, isbb, ssbb, sbb;
    const double Z3 = ::fma(Q0b, QK0, ::fma(Q1b, QK1, ::fma(Q2b, QK2, Q3b * QK3)));
    const double Z4 = ::fma(R1, RKK, R2 * ROK), Z5 = f9 * SK;
    {
        double q0b = Q0b * sc3, q1b = Q1b * sc3, q2b = Q2b * sc3;
        const double q3b = Q3b * sc3, r1 = R1 * sc4, r2 = R2 * sc4, s = f9 * sc5;
        const double yQyb = s * isb2;
        const double Wqb = s * om1, mKKb = Wqb * vK, mKOb = Wqb * vO;
        qsb = (s + s) * ssb * t;
        ssbb = s * ::fma(2.0, tq, -Wq);
        double vKb = Wqb * mKK, vOb = Wqb * mKO;
        const double c1b = ::fma(mKOb, b, mKKb * a), c2b = ::fma(mKOb, P2KO, mKKb * P2KK);
        bbar = mKOb * c1;
        ab = mKKb * c1;
        const double m20K = 20.0 * mKKb, k = 20.0 * mKOb;
        double P2KOb = ::fma(k, P2s, ::fma(m20K, dP2KO, mKOb * c2));
        const double kP = k * P2KO;
        double P2KKb = ::fma(m20K + m20K, P2KK, ::fma(mKKb, c2, kP)), P2OOb = kP;
        T2b = ::fma(14.0, c2b, -(t + t) * c1b);
        const double trP3b = 12.0 * c1b;
        const double t1b = ::fma(yQyb, yK, r1 * isb), t2b = ::fma(yQyb, yO, r2 * isb);
        yKb = ::fma(yQyb, t1, ::fma(t1b, q0, t2b * q1));
        yOb = ::fma(yQyb, t2, ::fma(t1b, q1, t2b * q2));
        isbb = ::fma((s + s) * yQy, isb, ::fma(r1, t1, r2 * t2));
        q0b = ::fma(t1b, yK, q0b);
        q1b = ::fma(t1b, yO, ::fma(t2b, yK, q1b));
        q2b = ::fma(t2b, yO, q2b);
        sbb = -2.0 * ::fma(r1, P2KK, r2 * P2KO);
        ab = ::fma(t, r1, ab);
        bbar = ::fma(t, r2, bbar);
        // q. = w P^2
        double wKb = ::fma(tP2KK, q0b, ::fma(dP2KO, q1b, ::fma(P2OO, q2b, P2zz * q3b)));
        double wOb = ::fma(P2KK, q1b, dP2KO * q2b);
        wKb += wKb;
        wOb += wOb;
        P2KKb = ::fma(3.0 * w2K, q0b, ::fma(w2O, q1b, ::fma(om2, r1, P2KKb)));
        P2KOb = ::fma(2.0, ::fma(w2K, q1b, w2O * q2b), ::fma(om2, r2, P2KOb));
        P2OOb = ::fma(w2K, q2b, P2OOb);
        // w = P* v
        ab = ::fma(wKb, vK, ab);
        bbar = ::fma(wKb, vO, ::fma(wOb, vK, bbar));
        db = wOb * vO;
        vKb = ::fma(wKb, a, ::fma(wOb, b, vKb));
        vOb = ::fma(wKb, b, ::fma(wOb, d, vOb));
        // v = B^-1 q*
        const double nK = vKb * iB, nO = vOb * iB;
        const double detb = -4.0 * ::fma(nK, vK, nO * vO);
        qsb = ::fma(nK, BOO, ::fma(-nO, BKO, qsb));
        qob = ::fma(nO, BKK, -nK * BKO);
        const double BKKb = ::fma(nO, qo, detb * BOO), BOOb = ::fma(nK, qs, detb * BKK);
        const double BKOb = -::fma(nK, qo, ::fma(nO, qs, (detb + detb) * BKO));
        ab = ::fma(h2, BKKb, ab);
        bbar = ::fma(h2, BKOb, bbar);
        db = ::fma(h2, BOOb, db);
        T2b = ::fma(0.5, ::fma(a, BKKb, ::fma(b, BKOb, d * BOOb)), T2b);
        // P*^3 = P*^2 P*
        const double P3KKb = ::fma(mKKb, c3, BKKb + trP3b), P3KOb = ::fma(mKOb, c3, BKOb);
        const double P3OOb = BOOb + trP3b;
        fb = trP3b * P2zz;
        const double P2zzb = ::fma(trP3b, f, w2K * q3b);
        P2KKb = ::fma(P3KKb, a, ::fma(P3KOb, b, P2KKb));
        P2KOb = ::fma(P3KKb, b, ::fma(P3KOb, d, ::fma(P3OOb, b, P2KOb)));
        P2OOb = ::fma(P3OOb, d, P2OOb);
        ab = ::fma(P3KKb, P2KK, ab);
        bbar = ::fma(P3KKb, P2KO, ::fma(P3KOb, P2KK, ::fma(P3OOb, P2KO, bbar)));
        db = ::fma(P3KOb, P2KO, ::fma(P3OOb, P2OO, db));
        // P*^2
        const double bP = b * P2KOb;
        ab += ::fma(a + a, P2KKb, bP);
        db += ::fma(d + d, P2OOb, bP);
        bbar = ::fma(b + b, P2KKb + P2OOb, ::fma(apd, P2KOb, bbar));
        fb = ::fma(f + f, P2zzb, fb);
    }
    // ---- reverse of the wave speeds: hi = u + lp ks, lo = u - lm ks
    double Zs;                   // adjoint of sqrt(theta) times sqrt(theta)
    {
        uKb += w.hib + w.lob;
        Zs = ks * ::fma(w.hib, lp, -w.lob * lm);
        const double lpb = w.hib * ks, lmb = -w.lob * ks;
        const double preb = ::fma(lpb, Bp.h, lmb * Bm.h);
        double Eb = lpb + lmb, Dp, Dm;
        double zpb = bracket_rev(Bp, lpb * pre, Dp), zmb = bracket_rev(Bm, lmb * pre, Dm);
        const double baseb = Dp + Dm, sEb = -::fma(zp, Dp, zm * Dm);
        zpb = ::fma(-sbE, Dp, zpb);
        zmb = ::fma(-sbE, Dm, zmb);
        const double sdb = 8.0 * sd * baseb, ddb = sb * sdb;
        sbb = ::fma(E, sEb, ::fma(dd, sdb, sbb));
        Eb = ::fma(sb, sEb, Eb) - ddb;
        const double Bb = 0.5 * ddb * isB;
        ssbb = ::fma(-4.0, Bb, ssbb);
        if (gt0(sR)) ssbb = ::fma(0.5 * Bb * isR, ::fma(12.0, ssb, -16.0), ssbb);
        double Pb = 0.0;
        if (gt0(C)) {
            const double vb = 0.4 * Eb * iC;                 // E = 0.8 C, C^2 = 3 (1 - sigma) P
            sbb = ::fma(-a3, vb, sbb);
            Pb = ::fma(-3.0, sb, 3.0) * vb;
        }
        const double alb = zpb + zmb;
        const double qpb = ::fma(0.2 * qp, baseb, alb * poly);
        Pb = ::fma(alb * qp, ::fma(1.2, a, -0.38), Pb);
        qsb += zpb - zmb;
        if (((hi32(qo) & 0x7fffffffu) | lo32(qo)) != 0u) qob += is_neg(qo) ? -qpb : qpb;
        const double eab = 0.7 * preb * ea, x = preb * eb * 0.45;
        isbb = ::fma(preb, pb45, isbb);
        Pb = ::fma(x, isb, Pb);
        const double eb2 = -0.7 * (x * a) * isb * e1;        // 1.4 e1 (-eb/2) adjoint
        Pb = ::fma(-2.0 * a, eab, Pb);
        ab = ::fma(::fma(1.1, eab, eb2), rcp(a), ab + Pb);
        sbb = ::fma(0.5 * ssbb, rssb, ::fma(-isbb, isb2, sbb));
    }
    // ---- reverse of sigma
    double Ab = 0.0;
    if (!lt(sig, slim) && !lt(1.0, sig)) {
        double Xb = 0.0, rtb;
        const double k = sbb * rden;
        if (!Aneg) {                         // sigma = (A + rt) / T4
            Ab = rtb = k;
            T2b = ::fma(-4.0 * k, sig, T2b);
        } else {                             // sigma = X / (T4 (rt - A))
            Xb = k;
            const double Db = -k * sig;
            T2b = ::fma(4.0 * srt, Db, T2b);
            rtb = Db * T4;
            Ab = -rtb;
        }
        if (gt0(rt)) {
            const double v = rtb * irt;
            Ab = ::fma(v, A, Ab);
            Xb = ::fma(0.5, v, Xb);
        }
        T2b = ::fma(2.0, Ab, ::fma(8.0 * qPq, Xb, T2b));
        const double k8 = (T4 + T4) * Xb;
        qsb = ::fma(k8, yK, qsb);
        qob = ::fma(k8, yO, qob);
        yKb = ::fma(k8, qs, yKb);
        yOb = ::fma(k8, qo, yOb);
    }
    // ---- y = P*^-1 q*, T2, and the scalings
    const double nK = yKb * i2, nO = yOb * i2, det = -::fma(nK, yK, nO * yO);
    qsb = ::fma(nK, d, ::fma(-nO, b, qsb));
    qob = ::fma(nO, a, ::fma(-nK, b, qob));
    const double T2x = T2b + T2b;
    ab = ::fma(nO, qo, ::fma(det, d, ::fma(a, T2x, ab)));
    db = ::fma(nK, qs, ::fma(det, a, ::fma(d, T2x, db)));
    bbar = ::fma(-nK, qo, ::fma(-nO, qs, ::fma(b + b, T2x - det, bbar)));
    fb = ::fma(f, T2x, fb);
    const double ZR = -Ab * Rs, Zq = ::fma(qsb, qs, qob * qo);
    const double ZP = ::fma(ab, a, ::fma(bbar, b, ::fma(db, d, fb * f)));
    Zs += Z3 + Z5 - Zq;                                      // ln sqrt(theta)
    const double Zt = ::fma(0.5, Zs, Z4 + Z5);               // ln theta
    const double Zp = Z3 + Z4 + Z5 - Zq - ZP - (ZR + ZR) + Zt;   // ln p
    Qb[0] = ::fma(ZR - Zt, ir, rhob);
    Qb[iK] = uKb;
    Qb[iO] = uOb;
    const double pd = ::fma(Zp, ip * (1.0 / 3.0), trb);      // to each diagonal pressure
    Qb[kKK] = ::fma(ab, ip, PKKb + pd);
    Qb[4] = ::fma(bbar, ip, PKOb);
    Qb[kOO] = ::fma(db, ip, POOb + pd);
    Qb[6] = ::fma(fb, ip, Qb[6] + pd);
    Qb[qK] = ::fma(qsb, isc3, qKb);
    Qb[qO] = ::fma(qob, isc3, qOb);
    Qb[9] = ::fma(-Ab, rip2, Qb[9]);
}

// Reverse of source_p: W = adjoint of the source vector -> Qb (added); returns
// the adjoint of tau_ref.  it = 1/tau = k sqrt(rho p) (hard spheres) or k.
__device__ __forceinline__ double source_rev_p(int model, double it, double tau_ref,
                                               const double* Q, const double* W, double* Qb) {
    const double rho = Q[0], ux = Q[1], uy = Q[2], Pxy = Q[4];
    const double p = (Q[3] + Q[5] + Q[6]) * (1.0 / 3.0), ir = rcp(rho), pr = p * ir;
    const double Dx = Q[3] - p, Dy = Q[5] - p, Dz = Q[6] - p;
    // N = (P - p I, 2 a + q, 4 u.(a + q) + R - 15 p^2 / rho), a = (P - p I) u
    const double ax = ::fma(Dx, ux, Pxy * uy), ay = ::fma(Pxy, ux, Dy * uy);
    const double sx = ax + Q[7], sy = ay + Q[8];
    const double N9 = ::fma(4.0, ::fma(ux, sx, uy * sy), ::fma(-15.0 * p, pr, Q[9]));
    double WN = ::fma(W[3], Dx, ::fma(W[4], Pxy, ::fma(W[5], Dy, W[6] * Dz)));
    WN = ::fma(W[7], ax + sx, ::fma(W[8], ay + sy, ::fma(W[9], N9, WN)));
    const double nit = -it, n9 = W[9] * nit, n7 = W[7] * nit, n8 = W[8] * nit, k = 4.0 * n9;
    const double kx = k * ux, ky = k * uy;
    const double axb = ::fma(2.0, n7, kx), ayb = ::fma(2.0, n8, ky);
    const double Dxb = ::fma(W[3], nit, axb * ux), Dyb = ::fma(W[5], nit, ayb * uy);
    const double Dzb = W[6] * nit, L = WN * nit;             // adjoint of ln(1/tau)
    double rhob = (15.0 * pr) * pr * n9, pb = ::fma(-30.0 * pr, n9, -(Dxb + Dyb + Dzb));
    if (model != 1) {
        rhob = ::fma(0.5 * L, ir, rhob);
        pb = ::fma(0.5 * L, rcp(p), pb);
    }
    pb *= 1.0 / 3.0;
    Qb[0] += rhob;
    Qb[1] += ::fma(k, sx, ::fma(axb, Dx, ayb * Pxy));
    Qb[2] += ::fma(k, sy, ::fma(axb, Pxy, ayb * Dy));
    Qb[3] += Dxb + pb;
    Qb[4] += ::fma(W[4], nit, ::fma(axb, uy, ayb * ux));
    Qb[5] += Dyb + pb;
    Qb[6] += Dzb + pb;
    Qb[7] += kx + n7;
    Qb[8] += ky + n8;
    Qb[9] += n9;
    return -L * rcp(tau_ref);
}

// Reverse of the primitive recovery Q = prim(U): the transposed Jacobian of
// U(Q) is triangular, so U-bar follows from Q-bar by back substitution.
__device__ __forceinline__ void cons2prim_rev_p(const double* Q, const double* Qb, double* Ub) {
    const double rho = Q[0], ux = Q[1], uy = Q[2], Pxx = Q[3], Pxy = Q[4], Pyy = Q[5];
    const double tr = Pxx + Pyy + Q[6], ir = rcp(rho);
    const double u2 = ::fma(ux, ux, uy * uy), ru2 = rho * u2, e = ru2 + tr;
    const double sx = ::fma(Pxx, ux, ::fma(Pxy, uy, Q[7]));
    const double sy = ::fma(Pxy, ux, ::fma(Pyy, uy, Q[8]));
    const double h9 = Qb[9], k = 4.0 * h9, kx = k * ux, ky = k * uy;
    const double h7 = Qb[7] - kx, h8 = Qb[8] - ky;
    const double Px = ::fma(2.0, h7, kx), Py = ::fma(2.0, h8, ky);      // adjoints of P u
    const double eb = ::fma(ux, h7, uy * h8);
    const double rb = ::fma(u2, h9, eb), tb = ::fma(u2 + u2, h9, eb);   // of rho u^2 and tr P
    const double h3 = ::fma(-Px, ux, Qb[3] - tb), h5 = ::fma(-Py, uy, Qb[5] - tb);
    const double h4 = ::fma(-Px, uy, ::fma(-Py, ux, Qb[4]));
    const double u2b = ::fma(::fma(2.0, tr, ru2), h9, rho * rb);
    const double mx = rho * ux, my = rho * uy, v2 = u2b + u2b;
    double Sx = ::fma(k, sx, ::fma(e, h7, ::fma(Pxx, Px, ::fma(Pxy, Py, v2 * ux))));
    double Sy = ::fma(k, sy, ::fma(e, h8, ::fma(Pxy, Px, ::fma(Pyy, Py, v2 * uy))));
    Sx = ::fma(mx + mx, h3, ::fma(my, h4, Sx));
    Sy = ::fma(my + my, h5, ::fma(mx, h4, Sy));
    const double h1 = (Qb[1] - Sx) * ir, h2 = (Qb[2] - Sy) * ir;
    Ub[1] = h1;
    Ub[2] = h2;
    Ub[3] = h3;
    Ub[4] = h4;
    Ub[5] = h5;
    Ub[6] = Qb[6] - tb;
    Ub[7] = h7;
    Ub[8] = h8;
    Ub[9] = h9;
    Ub[0] = Qb[0] - ::fma(u2, rb, ::fma(ux, ::fma(ux, h3, ::fma(uy, h4, h1)),
                                        uy * ::fma(uy, h5, h2)));
}

// Shared limiter of a stencil (limiter_at) with the partial derivatives of
// phi with respect to the setting field's differences.
template <class At>
__device__ __forceinline__ adj::PhiAdj<double> phi_adj_at(const At& at, int lim, bool frozen) {
    adj::PhiAdj<double> r{1.0, 0.0, 0.0, -1};
    r.phi = limiter_at<NP>(at, lim, r.ks);
    if (frozen) r.ks = -1;
    if (r.ks < 0) return r;
    const double dm = at(0, r.ks) - at(-1, r.ks), dp = at(1, r.ks) - at(0, r.ks);
    if (lim == 1) {
        const double d2 = dm * dm, e2 = dp * dp, is = rcp(d2 + e2), q = 2.0 * (e2 - d2) * is * is;
        r.ddm = q * dp;
        r.ddp = -q * dm;
    } else {
        const double am = abs_(dm), ap = abs_(dp), is = rcp(am + ap), q = 2.0 * is * is;
        const double sg = is_neg(dm) ? -q : q;               // both differences have its sign
        r.ddm = lt(am, ap) ? sg * ap : -sg * ap;
        r.ddp = lt(am, ap) ? -sg * am : sg * am;
    }
    return r;
}

}  // namespace f64
}  // namespace mxe
