// mxe_general_x2.cuh -- the general 14-moment face-state evaluation for the
// two states of a face at once, in packed FP32 (f32x2): the formulas of
// dimless14 / closure14_slice / prim2cons14 / flux14 / lam14_star, arranged as
// in mxe_planar_x2.cuh (wave speeds first, each field's U and K-flux weighed
// into the face flux as it is formed, one reciprocal per denominator).
#pragma once
#include "mxe_planar_x2.cuh"

namespace mxe {
namespace x2 {

// the jump of a product x y from the jumps of its factors
__device__ __forceinline__ float djump(v2 x, float dx, v2 y, float dy) {
    return fmaf(x.y, dy, y.x * dx);
}
// cofactors of a symmetric 3 x 3 matrix (xx, xy, xz, yy, yz, zz); returns det
__device__ __forceinline__ v2 cofactors(const v2* A, v2* c) {
    const v2 n1 = neg(A[1]), n2 = neg(A[2]), n4 = neg(A[4]);
    c[0] = fma(A[3], A[5], mul(A[4], n4));
    c[1] = fma(A[2], A[4], mul(n1, A[5]));
    c[2] = fma(A[1], A[4], mul(n2, A[3]));
    c[3] = fma(A[0], A[5], mul(A[2], n2));
    c[4] = fma(A[1], A[2], mul(n4, A[0]));
    c[5] = fma(A[0], A[3], mul(A[1], n1));
    return fma(A[0], c[0], fma(A[1], c[1], mul(A[2], c[2])));
}
__device__ __forceinline__ v2 dot3(v2 a0, v2 a1, v2 a2, const v2* v) {
    return fma(a0, v[0], fma(a1, v[1], mul(a2, v[2])));
}
__device__ __forceinline__ void symv(const v2* A, const v2* v, v2* o) {
    o[0] = dot3(A[0], A[1], A[2], v);
    o[1] = dot3(A[1], A[3], A[4], v);
    o[2] = dot3(A[2], A[4], A[5], v);
}
// C = A B of two commuting symmetric matrices
__device__ __forceinline__ void symm(const v2* A, const v2* B, v2* C) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j)
            C[sidx(i, j)] = fma(A[sidx(i, 0)], B[sidx(0, j)],
                                fma(A[sidx(i, 1)], B[sidx(1, j)],
                                    mul(A[sidx(i, 2)], B[sidx(2, j)])));
}

template <int K, bool RUS>
__device__ __forceinline__ void face_eval14_x2(const v2* Q, const float* D, float sigma_lim,
                                               float k_ws, float* Fn, v2& sig, v2& det) {
    constexpr int E1 = (K + 1) % 3, E2 = (K + 2) % 3;
    const v2 rho = Q[0];
    const v2* u = Q + 1;
    const v2* Pd = Q + 4;
    // ---- dimensionless state
    const v2 tr = add(add(Q[4], Q[7]), Q[9]), p = mul(tr, S(1.0f / 3.0f));
    const v2 ip = rcp(p), th = mul(p, rcp(rho)), rsq = rsqrt_(th), sq = mul(th, rsq);
    const v2 isc3 = mul(ip, rsq);
    v2 P[6], q[3], y[3];
#pragma unroll
    for (int n = 0; n < 6; ++n) P[n] = mul(Q[4 + n], ip);
#pragma unroll
    for (int n = 0; n < 3; ++n) q[n] = mul(Q[10 + n], isc3);
    const v2 nRs = mul(mul(Q[13], rho), mul(ip, neg(ip)));
    const v2 t = add(add(P[0], P[3]), P[5]);
    const v2 off = fma(P[1], P[1], fma(P[2], P[2], mul(P[4], P[4])));
    const v2 T2 = fma(P[0], P[0], fma(P[3], P[3], fma(P[5], P[5], add(off, off))));
    {
        v2 c[6];
        det = cofactors(P, c);
        const v2 id = rcp(det);
        symv(c, q, y);
#pragma unroll
        for (int n = 0; n < 3; ++n) y[n] = mul(y[n], id);
    }
    sig = sigma_root_x2(fma(t, t, fma(T2, S(2.0f), nRs)),
                        mul(mul(T2, S(8.0f)), dot3(q[0], q[1], q[2], y)), T2);
    const v2 sb = clamp_sigma_x2(sig, sigma_lim);
    const v2 rsb = rsqrt_(sb), isb = mul(rsb, rsb), ssb = mul(sb, rsb);
    FluxWeights w;
    {
        v2 lp, lm;
        lam_core_x2(P[sidx(K, K)], q[K], sqrt_(fma(q[E1], q[E1], mul(q[E2], q[E2]))), sb, isb, ssb,
                    lp, lm);
        const v2 ks = mul(sq, S(k_ws));
        w = flux_weights<RUS>(fma(lm, ks, u[K]), fma(lp, ks, u[K]));
    }
    // ---- closure slice along K: Qk = Q_Kij, Rk = R_Kijj, Sk = S_Kiijj
    v2 Qk[6], Rk[3], Sk;
    {
        v2 P2[6], P3[6], v[3], T[3], wv[3];
        symm(P, P, P2);
        symm(P2, P, P3);
        {
            v2 B[6], c[6];                               // B / 4 = (T2/2) P* + P*^3
            const v2 h2 = mul(T2, S(0.5f));
#pragma unroll
            for (int n = 0; n < 6; ++n) B[n] = fma(h2, P[n], P3[n]);
            const v2 iB = rcp(cofactors(B, c));          // v: 4 B^-1 q*
            symv(c, q, v);
#pragma unroll
            for (int n = 0; n < 3; ++n) v[n] = mul(v[n], iB);
        }
        symv(P, v, wv);
#pragma unroll
        for (int n = 0; n < 3; ++n) wv[n] = mul(wv[n], S(0.5f));     // 2 w
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = a; b < 3; ++b) {
                if (a == K && b == K) {
                    Qk[sidx(a, b)] = mul(mul(wv[K], P2[sidx(K, K)]), S(3.0f));
                } else if (a == K || b == K) {
                    const int o = a == K ? b : a;
                    Qk[sidx(a, b)] = fma(add(wv[K], wv[K]), P2[sidx(K, o)],
                                         mul(wv[o], P2[sidx(K, K)]));
                } else {
                    Qk[sidx(a, b)] = fma(wv[K], P2[sidx(a, b)],
                                         fma(wv[a], P2[sidx(K, b)], mul(wv[b], P2[sidx(K, a)])));
                }
            }
        symv(Qk, y, T);
        const v2 om2 = fma(sb, S(-2.0f), S(2.0f)), sc4 = mul(p, th);
#pragma unroll
        for (int a = 0; a < 3; ++a)
            Rk[a] = mul(sc4, fma(T[a], isb, fma(om2, P2[sidx(a, K)], mul(P[sidx(a, K)], t))));
        const v2 yQy = dot3(y[0], y[1], y[2], T);
        // row K of the W bracket over 4, against v
        const v2 tt = mul(t, t), trP3 = add(add(P3[0], P3[3]), P3[5]);
        const v2 c1 = fma(trP3, S(3.0f), mul(mul(t, S(0.5f)), sub(tt, T2)));
        const v2 c2 = fma(T2, S(3.5f), mul(tt, S(-1.5f))), c3 = mul(t, S(5.0f));
        v2 m[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const v2 P4 = fma(P2[sidx(K, 0)], P2[sidx(0, a)],
                              fma(P2[sidx(K, 1)], P2[sidx(1, a)],
                                  mul(P2[sidx(K, 2)], P2[sidx(2, a)])));
            m[a] = fma(c1, P[sidx(K, a)],
                       fma(c2, P2[sidx(K, a)], fma(c3, P3[sidx(K, a)], mul(P4, S(5.0f)))));
        }
        const v2 Wq = dot3(m[0], m[1], m[2], v);
        const v2 Ss = fma(yQy, mul(isb, isb),
                          fma(add(ssb, ssb), mul(t, q[K]), mul(sub(S(1.0f), ssb), Wq)));
        Sk = mul(Ss, mul(sc4, sq));
        const v2 sc3 = mul(p, sq);
#pragma unroll
        for (int n = 0; n < 6; ++n) Qk[n] = mul(Qk[n], sc3);
    }
    // ---- conserved state and flux u_K U + central part, field by field
    const v2 uK = u[K];
    const float *du = D + 1, *dP = D + 4, *dq = D + 10;
    v2 mo[3];
    float dmo[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        mo[i] = mul(rho, u[i]);
        dmo[i] = RUS ? djump(rho, D[0], u[i], du[i]) : jump(mo[i]);
    }
    Fn[0] = weigh<RUS>(w, mo[K], RUS ? D[0] : jump(rho));
#pragma unroll
    for (int i = 0; i < 3; ++i) Fn[1 + i] = weigh<RUS>(w, fma(uK, mo[i], Pd[sidx(i, K)]), dmo[i]);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
            const int n = sidx(i, j);
            const v2 Un = fma(mo[i], u[j], Pd[n]);
            const v2 c = i == j ? fma(add(u[i], u[i]), Pd[sidx(i, K)], Qk[n])
                                : fma(u[i], Pd[sidx(j, K)], fma(u[j], Pd[sidx(i, K)], Qk[n]));
            Fn[4 + n] = weigh<RUS>(w, fma(uK, Un, c),
                              RUS ? djump(mo[i], dmo[i], u[j], du[j]) + dP[n] : jump(Un));
        }
    const v2 u2 = dot3(u[0], u[1], u[2], u), ru2 = mul(rho, u2), e = add(ru2, tr);
    v2 Pu[3], Qu[3], Pq[3];
    symv(Pd, u, Pu);
    symv(Qk, u, Qu);
    const v2 gK = fma(Pu[K], S(2.0f), Q[10 + K]);
    float du2 = 0.0f, dru2 = 0.0f, dtr = 0.0f, dPu[3] = {0.0f, 0.0f, 0.0f};
    if (RUS) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            du2 = fmaf(u[i].x + u[i].y, du[i], du2);
#pragma unroll
            for (int j = 0; j < 3; ++j)
                dPu[i] += djump(Pd[sidx(i, j)], dP[sidx(i, j)], u[j], du[j]);
        }
        dru2 = djump(rho, D[0], u2, du2);
        dtr = dP[0] + dP[3] + dP[5];
    }
    float duPq = 0.0f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const v2 Un = fma(u[i], e, fma(Pu[i], S(2.0f), Q[10 + i]));
        const v2 c = fma(u[i], gK, fma(u2, Pd[sidx(i, K)], fma(Qu[i], S(2.0f), Rk[i])));
        Fn[10 + i] = weigh<RUS>(w, fma(uK, Un, c),
                           RUS ? djump(u[i], du[i], e, dru2 + dtr) + fmaf(2.0f, dPu[i], dq[i])
                               : jump(Un));
        Pq[i] = add(Pu[i], Q[10 + i]);
        Rk[i] = add(Qu[i], Rk[i]);
        if (RUS) duPq += djump(u[i], du[i], Pq[i], dPu[i] + dq[i]);
    }
    const v2 e2 = fma(tr, S(2.0f), ru2);
    const v2 U13 = fma(u2, e2, fma(dot3(u[0], u[1], u[2], Pq), S(4.0f), Q[13]));
    const v2 c13 = fma(add(u2, u2), gK, fma(dot3(u[0], u[1], u[2], Rk), S(4.0f), Sk));
    Fn[13] = weigh<RUS>(w, fma(uK, U13, c13),
                   RUS ? djump(u2, du2, e2, fmaf(2.0f, dtr, dru2)) + fmaf(4.0f, duPq, D[13])
                       : jump(U13));
}

}  // namespace x2
}  // namespace mxe
