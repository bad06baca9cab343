// jxf_adjoint.cuh -- hand-written reverse mode (vector-Jacobian products) of
// the single-phase, inviscid right-hand side of §3.2 (the differentiable
// solver of §6 with dt held fixed).
//
// R(U): W = prim(U) per cell; per face F = HLLC(recon(W-stencil));
// R_i = -sum_d (F_{i+1/2} - F_{i-1/2})/dx_d.  Given Rbar, the adjoint is
//   Fbar_f = (Rbar_f - Rbar_{f-1})/dx_d                  (transposed divergence)
//   (WLbar, WRbar) = HLLC^T Fbar, Sbar = recon^T (WLbar, WRbar) per face
//   Wbar_c = sum over the stencil slots that map to c    (atomic scatter)
//   Ubar_c = prim^T Wbar_c.
// Every branch (min/max of the wave speeds, sign(s*), the WENO weights'
// smooth dependence) is differentiated along the branch the forward pass
// takes.  Each face recomputes its forward intermediates.
#pragma once
#include "jxf_impl.cuh"

namespace jxf {

// --------------------------------------------------------------- WENO5 VJP --
// Reverse of one side of weno5_pair: value = centre + sum a_k e_k / sum a_k.
// Returns the adjoints of q_k and e_k (the centre's adjoint is vbar).  With
// omega the normalised weights, Delta = value - centre and
// g_k = vbar (e_k - Delta) / sum a (the adjoint of a_k):
//   Jiang-Shu, a_k = d_k/q_k^2:            qbar_k = -2 g_k a_k / q_k;
//   WENO5-Z, a_k = d_k (1 + tau/q_k), tau = |q_0 - q_2|:
//     qbar_k = -g_k d_k tau/q_k^2, taubar = sum_k g_k d_k/q_k,
//     qbar_0 += s taubar, qbar_2 -= s taubar with s = sign(q_0 - q_2)
//     (+1 at a tie, the branch the forward takes).
template <typename T>
__device__ __forceinline__ void weno5_side_vjp(T q0, T q1, T q2, T e0, T e1, T e2, T vbar, bool z,
                                               T &qb0, T &qb1, T &qb2, T &eb0, T &eb1, T &eb2) {
    const T r0 = rcp(q0), r1 = rcp(q1), r2 = rcp(q2);
    if (z) {
        const T dq = q0 - q2;
        const T tau = dq < T(0) ? -dq : dq;
        const T s = dq < T(0) ? T(-1) : T(1);
        const T w0 = T(0.1) * (T(1) + tau * r0), w1 = T(0.6) * (T(1) + tau * r1);
        const T w2 = T(0.3) * (T(1) + tau * r2);
        const T iw = rcp(w0 + w1 + w2);
        const T o0 = w0 * iw, o1 = w1 * iw, o2 = w2 * iw;
        const T delta = o0 * e0 + o1 * e1 + o2 * e2;
        eb0 = vbar * o0;
        eb1 = vbar * o1;
        eb2 = vbar * o2;
        const T g0 = vbar * (e0 - delta) * iw, g1 = vbar * (e1 - delta) * iw;
        const T g2 = vbar * (e2 - delta) * iw;
        qb0 = -g0 * T(0.1) * tau * r0 * r0;
        qb1 = -g1 * T(0.6) * tau * r1 * r1;
        qb2 = -g2 * T(0.3) * tau * r2 * r2;
        const T taub = g0 * T(0.1) * r0 + g1 * T(0.6) * r1 + g2 * T(0.3) * r2;
        qb0 += s * taub;
        qb2 -= s * taub;
        return;
    }
    const T w0 = T(0.1) * r0 * r0, w1 = T(0.6) * r1 * r1, w2 = T(0.3) * r2 * r2;
    const T iw = rcp(w0 + w1 + w2);
    const T o0 = w0 * iw, o1 = w1 * iw, o2 = w2 * iw;
    const T delta = o0 * e0 + o1 * e1 + o2 * e2;
    eb0 = vbar * o0;
    eb1 = vbar * o1;
    eb2 = vbar * o2;
    qb0 = vbar * T(-2) * o0 * (e0 - delta) * r0;
    qb1 = vbar * T(-2) * o1 * (e1 - delta) * r1;
    qb2 = vbar * T(-2) * o2 * (e2 - delta) * r2;
}

// Reverse of weno5_pair: accumulates into xb[0..5] the adjoint of the six
// cell values given the adjoints of the left and right face values.
template <typename T>
__device__ __forceinline__ void weno5_pair_vjp(const T (&x)[6], T eps, bool z, T vlb, T vrb,
                                               T (&xb)[6]) {
    const T D0 = x[1] - x[0], D1 = x[2] - x[1], D2 = x[3] - x[2];
    const T D3 = x[4] - x[3], D4 = x[5] - x[4];
    const T k13 = T(1.0408329997330663);
    const T a0 = (D1 - D0) * k13, a1 = (D2 - D1) * k13;
    const T a2 = (D3 - D2) * k13, a3 = (D4 - D3) * k13;
    const T c0 = a0 * a0 + eps, c1 = a1 * a1 + eps, c2 = a2 * a2 + eps, c3 = a3 * a3 + eps;
    const T sixth = T(1.0 / 6.0);
    T Db0 = 0, Db1 = 0, Db2 = 0, Db3 = 0, Db4 = 0;
    T ab0 = 0, ab1 = 0, ab2 = 0, ab3 = 0;
    {  // left
        const T h0 = T(1.5) * D1 - T(0.5) * D0, h1 = T(0.5) * (D1 + D2), h2 = T(0.5) * D3 - T(1.5) * D2;
        const T q0 = h0 * h0 + c0, q1 = h1 * h1 + c1, q2 = h2 * h2 + c2;
        const T e0 = (T(5) * D1 - T(2) * D0) * sixth, e1 = (D1 + T(2) * D2) * sixth;
        const T e2 = (T(4) * D2 - D3) * sixth;
        T qb0, qb1, qb2, eb0, eb1, eb2;
        weno5_side_vjp(q0, q1, q2, e0, e1, e2, vlb, z, qb0, qb1, qb2, eb0, eb1, eb2);
        xb[2] += vlb;
        // e
        Db1 += (T(5) * eb0 + eb1) * sixth;
        Db0 += T(-2) * eb0 * sixth;
        Db2 += (T(2) * eb1 + T(4) * eb2) * sixth;
        Db3 += -eb2 * sixth;
        // q = h^2 + a^2 + eps
        const T hb0 = T(2) * h0 * qb0, hb1 = T(2) * h1 * qb1, hb2 = T(2) * h2 * qb2;
        ab0 += T(2) * a0 * qb0;
        ab1 += T(2) * a1 * qb1;
        ab2 += T(2) * a2 * qb2;
        Db1 += T(1.5) * hb0 + T(0.5) * hb1;
        Db0 += T(-0.5) * hb0;
        Db2 += T(0.5) * hb1 - T(1.5) * hb2;
        Db3 += T(0.5) * hb2;
    }
    {  // right (mirrored)
        const T h0 = T(0.5) * D4 - T(1.5) * D3, h1 = T(0.5) * (D2 + D3), h2 = T(1.5) * D2 - T(0.5) * D1;
        const T q0 = h0 * h0 + c3, q1 = h1 * h1 + c2, q2 = h2 * h2 + c1;
        const T e0 = (T(2) * D4 - T(5) * D3) * sixth, e1 = -(D3 + T(2) * D2) * sixth;
        const T e2 = (D1 - T(4) * D2) * sixth;
        T qb0, qb1, qb2, eb0, eb1, eb2;
        weno5_side_vjp(q0, q1, q2, e0, e1, e2, vrb, z, qb0, qb1, qb2, eb0, eb1, eb2);
        xb[3] += vrb;
        Db4 += T(2) * eb0 * sixth;
        Db3 += (T(-5) * eb0 - eb1) * sixth;
        Db2 += (T(-2) * eb1 - T(4) * eb2) * sixth;
        Db1 += eb2 * sixth;
        const T hb0 = T(2) * h0 * qb0, hb1 = T(2) * h1 * qb1, hb2 = T(2) * h2 * qb2;
        ab3 += T(2) * a3 * qb0;
        ab2 += T(2) * a2 * qb1;
        ab1 += T(2) * a1 * qb2;
        Db4 += T(0.5) * hb0;
        Db3 += T(-1.5) * hb0 + T(0.5) * hb1;
        Db2 += T(0.5) * hb1 + T(1.5) * hb2;
        Db1 += T(-0.5) * hb2;
    }
    // a_k = k13 (D_{k+1} - D_k)
    Db1 += k13 * ab0;
    Db0 -= k13 * ab0;
    Db2 += k13 * ab1;
    Db1 -= k13 * ab1;
    Db3 += k13 * ab2;
    Db2 -= k13 * ab2;
    Db4 += k13 * ab3;
    Db3 -= k13 * ab3;
    // D_k = x_{k+1} - x_k
    xb[1] += Db0;
    xb[0] -= Db0;
    xb[2] += Db1;
    xb[1] -= Db1;
    xb[3] += Db2;
    xb[2] -= Db2;
    xb[4] += Db3;
    xb[3] -= Db3;
    xb[5] += Db4;
    xb[4] -= Db4;
}

// The derivatives of both values of a resolved double face by the differences,
// in float pairs (see the split correction of the forward sweep): with the
// lanes' D_0..D_3 (D_3 = swapped D_1), G = sum_k w_k e_k, e = (2 T_0, 0, T_1),
//   c_m = d(D_1 + 2 D_2 - G)/dD_m,
//   dG/dT_0 = 2 w_0, dG/dT_1 = w_2, dG/dQ_k = -2 w_k (e_k - G)/Q_k
// for Jiang-Shu weights; WENO5-Z (a_k = d_k (1 + tau/Q_k), tau = |Q_0 - Q_2|)
//   dG/dQ_k = -(e_k - G) d_k tau/(Q_k^2 sum a), dG/dtau = sum_k (e_k - G) d_k/(Q_k sum a).
// They multiply the adjoints, so an error of theirs is one relative to the
// result: pairs alone (2^-48) are not enough.  What is carried in pairs is their
// difference from the constants of the linear weights, (-0.2, 1.1, 2.4, -0.3),
// every term of which is a multiple of a third difference, told without
// cancellation:
//   Q_1 - Q_0 = T_0 ((H_0 + H_1) + 13/3 (A_0 + A_1)),
//   Q_1 - Q_2 = T_1 ((H_1 - H_2) - 13/3 (A_1 + A_2)),
//   w_k - d_k = d_k (y_k - s)/(1 + s), s = sum_k d_k y_k, with 1 + y_k the
//   weights before normalisation over that of k = 1 (Jiang-Shu), over d_k (Z);
// T itself comes from double differences.  Where max |T| is at most `bound`
// times sqrt(Q) (the smallest Q over the root of the largest) these terms are
// small enough; elsewhere, variable by variable, all is double.  Mean errors
// against quadruple precision over those of the all-double sweep, every variable,
// both modes and weights, 161 x 141 at Mach 0.001 to 0.3: waves of 50 cells and more
// 0.69-1.00, of 20 cells 0.73-1.00 (pairs without the linear part kept apart: up
// to 6.2; bounds of 1/4: up to 1.25 component-wise).  Step adjoint at 256^2
// (characteristic) 2.09 ms all double with a second forward reconstruction, 1.52
// with the forward sweep's face states and square roots from reciprocal square
// roots, 0.96 so (0.88 with the linear part in pairs as well).
constexpr float kSplitVjpComp = 1.f / 32.f, kSplitVjpChar = 1.f / 16.f;
__device__ __forceinline__ d2 drcp(d2 a) {  // 1/a
    const f2 r = rcp2(a.h), n = neg2(r);
    return {r, mul2(r, add2(fma2(n, a.h, bc2(1.f)), mul2(n, a.l)))};
}
__device__ __forceinline__ d2 bcd2(double x) {
    float h, l;
    split_double(x, h, l);
    return bcd(h, l);
}
__device__ __forceinline__ bool weno5_derivs_split(bool z, const Cst<float> &C, d2 D0, d2 D1, d2 D2, d2 T0, d2 T1,
                                                   float bound, d2 (&c)[4]) {
    const f2 two = bc2(2.f);
    const d2 D3 = swapd(D1);
    const d2 A0 = dsub(D1, D0), A1 = dsub(D2, D1), A2 = dsub(D3, D2);
    const d2 H0 = dadd(dscale(D1, two), A0), H1 = dadd(D1, D2), H2 = dsub(A2, dscale(D2, two));
    const f2 e4 = bc2(C.weno_eps4), e4l = bc2(C.weno_eps4l);
    const float k0 = (float)(13.0 / 3.0), k1 = (float)(13.0 / 3.0 - (double)k0);
    const d2 k13 = bcd(k0, k1);
    auto q = [&](d2 H, d2 A) {
        const d2 h = dsq(H), a = dmul(dsq(A), k13);
        f2 s, e, t, g;
        two_sum2(h.h, a.h, s, e);
        two_sum2(s, e4, t, g);
        return renorm({t, add2(add2(add2(e, g), e4l), add2(h.l, a.l))});
    };
    d2 Q0 = q(H0, A0), Q1 = q(H1, A1), Q2 = q(H2, A2);
    auto pow2 = [](float m) { return __uint_as_float(0x7F000000u - (__float_as_uint(m) & 0x7F800000u)); };
    const f2 sc = mk2(pow2(fmaxf(Q0.h.v.x, fmaxf(Q1.h.v.x, Q2.h.v.x))),
                      pow2(fmaxf(Q0.h.v.y, fmaxf(Q1.h.v.y, Q2.h.v.y))));
    Q0 = dscale(Q0, sc), Q1 = dscale(Q1, sc), Q2 = dscale(Q2, sc);
    {   // the largest Q is between 1 and 2 now
        auto small = [&](float t0, float t1, float q0, float q1, float q2, float s) {
            const float t = fmaxf(fabsf(t0), fabsf(t1)), qm = fminf(q0, fminf(q1, q2));
            return t * t * s <= (0.5f * bound * bound) * (qm * qm);
        };
        if (!(small(T0.h.v.x, T1.h.v.x, Q0.h.v.x, Q1.h.v.x, Q2.h.v.x, sc.v.x) &&
              small(T0.h.v.y, T1.h.v.y, Q0.h.v.y, Q1.h.v.y, Q2.h.v.y, sc.v.y)))
            return false;
    }
    const d2 r0 = renorm(drcp(Q0)), r1 = renorm(drcp(Q1)), r2 = renorm(drcp(Q2));
    // Q_1 - Q_0, Q_1 - Q_2
    const d2 m0 = renorm(dscale(dmul(T0, renorm(dadd(dadd(H0, H1), dmul(k13, renorm(dadd(A0, A1)))))), sc));
    const d2 m2 = renorm(dscale(dmul(T1, renorm(dsub(dsub(H1, H2), dmul(k13, renorm(dadd(A1, A2)))))), sc));
    d2 y0, y1 = bcd(0.f, 0.f), y2, tau = y1;
    f2 sg = bc2(0.f);
    if (z) {
        tau = renorm(dsub(m2, m0));  // Q_0 - Q_2
        sg = mk2(tau.h.v.x < 0.f ? -1.f : 1.f, tau.h.v.y < 0.f ? -1.f : 1.f);
        tau = dscale(tau, sg);
        y0 = renorm(dmul(tau, r0)), y1 = renorm(dmul(tau, r1)), y2 = renorm(dmul(tau, r2));
    } else {
        const d2 x0 = renorm(dmul(m0, r0)), x2 = renorm(dmul(m2, r2));
        y0 = renorm(dadd(dscale(x0, two), dsq(x0)));
        y2 = renorm(dadd(dscale(x2, two), dsq(x2)));
    }
    const d2 s10 = renorm(dadd(dadd(y0, dmulf(y1, 6.f)), dmulf(y2, 3.f)));  // 10 s
    const d2 ia = renorm(drcp(renorm(dadd(bcd(10.f, 0.f), s10))));          // 1/sum of (1, 6, 3) (1 + y)
    const float c0 = 0.1f, c1 = (float)(0.1 - (double)c0);
    const d2 ia1 = renorm(dmul(ia, bcd(c0, c1)));
    const d2 one = bcd(1.f, 0.f);
    const d2 w0 = renorm(dmul(renorm(dadd(one, y0)), ia)), w2 = renorm(dmulf(dmul(renorm(dadd(one, y2)), ia), 3.f));
    const d2 v0 = renorm(dmul(renorm(dsub(dmulf(y0, 10.f), s10)), ia1));  // w_0 - 0.1, w_2 - 0.3
    const d2 v2 = renorm(dmulf(dmul(renorm(dsub(dmulf(y2, 10.f), s10)), ia1), 3.f));
    const d2 e0 = dscale(T0, two);
    const d2 G = renorm(dadd(dmul(w0, e0), dmul(w2, T1)));
    const d2 x0 = renorm(dsub(e0, G)), x2 = renorm(dsub(T1, G));  // e_k - G; e_1 - G = -G
    // minus dG/dQ_k (of the unscaled Q_k)
    d2 g0, g1, g2;
    if (z) {
        const d2 u0 = renorm(dmul(dmul(x0, ia), r0)), u1 = renorm(dmulf(dmul(dmul(G, ia), r1), -6.f));
        const d2 u2 = renorm(dmulf(dmul(dmul(x2, ia), r2), 3.f));
        const d2 tb = dscale(renorm(dadd(dadd(u0, u1), u2)), sg);  // dG/dQ_0 through tau, -dG/dQ_2
        g0 = dsub(dmul(u0, y0), tb);
        g1 = dmul(u1, y1);
        g2 = dadd(dmul(u2, y2), tb);
    } else {
        const d2 w1 = renorm(dmulf(ia, 6.f));
        g0 = dscale(dmul(dmul(w0, x0), r0), two);
        g1 = dscale(dmul(dmul(w1, G), r1), bc2(-2.f));
        g2 = dscale(dmul(dmul(w2, x2), r2), two);
    }
    g0 = renorm(dscale(g0, sc)), g1 = renorm(dscale(g1, sc)), g2 = renorm(dscale(g2, sc));
    // through Q_k = H_k^2 + 13/3 A_k^2 (both minus their derivatives of G)
    const d2 h0 = dscale(dmul(H0, g0), two), h1 = dscale(dmul(H1, g1), two), h2 = dscale(dmul(H2, g2), two);
    const d2 kk = bcd(2.f * k0, 2.f * k1);
    const d2 t0 = dscale(v0, two);
    const d2 b0 = renorm(dadd(dmul(dmul(kk, A0), g0), t0));
    const d2 b1 = renorm(dsub(dadd(dmul(dmul(kk, A1), g1), v2), t0));
    const d2 b2 = renorm(dsub(dmul(dmul(kk, A2), g2), v2));
    c[0] = renorm(dscale(dadd(h0, b0), bc2(-1.f)));
    c[1] = renorm(dadd(dadd(dmulf(renorm(h0), 3.f), h1), dsub(b0, b1)));
    c[2] = renorm(dadd(dsub(h1, dmulf(renorm(h2), 3.f)), dsub(b1, b2)));
    c[3] = renorm(dadd(h2, b2));
    return true;
}

// What the derivatives of one variable are formed from: the lanes' differences
// (D_0, D_4), (D_1, D_3), (D_2, D_2) and third differences (T_0, T_2), (T_1, T_1).
struct SplitDiffs {
    d2 D[3], T0, T1;
};
template <class X> __device__ __forceinline__ SplitDiffs split_diffs(X x) {  // x(j): cell value j
    double D[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) D[k] = x(k + 1) - x(k);
    const double A0 = D[1] - D[0], A1 = D[2] - D[1], A2 = D[3] - D[2], A3 = D[4] - D[3];
    return {{lanes(D[0], D[4]), lanes(D[1], D[3]), bcd2(D[2])}, lanes(A1 - A0, A3 - A2), bcd2(A2 - A1)};
}

// xb += the adjoint of the six values from those of the face's two; false where
// the derivatives are not small enough beside the linear ones for pairs.
__device__ __forceinline__ bool weno5_apply_split(bool z, const Cst<float> &C, const SplitDiffs &s, float bound,
                                                  double vlb, double vrb, double (&xb)[6]) {
    d2 c[4];
    if (!weno5_derivs_split(z, C, s.D[0], s.D[1], s.D[2], s.T0, s.T1, bound, c)) return false;
    const double l = (1.0 / 6.0) * vlb, r = (-1.0 / 6.0) * vrb, lin[4] = {-0.2, 1.1, 2.4, -0.3};
    double Db[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        Db[k] = fma(l, lin[k] + (widen(c[k].h.v.x) + widen(c[k].l.v.x)), Db[k]);
        Db[4 - k] = fma(r, lin[k] + (widen(c[k].h.v.y) + widen(c[k].l.v.y)), Db[4 - k]);
    }
    xb[0] -= Db[0];
    xb[1] += Db[0] - Db[1];
    xb[2] += (Db[1] - Db[2]) + vlb;
    xb[3] += (Db[2] - Db[3]) + vrb;
    xb[4] += Db[3] - Db[4];
    xb[5] += Db[4];
    return true;
}

// ----------------------------------------------------- reconstruction VJP --
// Reverse of reconstruct() for the single-phase model: Sb[j][v] accumulates
// the adjoint of the six stencil primitives from the face-state adjoints.  WL,
// WR: the face states; split: the face took the split correction (double).
template <typename T, int NDIM, int d>
__device__ __forceinline__ void reconstruct_vjp(const Dev &P, const T (&S)[6][MAXV], const T *WL, const T *WR,
                                                bool split, const T *WLb, const T *WRb, T (&Sb)[6][MAXV]) {
    using V = Vars<JXF_SPM, NDIM>;
    constexpr int NV = V::NV, IE = V::IE, in = 1 + d;
    const T eps = cst<T>(P).weno_eps;
    const bool z = P.weno_z != 0;
    if (P.recon == JXF_WENO5JS_COMP) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const T x[6] = {S[0][v], S[1][v], S[2][v], S[3][v], S[4][v], S[5][v]};
            T xb[6] = {0, 0, 0, 0, 0, 0};
            bool done = false;
            if constexpr (std::is_same<T, double>::value)
                done = split && weno5_apply_split(z, cst<float>(P), split_diffs([&](int j) { return x[j]; }), kSplitVjpComp,
                                                   WLb[v], WRb[v], xb);
            if (!done) weno5_pair_vjp(x, eps, z, WLb[v], WRb[v], xb);
#pragma unroll
            for (int j = 0; j < 6; ++j) Sb[j][v] += xb[j];
        }
        return;
    }
    // forward: frozen state and projection
    const Cst<T> &C = cst<T>(P);
    T Wb[MAXV];
#pragma unroll
    for (int v = 0; v < NV; ++v) Wb[v] = T(0.5) * (S[2][v] + S[3][v]);
    const T rho = Wb[0];
    const T rc2 = C.gamma0 * (Wb[IE] + C.pinf0);
    // one reciprocal square root t = 1/(rho c) gives c, 1/c, 1/rho and 1/(rho c^2)
    const T t = rsq(rho * rc2);
    const T cb = rc2 * t, icb = rho * t, irc2 = icb * t, irho = cb * t;
    const T xcs = cb * cb;
    const T h_c = T(0.5) * icb;
    const T h_rc2 = T(0.5) * irc2;
    const T ent = Wb[0] * irc2;
    // reverse of the back-projection o = K q (both sides)
    T qLb[MAXV], qRb[MAXV];
    T Wb0b = 0, cbb = 0, rc2b = 0;
    const T *ob[2] = {WLb, WRb};
    const T *Ws[2] = {WL, WR};
    T *qbs[2] = {qLb, qRb};
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const T *o = ob[s];
        T *qb = qbs[s];
        // of the face state o = K q: q_in + q_IE = p/(rho c^2), q_IE - q_in = u/c
        const T qsum = Ws[s][IE] * irc2, qdif = Ws[s][in] * icb;
#pragma unroll
        for (int v = 0; v < NV; ++v) qb[v] = o[v];
        // o[0] = Wb0 q[in] + q[0] + Wb0 q[IE]
        qb[0] = o[0];
        qb[in] = o[0] * Wb[0];
        qb[IE] = o[0] * Wb[0];
        Wb0b += o[0] * qsum;
        // o[in] = cb (q[IE] - q[in])
        qb[IE] += o[in] * cb;
        qb[in] -= o[in] * cb;
        cbb += o[in] * qdif;
        // o[IE] = rc2 (q[in] + q[IE])
        qb[in] += o[IE] * rc2;
        qb[IE] += o[IE] * rc2;
        rc2b += o[IE] * qsum;
    }
    // reverse of the WENO reconstructions of q = K^{-1} S
    T qb[MAXV][6];
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int j = 0; j < 6; ++j) qb[v][j] = T(0);
    bool done[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) done[v] = false;
    if constexpr (std::is_same<T, double>::value) {
        if (split) {
            const Cst<float> &C32 = cst<float>(P);
            SplitDiffs s[NV];  // of the primitives, then of q
#pragma unroll
            for (int v = 0; v < NV; ++v) s[v] = split_diffs([&](int j) { return S[j][v]; });
            const d2 e = bcd2(ent), hc = bcd2(h_c), hr = bcd2(h_rc2);
            auto project = [&](d2 &x0, d2 &xi, d2 &xe) {
                const d2 x = dmul(hc, xi), y = dmul(hr, xe);
                x0 = renorm(dsub(x0, dmul(e, xe)));
                xe = renorm(dadd(y, x));
                xi = renorm(dsub(y, x));
            };
#pragma unroll
            for (int k = 0; k < 3; ++k) project(s[0].D[k], s[in].D[k], s[IE].D[k]);
            project(s[0].T0, s[in].T0, s[IE].T0);
            project(s[0].T1, s[in].T1, s[IE].T1);
#pragma unroll
            for (int v = 0; v < NV; ++v) done[v] = weno5_apply_split(z, C32, s[v], kSplitVjpChar, qLb[v], qRb[v], qb[v]);
        }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        if (done[v]) continue;
        T q[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            if (v == 0) q[j] = S[j][0] - ent * S[j][IE];
            else if (v == in) q[j] = fma(h_rc2, S[j][IE], -(h_c * S[j][in]));  // as in the forward sweep
            else if (v == IE) q[j] = fma(h_rc2, S[j][IE], h_c * S[j][in]);
            else q[j] = S[j][v];
        }
        weno5_pair_vjp(q, eps, z, qLb[v], qRb[v], qb[v]);
    }
    // reverse of the projection q = K^{-1} S
    T entb = 0, h_cb = 0, h_rc2b = 0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
#pragma unroll
        for (int v = 0; v < NV; ++v)
            if (v != 0 && v != in && v != IE) Sb[j][v] += qb[v][j];
        // q0 = S0 - ent S_IE
        Sb[j][0] += qb[0][j];
        Sb[j][IE] -= qb[0][j] * ent;
        entb -= qb[0][j] * S[j][IE];
        // q_in = -h_c S_in + h_rc2 S_IE ; q_IE = h_c S_in + h_rc2 S_IE
        Sb[j][in] += (qb[IE][j] - qb[in][j]) * h_c;
        Sb[j][IE] += (qb[IE][j] + qb[in][j]) * h_rc2;
        h_cb += (qb[IE][j] - qb[in][j]) * S[j][in];
        h_rc2b += (qb[IE][j] + qb[in][j]) * S[j][IE];
    }
    // frozen-state intermediates
    T irc2b = entb * Wb[0] + T(0.5) * h_rc2b;
    Wb0b += entb * irc2;
    cbb -= h_cb * h_c * icb;
    const T xb = cbb * (T(0.5) * icb);
    rc2b += xb * irho;
    Wb0b -= xb * xcs * irho;  // rho = Wb[0]
    rc2b -= irc2b * irc2 * irc2;
    T Wbb[MAXV];
#pragma unroll
    for (int v = 0; v < NV; ++v) Wbb[v] = T(0);
    Wbb[0] = Wb0b;
    Wbb[IE] += rc2b * C.gamma0;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        Sb[2][v] += T(0.5) * Wbb[v];
        Sb[3][v] += T(0.5) * Wbb[v];
    }
}

// ---------------------------------------------------------------- HLLC VJP --
// Reverse of hllc() for the single-phase model: from the adjoint of the face
// flux (Fb, uhb ignored: inviscid single phase has no face-velocity source)
// to the adjoints of the two primitive face states.
template <typename T, int NDIM, int d>
__device__ __forceinline__ void hllc_vjp(const Dev &P, const T *WL, const T *WR, const T *Fb,
                                         T *WLb, T *WRb) {
    using V = Vars<JXF_SPM, NDIM>;
    constexpr int NV = V::NV, IE = V::IE, in = 1 + d;
    const Cst<T> &C = cst<T>(P);
    const T g = C.gamma0, pinf = C.pinf0, A = C.A1;  // A = 1/(gamma-1)
    // ---- forward
    const T rhoL = WL[0], rhoR = WR[0], uL = WL[in], uR = WR[in], pL = WL[IE], pR = WR[IE];
    // c, 1/c and sqrt(rho), 1/sqrt(rho), 1/rho from reciprocal square roots
    const T isL = rsq(rhoL), isR = rsq(rhoR);
    const T irhoL = isL * isL, irhoR = isR * isR;
    const T srL = rhoL * isL, srR = rhoR * isR;
    const T c2L = g * (pL + pinf) * irhoL, c2R = g * (pR + pinf) * irhoR;
    const T icL = rsq(c2L), icR = rsq(c2R);
    const T cL = c2L * icL, cR = c2R * icR;
    const T is = rcp(srL + srR);
    const T S2 = srL * uL + srR * uR;
    const T ubar = S2 * is;
    const T du = uR - uL;
    const T S1 = srL * c2L + srR * c2R;
    const T c2bar = S1 * is + T(0.5) * srL * srR * is * is * du * du;
    const T icbar = rsq(c2bar);
    const T cbar = c2bar * icbar;
    const bool Lfirst = !((uL - cL) < (ubar - cbar));  // tmin picks uL-cL when smaller
    const T sL = Lfirst ? ubar - cbar : uL - cL;
    const bool Rfirst = !((uR + cR) > (ubar + cbar));
    const T sR = Rfirst ? ubar + cbar : uR + cR;
    const T mL = rhoL * (sL - uL), mR = rhoR * (sR - uR);
    const T num = pR - pL + mL * uL - mR * uR, den2 = mL - mR;
    const T iden2 = rcp(den2);
    const T sstar = num * iden2;
    const T sm = sL < T(0) ? sL : T(0), sp = sR > T(0) ? sR : T(0);
    const int first = sstar < T(0) ? 1 : 0, last = sstar > T(0) ? 0 : 1;
    const T wgt = first == last ? T(1) : T(0.5);
    // ---- reverse
    T sLb = 0, sRb = 0, smb = 0, spb = 0, ssb = 0;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        WLb[v] = T(0);
        WRb[v] = T(0);
    }
#pragma unroll 1
    for (int side = first; side <= last; ++side) {
        const bool R = side == 1;
        T W[MAXV], Wbk[MAXV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            W[v] = R ? WR[v] : WL[v];
            Wbk[v] = T(0);
        }
        const T sK = R ? sR : sL, sPM = R ? sp : sm;
        const T rho = W[0], u = W[in], p = W[IE];
        T uu = T(0);
#pragma unroll
        for (int e = 0; e < NDIM; ++e) uu += W[1 + e] * W[1 + e];
        const T E = (p + C.gpinf0) * A + T(0.5) * rho * uu;
        T U[MAXV];
        U[0] = rho;
#pragma unroll
        for (int e = 0; e < NDIM; ++e) U[1 + e] = rho * W[1 + e];
        U[IE] = E;
        const T su = sK - u, den = sK - sstar;
        const T isu = rcp(su), iden = rcp(den);
        const T fac = su * iden;
        const T B = rho * sstar + p * isu;
        const T Aterm = E + (sstar - u) * B;
        T Us[MAXV];
        Us[0] = fac * rho;
#pragma unroll
        for (int e = 0; e < NDIM; ++e) Us[1 + e] = fac * (rho * W[1 + e]);
        Us[in] = fac * (rho * sstar);
        Us[IE] = fac * Aterm;
        // F = wgt (Fp + sPM (Us - U));  Fp: mass rho u, momentum U_e u (+p), energy u (E+p)
        T Fpb[MAXV], Usb[MAXV], Ub[MAXV];
        T sPMb = T(0);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const T fb = wgt * Fb[v];
            Fpb[v] = fb;
            Usb[v] = sPM * fb;
            Ub[v] = -sPM * fb;
            sPMb += fb * (Us[v] - U[v]);
        }
        T ub = T(0), pb = T(0), rhob = T(0), Eb = T(0), facb = T(0), ssk = T(0);
        // physical flux
        Ub[0] += Fpb[0] * u;
        ub += Fpb[0] * U[0];
#pragma unroll
        for (int e = 0; e < NDIM; ++e) {
            Ub[1 + e] += Fpb[1 + e] * u;
            ub += Fpb[1 + e] * U[1 + e];
        }
        pb += Fpb[in];
        ub += Fpb[IE] * (E + p);
        Eb += Fpb[IE] * u;
        pb += Fpb[IE] * u;
        // star state
        facb += Usb[0] * rho;
        rhob += Usb[0] * fac;
#pragma unroll
        for (int e = 0; e < NDIM; ++e) {
            if (e == d) continue;
            facb += Usb[1 + e] * rho * W[1 + e];
            rhob += Usb[1 + e] * fac * W[1 + e];
            Wbk[1 + e] += Usb[1 + e] * fac * rho;
        }
        facb += Usb[in] * rho * sstar;
        rhob += Usb[in] * fac * sstar;
        ssk += Usb[in] * fac * rho;
        facb += Usb[IE] * Aterm;
        const T Ab = Usb[IE] * fac;
        Eb += Ab;
        ssk += Ab * B;
        ub -= Ab * B;
        const T Bb = Ab * (sstar - u);
        rhob += Bb * sstar;
        ssk += Bb * rho;
        pb += Bb * isu;
        T sub = -Bb * p * (isu * isu);
        // fac = su / den
        sub += facb * iden;
        const T denb = -facb * fac * iden;
        T sKb = denb + sub;
        ssk -= denb;
        ub -= sub;
        // U = prim2cons(W)
        rhob += Ub[0];
#pragma unroll
        for (int e = 0; e < NDIM; ++e) {
            rhob += Ub[1 + e] * W[1 + e];
            Wbk[1 + e] += Ub[1 + e] * rho;
        }
        Eb += Ub[IE];
        rhob += Eb * T(0.5) * uu;
#pragma unroll
        for (int e = 0; e < NDIM; ++e) Wbk[1 + e] += Eb * rho * W[1 + e];
        pb += Eb * A;
        Wbk[0] += rhob;
        Wbk[in] += ub;
        Wbk[IE] += pb;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            if (R) WRb[v] += Wbk[v];
            else WLb[v] += Wbk[v];
        }
        if (R) {
            sRb += sKb;
            spb += sPMb;
        } else {
            sLb += sKb;
            smb += sPMb;
        }
        ssb += ssk;
    }
    // sm = min(0, sL), sp = max(0, sR)
    if (sL < T(0)) sLb += smb;
    if (sR > T(0)) sRb += spb;
    // s* = num / den2
    const T numb = ssb * iden2;
    const T den2b = -ssb * sstar * iden2;
    T mLb = numb * uL + den2b, mRb = -numb * uR - den2b;
    T pLb = -numb, pRb = numb, uLb = numb * mL, uRb = -numb * mR, rhoLb = 0, rhoRb = 0;
    // m = rho (s - u)
    rhoLb += mLb * (sL - uL);
    sLb += mLb * rhoL;
    uLb -= mLb * rhoL;
    rhoRb += mRb * (sR - uR);
    sRb += mRb * rhoR;
    uRb -= mRb * rhoR;
    // wave speeds
    T ubarb = 0, cbarb = 0, cLb = 0, cRb = 0;
    if (Lfirst) {
        ubarb += sLb;
        cbarb -= sLb;
    } else {
        uLb += sLb;
        cLb -= sLb;
    }
    if (Rfirst) {
        ubarb += sRb;
        cbarb += sRb;
    } else {
        uRb += sRb;
        cRb += sRb;
    }
    const T c2barb = cbarb * (T(0.5) * icbar);
    // c2bar = S1 is + 0.5 srL srR is^2 du^2
    const T S1b = c2barb * is;
    T isb = c2barb * S1 + c2barb * srL * srR * is * du * du;
    T srLb = c2barb * T(0.5) * srR * is * is * du * du;
    T srRb = c2barb * T(0.5) * srL * is * is * du * du;
    const T dub = c2barb * srL * srR * is * is * du;
    uRb += dub;
    uLb -= dub;
    T c2Lb = S1b * srL, c2Rb = S1b * srR;
    srLb += S1b * c2L;
    srRb += S1b * c2R;
    // ubar = S2 is
    const T S2b = ubarb * is;
    isb += ubarb * S2;
    srLb += S2b * uL;
    uLb += S2b * srL;
    srRb += S2b * uR;
    uRb += S2b * srR;
    // is = 1/(srL + srR)
    const T sumb = -isb * is * is;
    srLb += sumb;
    srRb += sumb;
    rhoLb += srLb * (T(0.5) * isL);
    rhoRb += srRb * (T(0.5) * isR);
    c2Lb += cLb * (T(0.5) * icL);
    c2Rb += cRb * (T(0.5) * icR);
    // c2 = g (p + pinf) / rho
    pLb += c2Lb * g * irhoL;
    rhoLb -= c2Lb * c2L * irhoL;
    pRb += c2Rb * g * irhoR;
    rhoRb -= c2Rb * c2R * irhoR;
    WLb[0] += rhoLb;
    WLb[in] += uLb;
    WLb[IE] += pLb;
    WRb[0] += rhoRb;
    WRb[in] += uRb;
    WRb[IE] += pRb;
}

// Start of axis d's section of the stencil-slot adjoints: the axes' sections
// ([slot][variable][face] each) follow one another.
__host__ __device__ inline size_t sbar_offset(const Dev &P, int ndim, int d, int nv) {
    size_t off = 0;
    for (int e = 0; e < d && e < ndim; ++e) {
        size_t nf = 1;
        for (int k = 0; k < 3; ++k) nf *= (size_t)(P.n[k] + (k == e ? 1 : 0));
        off += 6 * (size_t)nv * nf;
    }
    return off;
}

// ----------------------------------------------------------- k_flux_vjp ----
// One thread per face of axis d: Fbar from Rbar (transposed divergence),
// forward recomputation, reverse through HLLC and the reconstruction; the
// adjoints of the six stencil cells go to the face's slots of P.Sbar
// ([slot j][variable][face], mirrored slots with the normal velocity flipped
// back), and k_gather_vjp adds them to Wbar cell by cell in a fixed order --
// no atomics, so reverse mode gives the same bits on every run.
template <typename T, int NDIM, int d>
__global__ void __launch_bounds__(kFluxThreads) k_flux_vjp(const Dev P) {
    using V = Vars<JXF_SPM, NDIM>;
    constexpr int NV = V::NV;
    int m[3] = {P.n[0], P.n[1], P.n[2]};
    m[d] += 1;
    const long long nface = (long long)m[0] * m[1] * m[2];
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= nface) return;
    const unsigned gu = (unsigned)g;
    const unsigned q0 = P.fd_face[d][0].div(gu);
    const unsigned q1 = P.fd_face[d][1].div(q0);
    int c[3] = {(int)(gu - q0 * (unsigned)m[0]), (int)(q0 - q1 * (unsigned)m[1]), (int)q1};
    const int sd = d == 0 ? 1 : (d == 1 ? P.n[0] : P.n[0] * P.n[1]);
    const int base = ((c[2] * P.n[1] + c[1]) * P.n[0] + c[0]) - c[d] * sd;
    const size_t nc = (size_t)P.ncell;
    // Fbar_f = (Rbar_f - Rbar_{f-1}) / dx_d, cells outside the line contribute 0
    const T *Rb = static_cast<const T *>(P.Rbar);
    const T idx_d = cst<T>(P).inv_dx[d];
    T Fb[MAXV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const T right = c[d] < P.n[d] ? Rb[v * nc + chk_cell(P, base + c[d] * sd)] : T(0);
        const T left = c[d] > 0 ? Rb[v * nc + chk_cell(P, base + (c[d] - 1) * sd)] : T(0);
        Fb[v] = (right - left) * idx_d;
    }
    int idx[6];
    unsigned mir = 0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        int mj = 0;
        const int cj = map_axis(c[d] + j - 3, P.n[d], P.bc[d][0], P.bc[d][1], mj, 1);
        idx[j] = chk_cell(P, base + cj * sd);
        mir |= (unsigned)mj << j;
    }
    const T *W = static_cast<const T *>(P.W);
    T S[6][MAXV];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
#pragma unroll
        for (int v = 0; v < NV; ++v) S[j][v] = __ldg(W + v * nc + idx[j]);
        if ((mir >> j) & 1u) S[j][1 + d] = -S[j][1 + d];
    }
    T WL[MAXV], WR[MAXV];
    const int how = reconstruct<T, JXF_SPM, NDIM, d, 0, FACE_TRY>(P, S, WL, WR);  // WENO5: no reverse mode for TENO6-A
    T WLb[MAXV], WRb[MAXV];
    hllc_vjp<T, NDIM, d>(P, WL, WR, Fb, WLb, WRb);
    T Sb[6][MAXV];
#pragma unroll
    for (int j = 0; j < 6; ++j)
#pragma unroll
        for (int v = 0; v < NV; ++v) Sb[j][v] = T(0);
    reconstruct_vjp<T, NDIM, d>(P, S, WL, WR, how == FACE_SPLIT, WLb, WRb, Sb);
    T *Sbar = static_cast<T *>(P.Sbar) + sbar_offset(P, NDIM, d, NV);
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        if ((mir >> j) & 1u) Sb[j][1 + d] = -Sb[j][1 + d];
#pragma unroll
        for (int v = 0; v < NV; ++v) Sbar[((size_t)j * NV + v) * (size_t)nface + (size_t)g] = Sb[j][v];
    }
}

// Wbar of every cell = the sum of the stencil-slot adjoints of the faces
// whose stencils reach it, axis by axis (one thread per cell, after every axis's k_flux_vjp).
// Face f (between cells f-1 and f) holds slot j = cell f-3+j mapped through
// the boundary conditions; away from the ends of the line that is cell
// f-3+j itself, so cell i collects slot j of face i+3-j for j = 0..5; within
// three cells of an end every face near either end and near the cell is
// tested against the map.  The order of the additions is fixed, so the
// result is reproducible.
template <typename T, int NDIM, int d>
__device__ __forceinline__ void gather_axis(const Dev &P, const int (&c)[3], T *acc) {
    constexpr int NV = Vars<JXF_SPM, NDIM>::NV;
    int m[3] = {P.n[0], P.n[1], P.n[2]};
    m[d] += 1;
    const size_t nface = (size_t)m[0] * m[1] * m[2];
    const int n = P.n[d], ci = c[d];
    const int fs = d == 0 ? 1 : (d == 1 ? m[0] : m[0] * m[1]);  // face stride along d
    const int f0 = (c[2] * m[1] + c[1]) * m[0] + c[0] - ci * fs;  // face 0 of the cell's line
    const T *Sbar = static_cast<const T *>(P.Sbar) + sbar_offset(P, NDIM, d, NV);
    // slots hold the adjoint of the mapped cell (mirror flips already applied)
    auto take = [&](int f, int j) {
        const int g = chk_face(P, (long long)f0 + (long long)f * fs, (long long)nface);
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] += Sbar[((size_t)j * NV + v) * nface + (size_t)g];
    };
    if (ci >= 3 && ci <= n - 4) {
#pragma unroll
        for (int j = 0; j < 6; ++j) take(ci + 3 - j, j);
        return;
    }
    // faces within 7 of either end, then those within 3 of the cell
    const int e1 = min(n, 7), s2 = max(e1 + 1, n - 7);
    for (int part = 0; part < 3; ++part) {
        const int lo = part == 0 ? 0 : (part == 1 ? s2 : max(0, ci - 2));
        const int hi = part == 0 ? e1 : (part == 1 ? n : min(n, ci + 3));
        for (int f = lo; f <= hi; ++f) {
            if (part == 2 && (f <= e1 || f >= s2)) continue;
            for (int j = 0; j < 6; ++j) {
                int mj = 0;
                if (map_axis(f + j - 3, n, P.bc[d][0], P.bc[d][1], mj, 1) == ci) take(f, j);
            }
        }
    }
}

template <typename T, int NDIM>
__global__ void __launch_bounds__(kCellThreads) k_gather_vjp(const Dev P) {
    constexpr int NV = Vars<JXF_SPM, NDIM>::NV;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.ncell) return;
    const unsigned iu = (unsigned)i;
    const unsigned qy = P.fd_cell[0].div(iu), qz = P.fd_cell[1].div(qy);
    const int c[3] = {(int)(iu - qy * (unsigned)P.n[0]), (int)(qy - qz * (unsigned)P.n[1]), (int)qz};
    T *Wb = static_cast<T *>(P.Wbar);  // written here only: no clearing needed
    const size_t nc = (size_t)P.ncell;
    T w[MAXV];
#pragma unroll
    for (int v = 0; v < NV; ++v) w[v] = T(0);
    gather_axis<T, NDIM, 0>(P, c, w);
    if constexpr (NDIM > 1) gather_axis<T, NDIM, 1>(P, c, w);
    if constexpr (NDIM > 2) gather_axis<T, NDIM, 2>(P, c, w);
#pragma unroll
    for (int v = 0; v < NV; ++v) Wb[v * nc + (size_t)i] = w[v];
}

// Ubar = (dW/dU)^T Wbar per cell (§2.1 state vectors, ideal / stiffened gas).
template <typename T, int NDIM>
__global__ void __launch_bounds__(kCellThreads) k_prim_vjp(const Dev P) {
    using V = Vars<JXF_SPM, NDIM>;
    constexpr int NV = V::NV, IE = V::IE;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.ncell) return;
    const T *U = static_cast<const T *>(P.Us);
    const T *Wb = static_cast<const T *>(P.Wbar);
    T *Ub = static_cast<T *>(P.Ubar);
    const T gm1 = cst<T>(P).gm1_0;
    const T rho = U[i];
    const T ir = rcp(rho);
    T u[3], wb[MAXV];
#pragma unroll
    for (int v = 0; v < NV; ++v) wb[v] = Wb[v * P.ncell + i];
    T uu = T(0);
#pragma unroll
    for (int e = 0; e < NDIM; ++e) {
        u[e] = U[(1 + e) * P.ncell + i] * ir;
        uu += u[e] * u[e];
    }
    // p = (gamma-1)(E - 1/2 sum m_e u_e) - gamma pinf
    T rb = wb[0] + wb[IE] * gm1 * T(0.5) * uu;
#pragma unroll
    for (int e = 0; e < NDIM; ++e) {
        rb -= wb[1 + e] * u[e] * ir;
        Ub[(1 + e) * P.ncell + i] = wb[1 + e] * ir - wb[IE] * gm1 * u[e];
    }
    Ub[i] = rb;
    Ub[IE * P.ncell + i] = wb[IE] * gm1;
}

// out = a x + b y + c z (elementwise over n values; y, z may be null).
template <typename T>
__global__ void k_axpbypcz(T *out, long long n, double a, const T *x, double b, const T *y, double c,
                           const T *z) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    T s = T(a) * x[k];
    if (y) s += T(b) * y[k];
    if (z) s += T(c) * z[k];
    out[k] = s;
}

}  // namespace jxf
