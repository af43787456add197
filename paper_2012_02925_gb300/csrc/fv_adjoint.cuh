// Reverse-mode (vector-Jacobian) form of one face of the residual.
//
// The forward face is the one of fv_face.cuh: MUSCL reconstruction with
// limiter, Eq. (flux) of Section 7.2, and Roe's flux times the face area
// (Section 2).  Given the cotangent of the face flux, roe_vjp returns the
// cotangents of the two face states; lim_derivatives and prim_bwd transpose
// the limiter and the primitive recovery (Section 2), once per cell.
//
// Written once for an arithmetic type T (fv_arith.cuh): binary64, or
// double-float on the FP32 pipe (~48-bit significand; GB300's FP64 unit runs
// at 1/64 of the binary32 rate, and the sweep costs ~3 forward faces).
//
// The paper has no adjoint; this is the discrete adjoint of its residual.
#pragma once
#include "fv_arith.cuh"

// method parameters (binary64, from the handle)
struct AdjParams {
  double gm1, g_gm1;       // gamma - 1, gamma / (gamma - 1)
  double e4km, e4kp, e2;   // eps/4 (1 - kappa), eps/4 (1 + kappa), eps/2
  double harten, va_d2;
  int limiter, fix_all;
};

// the same in the arithmetic type, with the constants the sweep uses
template <class T>
struct AdjC {
  T gm1, g_gm1, e4km, e4kp, e2, harten, va_d2, half, one, two;
  int limiter, fix_all;
  bool fix;
};

// On the host: taken by every thread (one per face or cell), the conversions
// held the FP64 unit for part of the sweeps' time (96^3, four stages and their gradient 6.51 -> 6.28 ms)
template <class T>
inline AdjC<T> adj_consts(const AdjParams& P) {
  using S = Sc<T>;
  AdjC<T> c;
  c.gm1 = S::c(P.gm1);
  c.g_gm1 = S::c(P.g_gm1);
  c.e4km = S::c(P.e4km);
  c.e4kp = S::c(P.e4kp);
  c.e2 = S::c(P.e2);
  c.harten = S::c(P.harten);
  c.va_d2 = S::c(P.va_d2);
  c.half = S::c(0.5);
  c.one = S::c(1.0);
  c.two = S::c(2.0);
  c.limiter = P.limiter;
  c.fix_all = P.fix_all;
  c.fix = P.harten > 0.0;
  return c;
}

// limited difference phi(a, b) = Psi(a/b) b
template <class T>
__device__ __forceinline__ T lim_value(const AdjC<T>& P, T a, T b) {
  using S = Sc<T>;
  if (P.limiter == 0) return b;
  const T ab = a * b, s = a + b;
  // van Leer: 2ab/(a+b) when ab > 0, else 0
  if (P.limiter == 1) return S::pos(ab) ? S::twice(S::div(ab, s)) : S::c(0.0);
  // van Albada product form: ab (a + b) / (a^2 + b^2 + delta^2)
  return S::div(ab * s, S::dot2(a, a, b, b) + P.va_d2);
}

// its partial derivatives, for the two limiters that are symmetric in a and b
template <class T>
__device__ __forceinline__ void lim_derivatives(const AdjC<T>& P, T a, T b, T& da, T& db) {
  using S = Sc<T>;
  const T ab = a * b, s = a + b;
  if (P.limiter == 1) {
    if (!S::pos(ab)) { da = S::c(0.0); db = S::c(0.0); return; }
    const T is = S::rcp(s), x = a * is, y = b * is;
    da = S::twice(y * y);
    db = S::twice(x * x);
    return;
  }
  const T iD = S::rcp(S::dot2(a, a, b, b) + P.va_d2);
  const T f2 = S::twice(ab * s * iD);
  // (2ab + b^2 - 2 f a) / D and (a^2 + 2ab - 2 f b) / D, f the limited difference
  da = (S::dot2(b, s, a, b) - f2 * a) * iD;
  db = (S::dot2(a, s, a, b) - f2 * b) * iD;
}

template <class T>
struct PrimFwd {
  T r, u, v, w, p, ri, k;
};

template <class T>
__device__ __forceinline__ PrimFwd<T> prim_fwd(const AdjC<T>& P, const T q[5]) {
  using S = Sc<T>;
  PrimFwd<T> s;
  s.r = q[0];
  s.ri = S::rcp(q[0]);
  s.u = q[1] * s.ri;
  s.v = q[2] * s.ri;
  s.w = q[3] * s.ri;
  s.k = s.u * s.u + s.v * s.v + s.w * s.w;
  s.p = P.gm1 * (q[4] - S::halve(q[0] * s.k));
  return s;
}

// qbar = (dV/dq)^T Vbar for V = (rho, u, v, w, p), from the primitives
// alone (rho u = r u etc.), so the conserved inputs need not stay live
template <class T>
__device__ __forceinline__ void prim_bwd(T gm1, const PrimFwd<T>& s, const T Vb[5], T qb[5]) {
  using S = Sc<T>;
  const T pb = gm1 * Vb[4];
  const T gpb = s.r * pb;
  const T ub = Vb[1] - gpb * s.u;
  const T vb = Vb[2] - gpb * s.v;
  const T wb = Vb[3] - gpb * s.w;
  qb[4] = pb;
  qb[1] = ub * s.ri;
  qb[2] = vb * s.ri;
  qb[3] = wb * s.ri;
  // d(1/rho)/d rho = -1/rho^2 against ub rho u + vb rho v + wb rho w
  qb[0] = (Vb[0] - S::halve(s.k * pb)) - S::dot3(ub, s.u, vb, s.v, wb, s.w) * s.ri;
}

template <class T>
__device__ __forceinline__ T fix_fwd(const AdjC<T>& P, T l, T d, bool on, T& dl, T& dd) {
  using S = Sc<T>;
  if (on && S::lt_nonneg(l, d)) {
    const T id = S::rcp(d);
    dl = l * id;
    dd = P.half - S::halve(dl * dl);
    return S::halve((l * l + d * d) * id);
  }
  dl = P.one; dd = S::c(0.0);
  return l;
}

// sign of x as +-1 (x = 0 counts as positive)
template <class T>
__device__ __forceinline__ T sgn(T x) {
  return Sc<T>::sel(Sc<T>::neg(x), Sc<T>::c(-1.0), Sc<T>::c(1.0));
}

// Cotangents (Lb, Rb) of the face states VL, VR = (rho, u, v, w, p) from the
// cotangent Fb of the Roe flux times the area A along the unit normal n:
// the forward flux of fv_face.cuh recomputed, then swept backwards statement
// by statement.
template <class T>
__device__ __forceinline__ void roe_vjp(const AdjC<T>& P, const T VL[5], const T VR[5], T nx, T ny, T nz, T A,
                                        const T Fb[5], T Lb[5], T Rb[5]) {
  using S = Sc<T>;
  const T zero = S::c(0.0);
  // ---------------- forward ----------------
  const T rL = VL[0], uL = VL[1], vL = VL[2], wL = VL[3], pL = VL[4];
  const T rR = VR[0], uR = VR[1], vR = VR[2], wR = VR[3], pR = VR[4];
  const T VnL = S::dot3(nx, uL, ny, vL, nz, wL), VnR = S::dot3(nx, uR, ny, vR, nz, wR);
  const T riL = S::rcp(rL), riR = S::rcp(rR);
  const T kL = P.g_gm1 * riL, kR = P.g_gm1 * riR;
  const T hL = kL * pL + S::halve(S::dot3(uL, uL, vL, vL, wL, wL));
  const T hR = kR * pR + S::halve(S::dot3(uR, uR, vR, vR, wR, wR));
  const T mL = rL * VnL, mR = rR * VnR;
  const T Rt = S::sqrt(rR * riL);
  const T rt = rL * Rt;
  const T w1 = S::rcp(P.one + Rt), w2 = Rt * w1;
  const T dr = rR - rL, du = uR - uL, dv = vR - vL, dw = wR - wL, dP = pR - pL, dVn = VnR - VnL, dh = hR - hL;
  const T ut = uL + w2 * du, vt = vL + w2 * dv, wt = wL + w2 * dw, ht = hL + w2 * dh;
  const T q2h = S::halve(S::dot3(ut, ut, vt, vt, wt, wt));
  const T c2 = P.gm1 * (ht - q2h);
  const T ct = S::sqrt(c2);
  const T ic2 = S::rcp(c2);
  const T Vnt = VnL + w2 * dVn;
  const T x1 = Vnt - ct, x5 = Vnt + ct;
  const T delta = P.harten * ct;
  T d1l, d1d, d2l, d2d, d5l, d5d;
  const T l1 = fix_fwd(P, S::abs(x1), delta, P.fix, d1l, d1d);
  const T l2 = fix_fwd(P, S::abs(Vnt), delta, P.fix && P.fix_all, d2l, d2d);
  const T l5 = fix_fwd(P, S::abs(x5), delta, P.fix, d5l, d5d);
  const T rc = rt * ct, rcd = rc * dVn;
  const T hic2 = S::halve(ic2);
  const T e1 = dP - rcd, e5 = dP + rcd, e2 = dr - dP * ic2;
  const T a1 = l1 * e1 * hic2, a5 = l5 * e5 * hic2, a2 = l2 * e2, a3 = l2 * rt;
  const T a15 = a1 + a5, a51 = a5 - a1;
  const T E4 = S::dot4(ut, du, vt, dv, wt, dw, -Vnt, dVn);
  // ---------------- reverse ----------------
  const T hA = S::halve(A);
  const T G0 = Fb[0] * hA, G1 = Fb[1] * hA, G2 = Fb[2] * hA, G3 = Fb[3] * hA, G4 = Fb[4] * hA;
  // central part
  const T mLb = G0 + S::dot4(G1, uL, G2, vL, G3, wL, G4, hL);
  const T mRb = G0 + S::dot4(G1, uR, G2, vR, G3, wR, G4, hR);
  const T pnb = S::dot3(nx, G1, ny, G2, nz, G3);
  T hLb = G4 * mL, hRb = G4 * mR;
  // dissipation (every D enters with -1): Gu = G.u~ + G0
  const T Gu = G0 + S::dot3(G1, ut, G2, vt, G3, wt);
  const T gd = S::dot3(G1, du, G2, dv, G3, dw);
  const T a15b = -(Gu + G4 * ht);
  const T d51b = -(pnb + G4 * Vnt);
  const T a2b = -(Gu + G4 * q2h);
  const T a3b = -(gd - pnb * dVn + G4 * E4);
  const T g4a3 = G4 * a3, sa = a15 + a2;
  T utb = -S::dot2(G1, sa, g4a3, du), vtb = -S::dot2(G2, sa, g4a3, dv), wtb = -S::dot2(G3, sa, g4a3, dw);
  T htb = -(G4 * a15);
  T Vntb = -(G4 * (a51 * ct - a3 * dVn));
  T q2hb = -(G4 * a2);
  const T dub = -S::dot2(G1, a3, g4a3, ut), dvb = -S::dot2(G2, a3, g4a3, vt), dwb = -S::dot2(G3, a3, g4a3, wt);
  T dVnb = a3 * (pnb + G4 * Vnt);
  T ctb = d51b * a51;
  const T dc = d51b * ct;
  const T a1b = a15b - dc, a5b = a15b + dc;
  const T t1 = a1b * hic2, t5 = a5b * hic2;
  const T s1 = t1 * l1, s5 = t5 * l5, s2 = a2b * l2;
  const T l2b = S::dot2(a3b, rt, a2b, e2), l5b = t5 * e5, l1b = t1 * e1;
  const T rcdb = s5 - s1;
  const T dPb = (s1 + s5) - s2 * ic2;
  // ic2 enters a2 directly and a1, a5 through its half
  const T ic2b = S::halve(S::dot2(a5b * l5, e5, a1b * l1, e1)) - s2 * dP;
  const T rv = rcdb * dVn;
  T rtb = S::dot2(a3b, l2, rv, ct);
  ctb = ctb + rv * rt;
  dVnb = dVnb + rcdb * rc;
  // eigenvalue magnitudes with the entropy fix (delta = harten ct)
  ctb = ctb + P.harten * S::dot3(l1b, d1d, l2b, d2d, l5b, d5d);
  const T x1b = l1b * d1l * sgn(x1), x2b = l2b * d2l * sgn(Vnt), x5b = l5b * d5l * sgn(x5);
  Vntb = Vntb + ((x1b + x2b) + x5b);
  ctb = ctb + (x5b - x1b);
  // sound speed, averaged normal velocity (VnL + w2 dVn)
  const T c2b = S::halve(ctb * (ct * ic2)) - ic2b * ic2 * ic2;
  const T gc = P.gm1 * c2b;
  htb = htb + gc;
  q2hb = q2hb - gc;
  utb = utb + q2hb * ut;
  vtb = vtb + q2hb * vt;
  wtb = wtb + q2hb * wt;
  // Roe averages phi~ = phi_L + w2 dphi, w2 = Rt / (1 + Rt)
  const T w2b = S::dot4(utb, du, vtb, dv, wtb, dw, htb, dh) + Vntb * dVn;
  const T dub2 = dub + w2 * utb, dvb2 = dvb + w2 * vtb, dwb2 = dwb + w2 * wtb, dhb = w2 * htb;
  dVnb = dVnb + w2 * Vntb;
  const T Rtb = w2b * w1 * w1 + rtb * rL;
  // Rt = sqrt(rR riL): d Rt = Rt / (2 z) dz, z = rR riL
  const T hz = S::halve(Rtb * Rt);                  // Rtb Rt / 2 = zb z
  hLb = hLb + (htb - dhb);
  hRb = hRb + dhb;
  const T VnLb = mLb * rL + (Vntb - dVnb), VnRb = mRb * rR + dVnb;
  const T drb = s2;
  // zb riL = hz / rR, and through riL = 1/rL: -hz / rL
  Lb[0] = S::dot2(mLb, VnL, rtb, Rt) - drb - riL * (hz + hLb * kL * pL);
  Rb[0] = mRb * VnR + drb + riR * (hz - hRb * kR * pR);
  Lb[1] = S::dot3(G1, mL, hLb, uL, nx, VnLb) + (utb - dub2);
  Lb[2] = S::dot3(G2, mL, hLb, vL, ny, VnLb) + (vtb - dvb2);
  Lb[3] = S::dot3(G3, mL, hLb, wL, nz, VnLb) + (wtb - dwb2);
  Rb[1] = S::dot3(G1, mR, hRb, uR, nx, VnRb) + dub2;
  Rb[2] = S::dot3(G2, mR, hRb, vR, ny, VnRb) + dvb2;
  Rb[3] = S::dot3(G3, mR, hRb, wR, nz, VnRb) + dwb2;
  Lb[4] = pnb + hLb * kL - dPb;
  Rb[4] = pnb + hRb * kR + dPb;
}
