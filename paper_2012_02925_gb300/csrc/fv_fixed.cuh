// The Roe flux of the binary64 form in block fixed point: 64-bit integers
// with scales picked per face, on the integer multipliers.
//
// GB300's FP64 unit issues 1.6 lanes per SM and clock, so one binary64
// operation occupies 80 of an SM's 128-lane issue slots; a signed 64 x 64 ->
// high 64 bit product costs about 23 (two IMAD.HI at 4.5, a signed wide IMAD
// at 9, the carries) and a 64-bit sum 3 (measured on the part).
//
// Two scales a face: the thermodynamic quantities and the speed (rho, p, c~,
// h, |u|^2) on the larger, what is proportional to the normal velocity or to
// the jumps (Vn, the mass flux, wave strengths, the energy flux) on one of
// their own, 2^-kn of it.  Both leave 2^-55 .. 2^-57 of the largest term of each
// quantity, where binary64 rounds each of its ~126 operations to 2^-53.  Vn
// and the momentum flux are binary64 (20 operations: a velocity component or a
// normal's may be any amount smaller than the others, and its momentum flux
// follows it).  So every component of the flux is as accurate as binary64's,
// at any Mach number: root mean squares of the error 0.4 .. 1.1 of its
// (tests/test_fixed_roe_accuracy.py).  With one scale and an integer momentum
// flux the 128^3 RK step took 4.20 ms instead of 4.68, but the mass flux had an error of
// 2^-64 of the speed of sound's, 100 times binary64's at Mach 0.001, and a
// momentum component lost the digits by which its velocity was the smaller.
//
// Scales: rho^ = rho 2^-mr in [1/4, 1/2) for the denser side, velocities
// u^ = u 2^-mv with |u^|^2 + 2 gamma/(gamma-1) p^/rho^ < 0.026 on both sides,
// p^ = p 2^-(mr + 2 mv), Vn^ = Vn 2^-mv < 2^-4-kn or kn = 0.  They depend on the
// face's two states and normal only, so a face has the same flux in whatever
// tile or block it is evaluated.  Formats
// ("Qn": integer = value 2^n): rho, velocities Q64; p Q71; Vn Q(64 + kn).
// Ranges that follow from the scales are stated at each line; what they do
// not confine (wave strengths, the flux) is checked, and a face outside its
// ranges (density ratio above about 4, sound speed ratio or Mach number too large,
// non-finite or non-positive states) is left to the binary64 evaluation.
#pragma once
#include <cmath>
#include <cstdint>
#ifdef __CUDACC__
#include <cuda_runtime.h>
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

using fx64 = long long;
using fxu64 = unsigned long long;

// hi 32 bits of the signed 32 x 32 product, plus c
FX_HD int fx_madhi(int a, int b, int c) {
#ifdef __CUDA_ARCH__
  int d;
  asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
#else
  return (int)((unsigned)(int)(((long long)a * b) >> 32) + (unsigned)c);
#endif
}
FX_HD unsigned fx_umulhi(unsigned a, unsigned b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (unsigned)(((fxu64)a * b) >> 32);
#endif
}
// a = h 2^32 + l with l a signed 32-bit number (a < 2^63 - 2^31: h must not wrap)
FX_HD void fx_split(fx64 a, int& h, int& l) {
  l = (int)a;
  h = (int)(a >> 32) + (int)((unsigned)l >> 31);
}
FX_HD fx64 fx_prod(int a, int b) { return (fx64)a * b; }
// a b / 2^64 for |a|, |b| < 2^63 - 2^31: the product of the low halves is left
// out and the two cross products are rounded down (error within 2.3 units;
// zero times anything is zero)
FX_HD fx64 fx_mul(fx64 a, fx64 b) {
  int ah, al, bh, bl;
  fx_split(a, ah, al);
  fx_split(b, bh, bl);
  const int cross = fx_madhi(ah, bl, fx_madhi(al, bh, 0));
  return fx_prod(ah, bh) + cross;
}
// a^2 / 2^64 of a magnitude below 2^63 (a number and its negative thus have the same square)
FX_HD fx64 fx_usqr(fxu64 a) {
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
  return (fx64)((fxu64)ah * ah + fx_umulhi(2 * ah, al));
}
FX_HD fxu64 fx_abs(fx64 a) {
  const fx64 s = a >> 63;
  return (fxu64)((a ^ s) - s);
}
// a b / 2^64 of non-negative numbers below 2^63
FX_HD fx64 fx_umul(fx64 a, fx64 b) {
  const unsigned al = (unsigned)a, ah = (unsigned)(a >> 32), bl = (unsigned)b, bh = (unsigned)(b >> 32);
  fxu64 t = (fxu64)al * bh + 0x80000000u;
  t = (fxu64)ah * bl + t;
  return (fx64)((fxu64)ah * bh + (t >> 32));
}// the same of a >= 0 and any b, the sign apart: a stream and its reverse have
// the same products
FX_HD fx64 fx_smul(fx64 a, fx64 b) {
  const fx64 s = b >> 63, t = fx_umul(a, (b ^ s) - s);
  return (t ^ s) - s;
}

FX_HD int fx_clz64(fxu64 x) {   // x > 0
#ifdef __CUDA_ARCH__
  const unsigned h = (unsigned)(x >> 32);
  return __clz((int)(h ? h : (unsigned)x)) + (h ? 0 : 32);
#else
  return __builtin_clzll(x);
#endif
}
FX_HD float fx_rcpf(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / x;
#endif
}
FX_HD float fx_rsqrtf(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / sqrtf(x);
#endif
}
FX_HD float fx_u2f(unsigned x) {
#ifdef __CUDA_ARCH__
  return __uint2float_rn(x);
#else
  return (float)x;
#endif
}
FX_HD unsigned fx_f2u(float x) {
#ifdef __CUDA_ARCH__
  return __float2uint_rz(x);
#else
  return (unsigned)x;
#endif
}

// 32-bit r with r = 2^31 / s (1 + e), |e| <= 2^-21, for s = S / 2^64 in [1/2, 1)
// (S's top bit set); below 2^32
FX_HD unsigned fx_rcp_seed(unsigned sh) {
  // 2^31 / s = 2^63 / sh; the factor keeps sh = 2^31 below 2^32
  return fx_f2u(fx_rcpf(fx_u2f(sh)) * (9223372036854775808.0f * 0.9999997f));
}

// 1 / s for S normalised as above, in Q62: the seed refined by the series
// 1/(s y0) = 1 + e + e^2 + ..., e = 1 - s y0, to its e^2 term
FX_HD fx64 fx_rcp(fxu64 S) {
  const unsigned sh = (unsigned)(S >> 32), sl = (unsigned)S;
  const unsigned r = fx_rcp_seed(sh);
  const fx64 e = (fx64)(0x8000000000000000ull - ((fxu64)sh * r + fx_umulhi(sl, r)));   // Q63, |e| < 2^43
  const int eh = (int)(e >> 12);                                                        // Q51
  const fx64 c = (e << 19) + ((fx64)fx_madhi(eh, eh, 0) << 12);                         // e + e^2, Q82
  // r (1 + c): r is Q31, c Q82 -> Q81 (hi) -> Q62
  const int rs = (int)(r >> 1);                                                         // Q30, signed
  int ch, cl;
  fx_split(c, ch, cl);
  const fx64 t = fx_prod(rs, ch) + fx_madhi(rs, cl, 0);                                 // Q80
  return ((fx64)r << 31) + (t >> 18) + ((r & 1u) ? (c >> 51) : 0);
}

// 1 / sqrt(x) for x = X / 2^64 in (1/16, 1/2), Q61: y0 (1 + e/2 + 3 e^2/8),
// e = 1 - x y0^2 (binomial series)
FX_HD fx64 fx_rsqrt(fx64 X) {
  const unsigned xh = (unsigned)((fxu64)X >> 32);
  const unsigned y = fx_f2u(fx_rsqrtf(fx_u2f(xh)) * 35184372088832.0f);   // Q29: 2^29 2^16
  const fxu64 yy = (fxu64)y * y;                                          // Q58
  const fx64 e = (1ll << 58) - fx_umul(X, (fx64)yy);                      // Q58, |e| < 2^37
  const int eh = (int)(e >> 6);                                           // Q52
  const fx64 c = (e << 22) + ((fx64)(3 * fx_madhi(eh, eh, 0)) << 6);      // e/2 + 3 e^2/8, Q81
  int ch, cl;
  fx_split(c, ch, cl);
  const fx64 t = fx_prod((int)y, ch) + fx_madhi((int)y, cl, 0);           // Q78
  return ((fx64)y << 32) + (t >> 17);
}

// ---------------------------------------------------------------------------
// the face
// ---------------------------------------------------------------------------
struct FxConsts {
  fx64 K;        // gamma/(gamma-1), Q60 (below 8)
  fx64 gm1;      // gamma - 1, Q63 (below 1)
  fx64 eta;      // entropy-fix width / c~, Q62 (below 1; 0: no fix)
  fx64 ieta;     // its reciprocal, Q59 (below 16)
  float k2;      // 2 gamma/(gamma-1), rounded up
  float g;       // gamma, rounded down
  int on;        // the scheme's constants fit these formats
};

// The constants; off (the binary64 evaluation everywhere) where gamma or the
// entropy-fix width does not fit the formats, or gamma is so near 1 that p^
// and c^ lose the bits that keep the error below binary64's
inline FxConsts fx_consts(double gamma, double harten) {
  FxConsts x = FxConsts();
  x.on = gamma >= 1.3 && gamma <= 1.95 && (harten <= 0.0 || (harten >= 0.0626 && harten <= 0.95));
  if (!x.on) return x;
  const long double g = gamma, gm1 = g - 1.0L;
  x.K = (fx64)std::ldexp(g / gm1, 60);
  x.gm1 = (fx64)std::ldexp(gm1, 63);
  if (harten > 0.0) {
    x.eta = (fx64)std::ldexp((long double)harten, 62);
    x.ieta = (fx64)std::ldexp(1.0L / (long double)harten, 59);
  }
  x.k2 = (float)(2.0L * g / gm1 * 1.000001L);
  x.g = (float)(g * 0.999999L);
  return x;
}

// magnitude bits of x's high word, for the range checks
FX_HD unsigned fx_mag(fx64 x) {
  const int h = (int)(x >> 32);
  return (unsigned)(h ^ (h >> 31));
}

// Harten's fix on an eigenvalue over c~ (Q(56 + ls)): (l^2/eta + eta)/2 below eta
FX_HD fx64 fx_entropy(const FxConsts& C, fx64 lam, int ls) {
  const fx64 eta = C.eta >> (6 - ls);
  if (lam < eta) {
    const fx64 l = lam << (7 - ls);                       // Q63
    const fx64 l2 = fx_umul(l, l);                        // Q62
    lam = ((fx_umul(l2, C.ieta) << 4) >> (6 - ls)) + (eta >> 1);   // Q57, halved Q58 -> Q62 -> Q(56 + ls)
  }
  return lam;
}

// What the flux is made of: density and pressure of both sides (rho Q64, p
// Q71), |u|^2 of both and |u_R - u_L|^2 (Q64) on the face's scales; normal
// velocities (Q(64 + kn)) and the jump of p (Q(71 + kn)) on theirs.  ls: the
// face's format of the eigenvalues over c~ (Q(56 + ls), 3..6).
struct FxFace {
  fx64 rL, rR, pL, pR, qL, qR, e, VnL, VnR, dp;
  int kn, ls;
};
// Twice the flux per unit area in four numbers: the mass flux M (Q(65 + kn)),
// the factor G of u_R - u_L (Q(65 + kn)), the dissipative pressure X (Q(67 + kn)) and
// the energy flux E (Q(69 + kn)); the momentum flux is M u_L + G (u_R - u_L) +
// n (p_L + p_R + X).  Where the entropy fix has raised |lambda_2|, which then does
// not get small with Vn~ (fixed), they are without the waves of that eigenvalue,
// a2 = l2 dr - t2 and a3 = l2 rt, and its parts follow: l2 (Q64), t2 (Q(65 + kn)),
// rt (Q64) and beta (Q62).
struct FxFlux {
  fx64 M, G, X, E, l2, t2, rt, beta;
  bool fixed;
};

// Returns nonzero when a quantity has left its range (the flux is then not to
// be used): |M| < 0.166, |G| < 3/16, |E| < 1/256, so that the intermediate
// sums cannot have wrapped unnoticed.
//
// The same flux as roe_flux's, regrouped: with m = rho Vn of the two sides,
// D0 = a1 + a5 + a2, beta the weight of R in the Roe averages, du = u_R - u_L,
//   F_mass = m_L + m_R - D0
//   F_mom  = F_mass u_L + (m_R - beta D0 - a3) du + n (p_L + p_R - d51 + a3 dVn)
//   F_en   = (F_mass + a2) h_L + (m_R - beta a15) dh - d51 Vn~ - a2 q~ - a3 (u~.du - Vn~ dVn)
// and c~^2 = (gamma-1)(H_L + beta dH + beta (1-beta) |du|^2/2), H = c^2/(gamma-1):
// no cancelling h~ - |u~|^2/2.
FX_HD unsigned fx_roe(const FxConsts& C, const FxFace& f, bool fix_all, FxFlux& F) {
  const fx64 rL = f.rL, rR = f.rR, VnL = f.VnL, VnR = f.VnR, qL = f.qL, qR = f.qR, e = f.e;
  const int kn = f.kn < 63 ? f.kn : 63, ls = f.ls;       // kn as a shift
  const fx64 mL = fx_smul(rL, VnL), mR = fx_smul(rR, VnR);                 // Q(64 + kn)
  const fx64 dVn = VnR - VnL;
  // 1/sqrt(rho): sqrt(rho) (Q63), 1/rho (Q59)
  const fx64 yL = fx_rsqrt(rL), yR = fx_rsqrt(rR);
  const fx64 sL = fx_umul(rL, yL) << 2, sR = fx_umul(rR, yR) << 2;
  // H = gamma/(gamma-1) p/rho, Q66
  const fx64 HL = fx_umul(fx_umul(f.pL, fx_umul(yL, yL) << 1) << 4, C.K);
  const fx64 HR = fx_umul(fx_umul(f.pR, fx_umul(yR, yR) << 1) << 4, C.K);
  const fx64 dq = qR - qL, dH = HR - HL;
  // beta = sqrt(rho_R)/(sqrt(rho_L) + sqrt(rho_R)), Q62; rho~, Q64
  const fxu64 ss = (fxu64)sL + (fxu64)sR;                // Q63, 1/2 .. sqrt 2
  const int nz = fx_clz64(ss);
  const fx64 beta = fx_umul((fx64)((fxu64)sR << nz >> 1), fx_rcp(ss << nz)) << 1;
  // sR (Q63) << nz = Q(63+nz) of sR, the reciprocal is of ss << nz: their
  // ratio is Q62 after >> 1 (Q63 x Q62 >> 64 = Q61) << 1
  const fx64 rt = fx_umul(sL, sR) << 2;
  const fx64 be = fx_mul(beta << 1, e) << 1;             // beta e, Q64 (e/2: Q65)
  const fx64 b2 = be - (fx_mul(beta << 1, be) << 1);     // beta (1 - beta) e
  const fx64 X = HL + (fx_mul(beta << 1, dH) << 1) + 2 * b2;   // Q66 (b2/2 is Q65)
  const fx64 c2 = fx_umul(C.gm1, X << 2) << 1;           // Q68, below 1/32
  // 1/c, Q56: c2 2^(z+4) lies in [1/8, 1/2) for the even shift z that moves
  // its leading bit to 2^62 or 2^61, so 1/c = y 2^(z/2+2)
  const int z = (fx_clz64((fxu64)c2 | 1) - 1) & 62;
  const int ish = 3 - (z >> 1);
  const fx64 yc = fx_rsqrt(c2 << z);
  const fx64 ic = ish >= 0 ? yc >> ish : yc << -ish;
  const fx64 c = fx_umul(c2, ic) << 4;                   // Q60 -> Q64
  const fx64 Vnt = VnL + (fx_mul(beta << 1, dVn) << 1);  // Q(64 + kn)
  const fxu64 an = fx_abs(Vnt);
  const fx64 Vc = Vnt >> kn, ac = (fx64)(an >> kn);      // Q64
  // eigenvalues over c~, Q(56 + ls): the scales keep them below 2^(7 - ls), ls = 3..6
  const fx64 k1 = fx_entropy(C, fx_umul((fx64)fx_abs(Vc - c), ic) << ls, ls);
  const fx64 k5 = fx_entropy(C, fx_umul((fx64)fx_abs(Vc + c), ic) << ls, ls);
  fx64 k2 = fx_umul(ac, ic) << ls;
  // wave strengths: P = dp/c~, kap = rho~ dVn
  const fx64 P = fx_mul(f.dp, ic) << 1;                  // Q(63 + kn) -> Q(64 + kn)
  const fx64 kap = fx_mul(rt, dVn);                      // Q(64 + kn)
  const fx64 a1 = fx_smul(k1, P - kap), a5 = fx_smul(k5, P + kap);      // x Q65 -> Q(57 + ls + kn)
  unsigned wild = (fx_mag(a1) | fx_mag(a5)) >> (20 + ls);               // each below 1/32
  wild |= fx_mag(c) >> 29;                                              // c~ below 1/8
  const fx64 a15 = (a1 + a5) << (8 - ls), a51 = (a5 - a1) << (8 - ls);  // Q(65 + kn) from here
  const bool fixed = fix_all && k2 < (C.eta >> (6 - ls));
  if (fixed) k2 = fx_entropy(C, k2, ls);
  const fx64 t2 = fx_mul(k2, P << 2);                                   // Q(58 + ls + kn)
  wild |= (fx_mag(t2) >> 1) >> (19 + ls);                               // below 1/64
  fx64 A2 = 0, a3 = 0;
  F.fixed = fixed;
  if (fixed) {
    F.l2 = fx_umul(k2 << (6 - ls), c) << 2;                             // Q62 -> Q64
    F.t2 = t2 << (7 - ls);
    F.rt = rt;
    F.beta = beta;
  } else {
    A2 = (fx_mul((fx64)an, rR - rL) << 1) - (t2 << (7 - ls));
    a3 = fx_mul((fx64)an, rt) << 1;
  }
  const fx64 M1 = ((mL + mR) << 1) - a15;
  const fx64 D0 = a15 + A2;
  const fx64 d51 = fx_mul(a51, c << 2);                                 // Q(67 + kn)
  const fx64 mR1 = mR << 1;
  F.M = M1 - A2;
  F.X = (fx_mul(a3, dVn) << 2 >> kn) - d51;
  F.G = mR1 - (fx_mul(beta << 1, D0) << 1) - a3;
  wild |= fx_mag(F.M) > 0x54fdf3b5u || fx_mag(F.G) > 0x5fffffffu;
  // energy, Q(69 + kn)
  const fx64 hL = (HL + 2 * qL) << 2, dh = (dH + 2 * dq) << 2;          // Q68
  const fx64 G4 = mR1 - (fx_mul(beta << 1, a15) << 1);
  F.E = fx_smul(hL, M1) + fx_mul(G4, dh) - (fx_mul(d51 << 2, Vnt) >> kn);
  if (!fixed) {
    fx64 qt = (qL + (fx_mul(beta << 1, dq) << 1) - b2) << 3;            // q~, Q65 -> Q68
    qt = qt > 0 ? qt : 0;                                               // (opposed velocities: down to rounding)
    const fx64 uw = (dq - e) + 2 * be;                                  // u~.du, Q65
    const fx64 ud = (uw << 1) - ((fx_mul(Vnt, dVn) >> kn) >> kn << 2);  // u~.du - Vn~ dVn, Q66
    F.E -= fx_smul(qt, A2) + (fx_smul(a3 << 1, ud) << 1);
  }
  return wild | (fx_mag(F.E) >> 29);
}

// ---------------------------------------------------------------------------
// scales and conversions
// ---------------------------------------------------------------------------
FX_HD int fx_hi(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  long long b;
  __builtin_memcpy(&b, &x, 8);
  return (int)(b >> 32);
#endif
}
FX_HD unsigned fx_lo(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(x);
#else
  long long b;
  __builtin_memcpy(&b, &x, 8);
  return (unsigned)b;
#endif
}
FX_HD float fx_asfloat(int b) {
#ifdef __CUDA_ARCH__
  return __int_as_float(b);
#else
  float f;
  __builtin_memcpy(&f, &b, 4);
  return f;
#endif
}
FX_HD int fx_asint(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_int(f);
#else
  int b;
  __builtin_memcpy(&b, &f, 4);
  return b;
#endif
}
// |x| as binary32 from its high word h (below by up to 2^-20 of it); zero
// under 2^-100, for |x| < 2^60
FX_HD float fx_approx(int h) {
  h &= 0x7fffffff;
  return h < (923 << 20) ? 0.0f : fx_asfloat((h - (896 << 20)) << 3);
}

struct FxScale {
  int mr, mv, ls;
  float ic;      // an upper bound of 1/c^ of both sides
};
// The face's scales from its two states; false when they do not fit
FX_HD bool fx_scale(const FxConsts& C, const double VL[5], const double VR[5], FxScale& S) {
  const int hrL = fx_hi(VL[0]), hrR = fx_hi(VR[0]), hpL = fx_hi(VL[4]), hpR = fx_hi(VR[4]);
  // rho within 2^+-40, p within 2^+-80 (unsigned: a negative or non-finite
  // value is beyond), velocities below 2^60
  int hu[6] = {fx_hi(VL[1]), fx_hi(VL[2]), fx_hi(VL[3]), fx_hi(VR[1]), fx_hi(VR[2]), fx_hi(VR[3])};
  int um = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    hu[i] &= 0x7fffffff;
    um = um > hu[i] ? um : hu[i];
  }
  const unsigned r0 = 983u << 20, rw = 80u << 20, p0 = 943u << 20, pw = 160u << 20;
  bool ok = (unsigned)hrL - r0 < rw && (unsigned)hrR - r0 < rw && (unsigned)hpL - p0 < pw && (unsigned)hpR - p0 < pw &&
            um < (1083 << 20);
  const int hM = hrL > hrR ? hrL : hrR, hm = hrL > hrR ? hrR : hrL;
  const int eM = (hM + 1) >> 20;                          // rho^ below 1/2 (1 - 2^-20): see fx_split
  ok = ok && hm >= ((eM - 2) << 20) + 0x1000;             // rho^ above 1/16
  const float rL = fx_approx(hrL), rR = fx_approx(hrR);
  const float tL = fx_approx(hpL) * fx_rcpf(rL), tR = fx_approx(hpR) * fx_rcpf(rR);
  const float a0 = fx_approx(hu[0]), a1 = fx_approx(hu[1]), a2 = fx_approx(hu[2]);
  const float b0 = fx_approx(hu[3]), b1 = fx_approx(hu[4]), b2 = fx_approx(hu[5]);
  const float uL = a0 * a0 + a1 * a1 + a2 * a2, uR = b0 * b0 + b1 * b1 + b2 * b2;
  const float vL = uL + C.k2 * tL, vR = uR + C.k2 * tR;
  const float vv = (vL > vR ? vL : vR) * (1.00003f / 0.026f);
  // vv < 2^e; the velocities' squares are scaled by 2^-2 mv <= 2^-e
  S.mv = ((fx_asint(vv) >> 23) - 126 + 1) >> 1;
  S.mr = eM - 1021;
  const float c2 = C.g * (tL < tR ? tL : tR) * 0.99997f, uu = (uL > uR ? uL : uR) * 1.00003f;
  // eigenvalues over c~ are below 1 + |u|/c
  S.ls = uu < 0.97f * c2 ? 6 : (uu < 8.8f * c2 ? 5 : (uu < 48.0f * c2 ? 4 : 3));
  // 1/c~ below 120 (Q56), and dp/c~ <= max p^ / min c^ < 0.12 (rho^ < 1/2)
  const float s2 = fx_asfloat((127 - 2 * S.mv) << 23), T = (tL > tR ? tL : tR) * s2;
  S.ic = fx_rsqrtf(c2 * s2) * 1.0001f;
  return ok && uu < 220.0f * c2 && c2 * s2 > 7.0e-5f && T * T < 0.0575f * (c2 * s2);
}

// The scale of what is proportional to the normal velocities or the jumps, 2^-kn
// of the face's: Vn^ < 2^-4-kn, rho^ |dVn^| and |dp^|/c^ < 2^-6-kn.  dn: |dVn| in
// Q(64 + kv), at the scale 2^-kv of Vn alone; dp: |dp| in Q(71 + kp).
FX_HD int fx_scale_n(const FxScale& S, int kv, fxu64 dn, int kp, fxu64 dp) {
  int k = kv;
  if (dn) {
    const int j = kv + fx_clz64(dn) - 5;
    k = k < j ? k : j;
  }
  if (dp) {
    const int z = fx_clz64(dp);
    const float f = fx_u2f((unsigned)((dp << z) >> 32)) * S.ic;
    const int j = 33 + z + kp - ((fx_asint(f) >> 23) - 126);
    k = k < j ? k : j;
  }
  return k < 0 ? 0 : k;
}

// binary64 value times 2^64 / 2^m (c = 1021 + m) truncated: the significand at
// bit 62 moved right by c - E; the scales keep the shift non-negative
FX_HD fxu64 fx_magnitude(double x, int c) {
  const int hi = fx_hi(x);
  const unsigned lo = fx_lo(x);
  const fxu64 M = ((fxu64)(((((unsigned)hi & 0xfffffu) | 0x100000u) << 10) | (lo >> 22)) << 32) | (lo << 10);
  const unsigned r = (unsigned)(c - ((hi >> 20) & 0x7ff));
  return M >> (r > 63u ? 63u : r);
}
FX_HD fx64 fx_sign(fxu64 v, double x) {
  const fx64 sg = (fx64)(fx_hi(x) >> 31);
  return ((fx64)v ^ sg) - sg;
}
FX_HD fx64 fx_convert(double x, int c) { return fx_sign(fx_magnitude(x, c), x); }

FX_HD double fx_double(int hi, unsigned lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, (int)lo);
#else
  const fxu64 b = ((fxu64)(unsigned)hi << 32) | lo;
  double d;
  __builtin_memcpy(&d, &b, 8);
  return d;
#endif
}

// x 2^e rounded to nearest (the result a normal number or zero).  On the
// integer units: the conversion instruction is held by the FP64 unit (five of
// them a face, 128^3 RK step 4.70 against 4.56 ms).
FX_HD double fx_to_double(fx64 x, int e) {
  const fxu64 H = fx_abs(x);
  const int z = fx_clz64(H | 1);
  const fxu64 N = H << z;
  const fxu64 b = (N >> 11) + ((N >> 10) & 1) + ((fxu64)(unsigned)(e + 1085 - z) << 52);
  const int sg = (int)(x >> 32) & (int)0x80000000;
  return fx_double(H ? (int)(b >> 32) | sg : 0, H ? (unsigned)b : 0u);
}

// 2^30 / s' for s' = (2^32 sh + sl) / 2^64 in [1/2, 1): 32 bits (the hardware's
// approximation to 22 bits, one Newton step), and e2 = 2^62 (1 - s' r / 2^30),
// |e2| < 2^34
FX_HD unsigned fx_rcp32(unsigned sh, unsigned sl, fx64& e2) {
  const float f = fx_asfloat((int)(0x3f800000u | ((sh >> 8) & 0x7fffffu)));   // 2 s'
#ifdef __CUDA_ARCH__
  const float g = __fmaf_rn(fx_rcpf(f), 4194302.0f, 8388608.0f);        // 2^23 + 2^22 / f (r0 below 2^31)
#else
  const float g = fmaf(fx_rcpf(f), 4194302.0f, 8388608.0f);
#endif
  const unsigned r0 = ((unsigned)fx_asint(g) & 0x7fffffu) << 9;         // 2^31 / f = 2^30 / s'
  const int e1 = (int)(0x40000000u - fx_umulhi(sh, r0));
  const unsigned r = r0 + (unsigned)fx_madhi((int)r0, e1 * 4, 0);
  e2 = (fx64)(0x4000000000000000ull - ((fxu64)sh * r + fx_umulhi(sl, r)));
  return r;
}
// P / s' from the reciprocal above, P in [2^60, 2^63): the product and its correction
FX_HD fxu64 fx_quot(fxu64 P, unsigned r, fx64 e2) {
  const fxu64 H0 = ((fxu64)(unsigned)(P >> 32) * r + fx_umulhi((unsigned)P, r)) << 2;
  return H0 + (fxu64)((fx64)fx_madhi((int)(H0 >> 32), (int)(e2 >> 3), 0) << 5);
}
// H 2^(e - 1086), H >= 2^32, rounded to binary64's 53 bits: its pattern
// without a sign (the exponent in the normal range)
FX_HD fxu64 fx_round(fxu64 H, int e) {
#ifdef __CUDA_ARCH__
  const int z = __clz((int)(unsigned)(H >> 32));
#else
  const int z = __builtin_clz((unsigned)(H >> 32));
#endif
  const fxu64 N = H << z;
  return (N >> 11) + ((N >> 10) & 1) + ((fxu64)(unsigned)(e - 1 - z) << 52);
}

// n / d for a finite d > 0, within 0.65 units in the last place; a quotient
// below the normal range is 0, above it infinite, of a non-finite n or a
// subnormal d NaN
FX_HD double fx_div(double n, double d) {
  const int hn = fx_hi(n), hd = fx_hi(d);
  const unsigned ln = fx_lo(n), ld = fx_lo(d);
  const int en = (hn >> 20) & 0x7ff, ed = (hd >> 20) & 0x7ff;
  const unsigned dh = ((((unsigned)hd & 0xfffffu) | 0x100000u) << 11) | (ld >> 21), dl = ld << 11;   // [2^63, 2^64)
  const fxu64 P = ((fxu64)(((((unsigned)hn & 0xfffffu) | 0x100000u) << 9) | (ln >> 23)) << 32) | (ln << 9);   // [2^61, 2^62)
  fx64 e2;
  const unsigned r = fx_rcp32(dh, dl, e2);
  const fxu64 H = fx_quot(P, r, e2);                                    // [2^61, 2^63)
  // n = P 2^(en - 1084), d = s' 2^64 2^(ed - 1086): H 2^(en - ed - 62)
  const int e = en - ed + 1024;
  const fxu64 b = fx_round(H, e);
  const int sg = hn & (int)0x80000000;
  const bool nan = en == 2047 || ed == 2047 || hd < (1 << 20);
  const bool zero = en == 0 || e < 4;
  const bool inf = (unsigned)(b >> 52) >= 2047u;
  const int hi = nan ? 0x7ff80000 : (zero ? sg : (inf ? sg | 0x7ff00000 : sg | (int)(b >> 32)));
  return fx_double(hi, nan || zero || inf ? 0u : (unsigned)b);
}

// Half the van Leer limited slope of differences a, b: a b/(a + b) when they
// have the same sign, else 0, within 0.65 units in the last place; 0 when
// both are below 2^-100 (rounding noise of a quantity that is zero).  The
// significands' product over their aligned sum, by a 32-bit reciprocal (the
// hardware's approximation, one Newton step) and one correction.  About 140
// issue slots where the six binary64 operations (product, sum, reciprocal of
// three, product) hold the FP64 unit for 480.  128^3 RK step: 5.83 -> 4.28 ms (autotuned),
// 64-block batch: 49.2 -> 39.4 ms.
FX_HD double fx_vanleer_half(double a, double b) {
  const int ha = fx_hi(a), hb = fx_hi(b);
  const unsigned la = fx_lo(a), lb = fx_lo(b);
  const int ea = (ha >> 20) & 0x7ff, eb = (hb >> 20) & 0x7ff;
  const unsigned ah = ((((unsigned)ha & 0xfffffu) | 0x100000u) << 10) | (la >> 22), al = la << 10;
  const unsigned bh = ((((unsigned)hb & 0xfffffu) | 0x100000u) << 10) | (lb >> 22), bl = lb << 10;
  const fxu64 A = ((fxu64)ah << 32) | al, B = ((fxu64)bh << 32) | bl;   // [2^62, 2^63): a = A 2^(ea - 1085)
  const int em = ea > eb ? ea : eb, en = ea > eb ? eb : ea;
  const int d = em - en;
  const fxu64 big = ea > eb ? A : B, small = ea > eb ? B : A;
  const fxu64 S0 = big + (d < 64 ? small >> (d & 63) : 0);              // [2^62, 2^64)
  const int n = (int)(~(unsigned)(S0 >> 32) >> 31);
  const fxu64 S = S0 << n;                                              // s' = S / 2^64 in [1/2, 1)
  fx64 e2;
  const unsigned r = fx_rcp32((unsigned)(S >> 32), (unsigned)S, e2);
  const fxu64 H = fx_quot((fxu64)fx_umul((fx64)A, (fx64)B), r, e2);     // product in [2^60, 2^62)
  // h = H 2^(n + ea + eb - em - 1085)
  const fxu64 bits = fx_round(H, en + 1 + n);
  // a NaN comes through whatever the signs, an infinity with a number of its sign gives one
  const int ma = ha & 0x7fffffff, mb = hb & 0x7fffffff;
  const bool nan = (ma > mb ? ma : mb) > 0x7ff00000;
  const bool zero = !nan && ((ha ^ hb) < 0 || em < 923 || en < 64);
  const int hh = (int)(bits >> 32) | (ha & (int)0x80000000);
  return fx_double(zero ? 0 : (em == 2047 ? 0x7ff80000 : hh), zero ? 0u : (unsigned)bits);
}

// Roe flux times the area A of the states VL, VR along the unit normal n in
// `out`; false (out not written) when the face does not fit.
FX_HD bool fx_roe_flux(const FxConsts& C, const double VL[5], const double VR[5], double nx, double ny, double nz,
                       double A, bool fix_all, double out[5]) {
  // |n_i| <= 1 up to rounding: a NaN or a larger value does not fit
  const int nm = (fx_hi(nx) & 0x7fffffff) > (fx_hi(ny) & 0x7fffffff) ? fx_hi(nx) & 0x7fffffff : fx_hi(ny) & 0x7fffffff;
  if ((nm > (fx_hi(nz) & 0x7fffffff) ? nm : fx_hi(nz) & 0x7fffffff) >= (1024 << 20)) return false;
  const int ah = fx_hi(A);
  if (!((unsigned)ah - (823u << 20) < (400u << 20))) return false;   // 2^-200 .. 2^200
  FxScale S;
  if (!fx_scale(C, VL, VR, S)) return false;
  const double VnL = fma(nx, VL[1], fma(ny, VL[2], nz * VL[3])), VnR = fma(nx, VR[1], fma(ny, VR[2], nz * VR[3]));
  FxFace f;
  const int cr = 1021 + S.mr, cv = 1021 + S.mv, cp = 1014 + S.mr + 2 * S.mv;
  // (2^-400 of the face's scale is zero)
  const int hn = (fx_hi(VnL) & 0x7fffffff) > (fx_hi(VnR) & 0x7fffffff) ? fx_hi(VnL) & 0x7fffffff : fx_hi(VnR) & 0x7fffffff;
  int kv = S.mv - 4 - ((hn >> 20) - 1022);
  if (kv < -2) return false;   // |Vn^| above 1/4: no unit normal
  kv = kv < 0 ? 0 : (kv < 400 ? kv : 400);
  f.VnL = fx_convert(VnL, cv - kv);
  f.VnR = fx_convert(VnR, cv - kv);
  const int em = (fx_hi(VL[4]) > fx_hi(VR[4]) ? fx_hi(VL[4]) : fx_hi(VR[4])) >> 20, kp = cp - em;
  f.pL = (fx64)fx_magnitude(VL[4], em);
  f.pR = (fx64)fx_magnitude(VR[4], em);
  f.dp = f.pR - f.pL;
  f.kn = fx_scale_n(S, kv, fx_abs(f.VnR - f.VnL), kp, fx_abs(f.dp));
  f.VnL >>= kv - f.kn < 63 ? kv - f.kn : 63;
  f.VnR >>= kv - f.kn < 63 ? kv - f.kn : 63;
  f.pL >>= kp;
  f.pR >>= kp;
  f.dp = f.kn > kp ? f.dp << (f.kn - kp < 63 ? f.kn - kp : 63) : f.dp >> (kp - f.kn);
  f.ls = S.ls;
  f.rL = (fx64)fx_magnitude(VL[0], cr);
  f.rR = (fx64)fx_magnitude(VR[0], cr);
  f.qL = f.qR = f.e = 0;
#pragma unroll
  for (int i = 1; i < 4; ++i) {
    const fxu64 a = fx_magnitude(VL[i], cv), b = fx_magnitude(VR[i], cv);
    f.qL += fx_usqr(a);
    f.qR += fx_usqr(b);
    f.e += fx_usqr(fx_abs(fx_sign(b, VR[i]) - fx_sign(a, VL[i])));
  }
  FxFlux F;
  if (fx_roe(C, f, fix_all, F)) return false;
  // the area's significand, Q63 in [1/2, 1) with its top kept from rounding
  // up to 1 (fx_split), and exponent; F is twice the flux
  const unsigned al = fx_lo(A);
  const int ea = (ah + 1) >> 20;
  const fx64 am = (fx64)((((fxu64)(((((unsigned)ah & 0xfffffu) | 0x100000u) << 10) | (al >> 22)) << 32) | (al << 10)) >>
                         (ea - (ah >> 20)));
  const int e = ea - 1022 - 65 + S.mr + S.mv;
  double M = fx_to_double(fx_smul(am, F.M), e - f.kn), G = fx_to_double(fx_mul(F.G, am), e - f.kn);
  double X = fx_to_double(fx_mul(F.X, am), e - 2 + S.mv - f.kn);
  double E = fx_to_double(fx_smul(am, F.E), e - 4 + 2 * S.mv - f.kn);
  const double hA = fx_double(ah - (1 << 20), al);
  if (fix_all && F.fixed) {
    const double b = fx_to_double(F.beta, -62), dVn = VnR - VnL;
    const double l2A = fx_to_double(F.l2, S.mv - 64) * hA;
    const double a2 = fma(l2A, VR[0] - VL[0], -fx_to_double(fx_mul(F.t2, am), e - f.kn));
    const double a3 = l2A * fx_to_double(F.rt, S.mr - 64);
    double ud = -fma(b, dVn, VnL) * dVn, q = 0.0;
#pragma unroll
    for (int i = 1; i < 4; ++i) {
      const double du = VR[i] - VL[i], ut = fma(b, du, VL[i]);
      ud = fma(ut, du, ud);
      q = fma(ut, ut, q);
    }
    M -= a2;
    G = fma(-b, a2, G) - a3;
    X = fma(a3, dVn, X);
    E = fma(-0.5 * a2, q, fma(-a3, ud, E));
  }
  const double P = fma(VL[4] + VR[4], hA, X);
  out[0] = M;
  out[1] = fma(nx, P, fma(M, VL[1], G * (VR[1] - VL[1])));
  out[2] = fma(ny, P, fma(M, VL[2], G * (VR[2] - VL[2])));
  out[3] = fma(nz, P, fma(M, VL[3], G * (VR[3] - VL[3])));
  out[4] = E;
  return true;
}
