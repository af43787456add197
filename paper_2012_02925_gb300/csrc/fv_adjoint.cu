// Discrete adjoint (vector-Jacobian product) of one Runge-Kutta stage; the
// face VJPs and the limiter's derivatives in binary64 or double-float
// arithmetic, everything else - sums, recovery, exchange - binary64.  Stage map: Q^(m) = Q^(0) - alpha_m dt / Omega * R(X(Q^(m-1)))
// with X the ghost exchange.  For a cotangent lam of Q^(m):
//   mu_c   = -alpha_m dt / Omega_c * lam_c              (cotangent of R_c)
//   Fbar_f = mu_L(f) - mu_R(f)                          (R_L holds +F_f, R_R holds -F_f)
//   per face: cotangents of its two states from Fbar_f    (roe_vjp)
//   per cell: slopes, then primitive recovery transposed  (adj_slope_kernel, adj_cell_kernel)
//   ghost cotangents are added into their donor cells (transpose of X),
//   fixed ghosts are constants.
// Deterministic: the faces' cotangents go to a scratch array and every cell
// gathers its own in a fixed order; connections are transposed one launch at
// a time in table order.
//
// 96^3 VJP stage (van Albada), double-float sweeps 1.80 -> 0.80 ms, binary64
// 4.58 -> 2.74 ms against one kernel per face that recovered its four cells'
// primitives, evaluated the limiter's derivatives (20 of them), and reversed
// all of it into 20 conserved cotangents (12,700 instructions a face, 160
// bytes written): a face now does its Roe part and writes 10 cotangents
// component by component; limiter derivatives and the recovery's transpose
// are taken per cell.
#include "fv_adjoint.cuh"
#include "fv_internal.h"

namespace {

__device__ __forceinline__ long long ghost_index(const FvBlockDev& B, int i, int j, int k) {
  return (long long)(k + FV_GHOST) * B.kstride + (long long)(j + FV_GHOST) * B.jstride + (i + FV_GHOST);
}

// storage of an arithmetic type's values (8 bytes either way)
template <class T> struct AdjMem;
template <> struct AdjMem<double> {
  using type = double;
  static __device__ __forceinline__ double ld(const double* p) { return __ldg(p); }
  static __device__ __forceinline__ void st(double* p, double v) { *p = v; }
  static __device__ __forceinline__ double to_d(double v) { return v; }
};
template <> struct AdjMem<df64> {
  using type = float2;
  static __device__ __forceinline__ df64 ld(const float2* p) {
    const float2 v = __ldg(p);
    return mk(v.x, v.y);
  }
  static __device__ __forceinline__ void st(float2* p, df64 v) { *p = make_float2(v.hi, v.lo); }
  // hi + lo (a normalised pair) rounded to binary64 on the integer units: a sum on
  // the FP64 unit stands for 80 issue slots
  static __device__ __forceinline__ double to_d(df64 v) {
    const unsigned h = (unsigned)__float_as_int(v.hi), l = (unsigned)__float_as_int(v.lo);
    const int eh = (int)(h >> 23) & 255, el = (int)(l >> 23) & 255, d = eh - el;
    const unsigned long long H = (unsigned long long)((h & 0x7fffffu) | 0x800000u) << 38;
    const unsigned long long L = el ? (unsigned long long)((l & 0x7fffffu) | 0x800000u) << 38 >> ((unsigned)d < 63u ? d : 63) : 0;
    const unsigned long long S = (int)(h ^ l) < 0 ? H - L : H + L;      // [2^60, 2^62 + 2^38)
    const int z = __clz((int)(S >> 32));
    const unsigned long long N = S << z;
    const unsigned long long b = (N >> 11) + ((N >> 10) & 1) + ((unsigned long long)(unsigned)(eh + 897 - z) << 52);
    if (eh == 255) return fv_f2d(v.hi);
    const int hi = eh ? (int)(b >> 32) | (int)(h & 0x80000000u) : 0;
    return __hiloint2double(hi, eh ? (int)b : 0);
  }
};

// A sum of double-float pairs to more bits than binary64 has, rounded to it at
// the end: the high parts error-free in s, their errors and the low parts in the
// pair (m, l).  20 binary32 operations a pair, where a binary64 addition holds
// the FP64 unit for 80 issue slots and needs the pair converted (64 blocks of
// 6..10 cells an axis, one VJP stage 7.37 -> 6.43 ms; 96^3 the same).  The binary64
// parts of a cell's sum apart, in d.
template <class T> struct AdjSum;
template <> struct AdjSum<df64> {
  float s = 0.0f, m = 0.0f, l = 0.0f;
  double d = 0.0;
  __device__ __forceinline__ void set(df64 v) { s = v.hi; m = v.lo; }
  __device__ __forceinline__ void add(double v) { d += v; }
  __device__ __forceinline__ void add(df64 v) {
    const df64 a = two_sum(s, v.hi), b = two_sum(m, v.lo), c = two_sum(b.hi, a.lo);
    s = a.hi;
    m = c.hi;
    l = FADD(l, FADD(b.lo, c.lo));
  }
  __device__ __forceinline__ void sub(df64 v) { add(mk(-v.hi, -v.lo)); }
  __device__ __forceinline__ double value() const {
    const df64 a = two_sum(s, m), b = two_sum(a.lo, l);
    return d + (fv_f2d(a.hi) + AdjMem<df64>::to_d(b));
  }
};
template <> struct AdjSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void set(double v) { s = v; }
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ void sub(double v) { s -= v; }
  __device__ __forceinline__ double value() const { return s; }
};

// Primitive variables of every ghosted cell of the block, once: a face and a
// cell sweep each read a cell's primitives up to twelve times.  (Corner
// ghosts hold no data; nothing reads theirs.)
template <class T>
__global__ void adj_prim_kernel(const FvBlockDev B, const double* __restrict__ qin, const AdjC<T> P,
                                typename AdjMem<T>::type* __restrict__ prim) {
  using S = Sc<T>;
  using M = AdjMem<T>;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < B.plane;
       x += (long long)gridDim.x * blockDim.x) {
    T q[5];
#pragma unroll
    for (int n = 0; n < 5; ++n) q[n] = S::from_d(__ldg(qin + B.qoff + x + n * B.plane));
    const PrimFwd<T> s = prim_fwd(P, q);
    typename M::type* o = prim + B.qoff + x;
    M::st(o, s.r);
    M::st(o + B.plane, s.u);
    M::st(o + 2 * B.plane, s.v);
    M::st(o + 3 * B.plane, s.w);
    M::st(o + 4 * B.plane, s.p);
  }
}

// The faces of direction `dir` of block B, (n_dir + 1) x (the other two
// extents): MUSCL states, then the cotangents of VL and VR from the Roe
// sweep, stored component by component (out[c * nf + f], c = 0..4 for VL,
// 5..9 for VR).  What the MUSCL reconstruction and the primitive recovery
// pass on is taken per cell (adj_cell_kernel), where it is needed once per
// cell and direction instead of four times per face.
template <class T, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) adj_face_kernel(const FvBlockDev B, int dir,
                                                       const typename AdjMem<T>::type* __restrict__ prim,
                                                       const double* __restrict__ lam_out,
                                                       const double* __restrict__ invvol, double alpha_dt,
                                                       const double* __restrict__ metric, const AdjC<T> P,
                                                       typename AdjMem<T>::type* __restrict__ out) {
  using S = Sc<T>;
  using M = AdjMem<T>;
  const int ei = B.ni + (dir == 0), ej = B.nj + (dir == 1), ek = B.nk + (dir == 2);
  const long long nf = (long long)ei * ej * ek;
  const long long ncell_b = (long long)B.ni * B.nj * B.nk;
  const double* lam = lam_out + 5 * B.cell_off;
  const long long f = blockIdx.x * (long long)NT + threadIdx.x;
  if (f >= nf) return;
  const int i = (int)(f % ei), j = (int)((f / ei) % ej), k = (int)(f / ((long long)ei * ej));
  const int g = dir == 0 ? i : (dir == 1 ? j : k);            // face between cells g-1 and g
  const int n_dir = dir == 0 ? B.ni : (dir == 1 ? B.nj : B.nk);
  const long long stride = dir == 0 ? 1 : (dir == 1 ? B.jstride : B.kstride);
  const long long c1 = ghost_index(B, i - (dir == 0), j - (dir == 1), k - (dir == 2));   // cell g-1
  const typename M::type* v = prim + B.qoff + c1;
  T VL[5], VR[5];
#pragma unroll
  for (int n = 0; n < 5; ++n) {
    const T v0 = M::ld(v - stride + n * B.plane), v1 = M::ld(v + n * B.plane);
    const T v2 = M::ld(v + stride + n * B.plane), v3 = M::ld(v + 2 * stride + n * B.plane);
    const T dm = v1 - v0, d0 = v2 - v1, dp = v3 - v2;
    if (P.limiter != 0) {
      VL[n] = v1 + P.e2 * lim_value(P, d0, dm);
      VR[n] = v2 - P.e2 * lim_value(P, d0, dp);
    } else {
      VL[n] = v1 + S::dot2(P.e4km, dm, P.e4kp, d0);
      VR[n] = v2 - S::dot2(P.e4kp, d0, P.e4km, dp);
    }
  }
  // cotangent of the face flux from the two cells' residual cotangents
  double Fd[5] = {0, 0, 0, 0, 0};
  if (g - 1 >= 0) {
    const int il = i - (dir == 0), jl = j - (dir == 1), kl = k - (dir == 2);
    const long long cl = ((long long)kl * B.nj + jl) * B.ni + il;
    const double fac = -alpha_dt * (B.cartesian ? B.cart_invvol : invvol[B.cell_off + cl]);
#pragma unroll
    for (int n = 0; n < 5; ++n) Fd[n] += fac * lam[n * ncell_b + cl];
  }
  if (g < n_dir) {
    const long long cr = ((long long)k * B.nj + j) * B.ni + i;
    const double fac = -alpha_dt * (B.cartesian ? B.cart_invvol : invvol[B.cell_off + cr]);
#pragma unroll
    for (int n = 0; n < 5; ++n) Fd[n] -= fac * lam[n * ncell_b + cr];
  }
  T Fb[5];
#pragma unroll
  for (int n = 0; n < 5; ++n) Fb[n] = S::from_d(Fd[n]);
  T nx, ny, nz, A;
  if (B.cartesian) {
    nx = S::from_d(B.cart_n[dir][0]); ny = S::from_d(B.cart_n[dir][1]); nz = S::from_d(B.cart_n[dir][2]);
    A = S::from_d(B.cart_area[dir]);
  } else {
    const long long fi = B.face_off[dir] + f;
    nx = S::from_d(metric[4 * fi]); ny = S::from_d(metric[4 * fi + 1]);
    nz = S::from_d(metric[4 * fi + 2]); A = S::from_d(metric[4 * fi + 3]);
  }
  T Lb[5], Rb[5];
  roe_vjp(P, VL, VR, nx, ny, nz, A, Fb, Lb, Rb);
#pragma unroll
  for (int n = 0; n < 5; ++n) {
    M::st(out + n * nf + f, Lb[n]);
    M::st(out + (5 + n) * nf + f, Rb[n]);
  }
}

// The slopes of direction `dir`, transposed: cells m = -1 .. n_dir along it
// (those with a face state), interior across it.  The cell's face states are
// V + h and V - h with h the limited half-slope of its forward difference a
// and backward difference b.  With L, R the cotangents of the two (zero where
// the face does not exist), alpha = dh/da (L - R) and beta = dh/db (L - R)
// (the unlimited scheme's two slopes differ), the cell itself gets
// L + R - alpha + beta, the next one alpha, the one before -beta: stored
// component by component (the sum in binary64, the shares as the sweep's type
// has them), one evaluation per cell, direction and variable
// (evaluated three times, by each cell that takes a share, the 96^3 VJP stage
// took 0.98 instead of 0.84 ms in double-float, 4.13 instead of 2.77 in binary64,
// measured before the sums were binary64 again).
template <class T>
__global__ void __launch_bounds__(128) adj_slope_kernel(const FvBlockDev B, int dir,
                                                        const typename AdjMem<T>::type* __restrict__ prim,
                                                        const typename AdjMem<T>::type* __restrict__ cot,
                                                        const AdjC<T> P, typename AdjMem<T>::type* __restrict__ out) {
  using S = Sc<T>;
  using M = AdjMem<T>;
  const int ei = B.ni + (dir == 0), ej = B.nj + (dir == 1), ek = B.nk + (dir == 2);
  const int ci = B.ni + 2 * (dir == 0), cj = B.nj + 2 * (dir == 1), ck = B.nk + 2 * (dir == 2);
  const long long nf = (long long)ei * ej * ek, nc = (long long)ci * cj * ck;
  const long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (x >= nc) return;
  const int i = (int)(x % ci) - (dir == 0), j = (int)((x / ci) % cj) - (dir == 1), k = (int)(x / ((long long)ci * cj)) - (dir == 2);
  const int m = dir == 0 ? i : (dir == 1 ? j : k), n_dir = dir == 0 ? B.ni : (dir == 1 ? B.nj : B.nk);
  const long long st = dir == 0 ? 1 : (dir == 1 ? B.jstride : B.kstride);
  const long long fs = dir == 0 ? 1 : (dir == 1 ? ei : (long long)ei * ej);
  const long long f = ((long long)k * ej + j) * ei + i;          // the cell's lower face
  const typename M::type* v = prim + B.qoff + ghost_index(B, i, j, k);
#pragma unroll 1
  for (int q = 0; q < 5; ++q) {
    const T L = m < n_dir ? M::ld(cot + q * nf + f + fs) : S::c(0.0);
    const T R = m >= 0 ? M::ld(cot + (5 + q) * nf + f) : S::c(0.0);
    const T vm = M::ld(v + q * B.plane - st), v0 = M::ld(v + q * B.plane), vp = M::ld(v + q * B.plane + st);
    T al, be;
    if (P.limiter != 0) {
      T da, db;
      lim_derivatives(P, vp - v0, v0 - vm, da, db);
      const T d = P.e2 * (L - R);
      al = d * da;
      be = d * db;
    } else {
      al = P.e4kp * L - P.e4km * R;
      be = P.e4km * L - P.e4kp * R;
    }
    AdjSum<T> own;
    own.set(L);
    own.add(R);
    own.sub(al - be);
    reinterpret_cast<double*>(out)[q * nc + x] = own.value();
    M::st(out + (5 + q) * nc + x, al);
    M::st(out + (10 + q) * nc + x, be);
  }
}

// The cells' cotangents: the slope kernel's shares in a fixed order (xi, eta,
// zeta; deterministic) and the primitive recovery's transpose, both in binary64
// in either form (summed in double-float it would keep 48 bits, and one 96^3 VJP
// stage with double-float sweeps take 0.76 instead of 0.80 ms).  Into lamg for
// every ghosted cell; or, when no connection has to be transposed (lam_in not
// null), straight to lam_in for the interior cells, with lam_q0 += lam_out.
template <class T>
__global__ void __launch_bounds__(128) adj_cell_kernel(const FvBlockDev B, const typename AdjMem<T>::type* __restrict__ prim,
                                                       const typename AdjMem<T>::type* __restrict__ sx,
                                                       const typename AdjMem<T>::type* __restrict__ sy,
                                                       const typename AdjMem<T>::type* __restrict__ sz, int three_d,
                                                       double gm1, double* __restrict__ lamg,
                                                       const double* __restrict__ lam_out, double* __restrict__ lam_in,
                                                       double* __restrict__ lam_q0) {
  using M = AdjMem<T>;
  const int g = lam_in ? 0 : FV_GHOST;
  const int gi = B.ni + 2 * g, gj = B.nj + 2 * g, gk = B.nk + 2 * g;
  const long long n = (long long)gi * gj * gk;
  const long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (x >= n) return;
  const int i = (int)(x % gi) - g, j = (int)((x / gi) % gj) - g, k = (int)(x / ((long long)gi * gj)) - g;
  const bool ii = i >= 0 && i < B.ni, jj = j >= 0 && j < B.nj, kk = k >= 0 && k < B.nk;
  const long long gx = B.qoff + ghost_index(B, i, j, k);
  AdjSum<T> share[5];
  const T zero = Sc<T>::c(0.0);
#pragma unroll 1
  for (int dir = 0; dir < 2 + three_d; ++dir) {
    if (!(dir == 0 ? jj && kk : (dir == 1 ? ii && kk : ii && jj))) continue;
    const int p = dir == 0 ? i : (dir == 1 ? j : k), nd = dir == 0 ? B.ni : (dir == 1 ? B.nj : B.nk);
    const typename M::type* s = dir == 0 ? sx : (dir == 1 ? sy : sz);
    const double* own = reinterpret_cast<const double*>(s);
    const long long ci = B.ni + 2 * (dir == 0), cj = B.nj + 2 * (dir == 1), ck = B.nk + 2 * (dir == 2);
    const long long nc = ci * cj * ck, st = dir == 0 ? 1 : (dir == 1 ? ci : ci * cj);
    const long long c = ((long long)(k + (dir == 2)) * cj + (j + (dir == 1))) * ci + (i + (dir == 0));
    const bool at = p >= -1 && p <= nd, lo = p >= 0 && p <= nd + 1, up = p >= -2 && p <= nd - 1;
    // all fifteen loads of the direction in flight before the first sum (loaded
    // where each is added, one after the other: 96^3 VJP stage 0.87 instead of 0.80 ms)
    double o[5];
    T a[5], b[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      o[q] = at ? __ldg(own + q * nc + c) : 0.0;
      a[q] = lo ? M::ld(s + (5 + q) * nc + c - st) : zero;
      b[q] = up ? M::ld(s + (10 + q) * nc + c + st) : zero;
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      share[q].add(o[q]);
      share[q].add(a[q]);
      share[q].sub(b[q]);
    }
  }
  double Vb[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) Vb[q] = share[q].value();
  // the cell's primitives and the transpose of the recovery
  using D = Sc<double>;
  const typename M::type* v = prim + gx;
  PrimFwd<double> s;
  s.r = M::to_d(M::ld(v));
  s.u = M::to_d(M::ld(v + B.plane));
  s.v = M::to_d(M::ld(v + 2 * B.plane));
  s.w = M::to_d(M::ld(v + 3 * B.plane));
  s.ri = fx_div(1.0, s.r);   // on the integer units
  s.k = D::dot3(s.u, s.u, s.v, s.v, s.w, s.w);
  double qb[5];
  prim_bwd(gm1, s, Vb, qb);
  if (lam_in) {
    const long long o = 5 * B.cell_off + x;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      lam_in[o + m * n] = qb[m];
      lam_q0[o + m * n] += lam_out[o + m * n];
    }
  } else {
    const bool any = (ii && jj) || (ii && kk) || (jj && kk);
#pragma unroll
    for (int m = 0; m < 5; ++m) lamg[gx + m * B.plane] = any ? qb[m] : 0.0;
  }
}

// transpose of one connection: donor interior cell += ghost cotangent
__global__ void adj_transpose_kernel(const FvBlockDev* __restrict__ blocks, const FvConnDev c, double* lamg) {
  const long long nitems = 2LL * c.L0 * c.L1;
  for (long long it = blockIdx.x * (long long)blockDim.x + threadIdx.x; it < nitems; it += (long long)gridDim.x * blockDim.x) {
    long long local = it;
    const int a = (int)(local % c.L0);
    local /= c.L0;
    const int b = (int)(local % c.L1);
    const int d = (int)(local / c.L1) + 1;
    const FvBlockDev& D = blocks[c.dst_block];
    const FvBlockDev& S = blocks[c.src_block];
    const int da = c.dst_face >> 1, sa = c.src_face >> 1;
    const int dext[3] = {D.ni, D.nj, D.nk}, sext[3] = {S.ni, S.nj, S.nk};
    int dc[3], sc[3];
    const int dt0 = da == 0 ? 1 : 0, dt1 = da == 2 ? 1 : 2;
    const int st0 = sa == 0 ? 1 : 0, st1 = sa == 2 ? 1 : 2;
    dc[dt0] = c.dlo0 + a;
    dc[dt1] = c.dlo1 + b;
    dc[da] = (c.dst_face & 1) ? dext[da] - 1 + d : -d;
    int st[2] = {c.slo0, c.slo1};
    const int u0 = (c.t0 < 0 ? -c.t0 : c.t0) - 1, u1 = (c.t1 < 0 ? -c.t1 : c.t1) - 1;
    st[u0] += c.t0 > 0 ? a : -a;
    st[u1] += c.t1 > 0 ? b : -b;
    sc[st0] = st[0];
    sc[st1] = st[1];
    sc[sa] = (c.src_face & 1) ? sext[sa] - d : d - 1;
    const long long di = D.qoff + ghost_index(D, dc[0], dc[1], dc[2]);
    const long long si = S.qoff + ghost_index(S, sc[0], sc[1], sc[2]);
#pragma unroll
    for (int v = 0; v < 5; ++v) lamg[si + v * S.plane] += lamg[di + v * D.plane];
  }
}

// lam_in <- interior of lamg; lam_q0 += lam_out
__global__ void adj_finish_kernel(const FvBlockDev B, const double* __restrict__ lamg, const double* __restrict__ lam_out,
                                  double* __restrict__ lam_in, double* __restrict__ lam_q0) {
  const long long nc = (long long)B.ni * B.nj * B.nk;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < 5 * nc; x += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(x / nc);
    const long long c = x - v * nc;
    const int i = (int)(c % B.ni), j = (int)((c / B.ni) % B.nj), k = (int)(c / ((long long)B.ni * B.nj));
    const long long o = 5 * B.cell_off + x;
    lam_in[o] = lamg[B.qoff + ghost_index(B, i, j, k) + v * B.plane];
    lam_q0[o] += lam_out[o];
  }
}

int grid_of(long long n, int threads) {
  long long g = (n + threads - 1) / threads;
  return (int)(g < 1 ? 1 : (g > 65535 * 8 ? 65535 * 8 : g));
}

}  // namespace

namespace {
AdjParams adj_params(const FvFaceParams& fp) {
  AdjParams P;
  P.gm1 = fp.gamma - 1.0;
  P.g_gm1 = fp.gamma / (fp.gamma - 1.0);
  P.e4km = fp.eps * 0.25 * (1.0 - fp.kappa);
  P.e4kp = fp.eps * 0.25 * (1.0 + fp.kappa);
  P.e2 = fp.eps * 0.5;
  P.harten = fp.harten;
  P.va_d2 = fp.va_delta2;
  P.limiter = fp.limiter;
  P.fix_all = fp.fix_all;
  return P;
}

template <class T, int MINB>
int adjoint_block(const FvBlockDev& B, int nd, const double* qin, const double* lam_out, const double* invvol,
                  double alpha_dt, const double* const metric[3], const FvFaceParams& fp, void* prim_mem, void* cot_mem,
                  void* slope_mem, double* lamg, double* lam_in, double* lam_q0, cudaStream_t s) {
  using MT = typename AdjMem<T>::type;
  const AdjC<T> P = adj_consts<T>(adj_params(fp));
  MT* prim = static_cast<MT*>(prim_mem);
  MT* cot = static_cast<MT*>(cot_mem);
  adj_prim_kernel<T><<<grid_of(B.plane, 256), 256, 0, s>>>(B, qin, P, prim);
  MT* sl[3] = {static_cast<MT*>(slope_mem), nullptr, nullptr};
  for (int d = 0; d < nd; ++d) {
    const long long nf = (long long)(B.ni + (d == 0)) * (B.nj + (d == 1)) * (B.nk + (d == 2));
    const long long nc = (long long)(B.ni + 2 * (d == 0)) * (B.nj + 2 * (d == 1)) * (B.nk + 2 * (d == 2));
    adj_face_kernel<T, 128, MINB><<<(unsigned)((nf + 127) / 128), 128, 0, s>>>(B, d, prim, lam_out, invvol, alpha_dt,
                                                                             metric[d], P, cot);
    adj_slope_kernel<T><<<(unsigned)((nc + 127) / 128), 128, 0, s>>>(B, d, prim, cot, P, sl[d]);
    if (d < 2) sl[d + 1] = sl[d] + 15 * nc;
  }
  const int g = lam_in ? 0 : FV_GHOST;
  const long long n = (long long)(B.ni + 2 * g) * (B.nj + 2 * g) * (B.nk + 2 * g);
  adj_cell_kernel<T><<<(unsigned)((n + 127) / 128), 128, 0, s>>>(B, prim, sl[0], sl[1], sl[2], nd == 3,
                                                               fp.gamma - 1.0, lamg, lam_out,
                                                               lam_in, lam_q0);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
}  // namespace

int fv_adjoint_block(const FvBlockDev& B, int nd, const double* qin, const double* lam_out, const double* invvol,
                     double alpha_dt, const double* const metric[3], const FvFaceParams& fp, int double_float,
                     void* prim, void* cot, void* slopes, double* lamg, double* lam_in, double* lam_q0, cudaStream_t s) {
  return double_float ? adjoint_block<df64, 4>(B, nd, qin, lam_out, invvol, alpha_dt, metric, fp, prim, cot, slopes, lamg,
                                               lam_in, lam_q0, s)
                      : adjoint_block<double, 3>(B, nd, qin, lam_out, invvol, alpha_dt, metric, fp, prim, cot, slopes,
                                                 lamg, lam_in, lam_q0, s);
}

int fv_adjoint_transpose(const FvBlockDev* d_blocks, const FvConnDev& c, double* lamg, cudaStream_t s) {
  const long long n = 2LL * c.L0 * c.L1;
  adj_transpose_kernel<<<grid_of(n, 256), 256, 0, s>>>(d_blocks, c, lamg);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int fv_adjoint_finish(const FvBlockDev& B, const double* lamg, const double* lam_out, double* lam_in, double* lam_q0,
                      cudaStream_t s) {
  const long long n = 5LL * B.ni * B.nj * B.nk;
  adj_finish_kernel<<<grid_of(n, 256), 256, 0, s>>>(B, lamg, lam_out, lam_in, lam_q0);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
