// C-GBR (Sec. 2.3): characteristic gradient-based reconstruction with MP5
// limiting and the wave-appropriate selection of Eq. (8), HLLC flux of
// Eq. (9)-(10), and the kernels of one RK stage.
#pragma once
#include <type_traits>
#include "cg_device.cuh"

namespace cgk {

struct GbrCfg {
  double gamma, gm1, thr, eps, alpha;
  int window;  // interface sensor window half-width
  float f_gamma, f_gm1, f_thr, f_eps, f_alpha;  // FP32 copies for the mixed form
  Divisor d_gm1;     // gamma - 1 as a divisor (FP64 form)
  int f64_fast;      // the parameters suit gbr_flux_f64
};

// interface frame: unit normal, tangents, averaged state and its sound speed
template <int ND, typename T = double>
struct Frame {
  T n[3], t1[3], t2[3];
  T ha, hb, ic2, cb, cr;
};

// orthonormal tangents of a curvilinear frame (2D: (-n_y, n_x); 3D: t1 from
// the two largest components of n, t2 = n x t1)
template <int ND, typename T = double>
__device__ __forceinline__ void tangents(const T* n, T* t1, T* t2) {
  if (ND == 2) {
    t1[0] = -n[1];
    t1[1] = n[0];
  } else if (ND == 3) {
    int s = 0;
    if (fabs(n[1]) < fabs(n[s])) s = 1;
    if (fabs(n[2]) < fabs(n[s])) s = 2;
    int a = (s + 1) % 3, b = (s + 2) % 3;
    T r = T(1.0) / sqrt(n[a] * n[a] + n[b] * n[b]);
    t1[s] = T(0);
    t1[a] = -n[b] * r;
    t1[b] = n[a] * r;
    t2[0] = n[1] * t1[2] - n[2] * t1[1];
    t2[1] = n[2] * t1[0] - n[0] * t1[2];
    t2[2] = n[0] * t1[1] - n[1] * t1[0];
  }
}

template <int ND, bool CART, int DIR, typename T = double>
__device__ __forceinline__ void to_char(const Frame<ND, T>& f, const T* w, T* c) {
  constexpr int IP = ND + 1;
  T un = sdot<ND, CART, DIR, 0, T>(f.n, w + 1);
  c[0] = f.ha * w[IP] - f.hb * un;
  c[1] = w[0] - f.ic2 * w[IP];
  if (ND >= 2) c[2] = sdot<ND, CART, DIR, 1, T>(f.t1, w + 1);
  if (ND == 3) c[3] = sdot<ND, CART, DIR, 2, T>(f.t2, w + 1);
  c[IP] = f.ha * w[IP] + f.hb * un;
}

template <int ND, bool CART, int DIR, typename T = double>
__device__ __forceinline__ void from_char(const Frame<ND, T>& f, const T* c, T* w) {
  constexpr int IP = ND + 1;
  T s = c[0] + c[IP];
  T un = (c[IP] - c[0]) * f.cr;
  w[0] = c[1] + s;
  w[IP] = (f.cb * f.cb) * s;
#pragma unroll
  for (int m = 0; m < ND; ++m) {
    // u_m = u_n n_m + C3 t1_m + C4 t2_m, structurally zero terms dropped
    T u = T(0);
    bool any = false;
    if (frame_nz(CART, ND, DIR, 0, m)) { u = un * f.n[m]; any = true; }
    if (ND >= 2 && frame_nz(CART, ND, DIR, 1, m)) { u = any ? u + c[2] * f.t1[m] : c[2] * f.t1[m]; any = true; }
    if (ND == 3 && frame_nz(CART, ND, DIR, 2, m)) { u = any ? u + c[3] * f.t2[m] : c[3] * f.t2[m]; any = true; }
    w[1 + m] = u;
  }
}

// HLLC flux (Eq. 9-10) with interface metrics xi (not normalised);
// g2 = |xi|^2, g = |xi|, ig2 = 1/|xi|^2 supplied by the caller.
template <int ND, bool CART, int DIR, typename T = double>
__device__ __forceinline__ void hllc(T gamma, T gm1, const T* WL, const T* WR, const T* xi, T g2, T g, T ig2, T* F) {
  constexpr int IP = ND + 1;
  T rL = WL[0], pL = WL[IP], rR = WR[0], pR = WR[IP];
  T UL = sdot<ND, CART, DIR, 0, T>(xi, WL + 1);
  T UR = sdot<ND, CART, DIR, 0, T>(xi, WR + 1);
  T qL = WL[1] * WL[1], qR = WR[1] * WR[1];
#pragma unroll
  for (int m = 1; m < ND; ++m) {
    qL = qL + WL[1 + m] * WL[1 + m];
    qR = qR + WR[1 + m] * WR[1 + m];
  }
  T EL = pL / gm1 + T(0.5) * rL * qL;
  T ER = pR / gm1 + T(0.5) * rR * qR;
  T cL = sqrt(gamma * pL / rL), cR = sqrt(gamma * pR / rR);
  T sL = sqrt(rL), sR = sqrt(rR);
  T iden = T(1.0) / (sL + sR);
  T uh[3];
#pragma unroll
  for (int m = 0; m < ND; ++m) uh[m] = (sL * WL[1 + m] + sR * WR[1 + m]) * iden;
  T qh = uh[0] * uh[0];
#pragma unroll
  for (int m = 1; m < ND; ++m) qh = qh + uh[m] * uh[m];
  T Uh = sdot<ND, CART, DIR, 0, T>(xi, uh);
  T HL = (EL + pL) / rL, HR = (ER + pR) / rR;
  T Hh = (sL * HL + sR * HR) * iden;
  T ch = sqrt(gm1 * (Hh - T(0.5) * qh));
  T SL = dmin(UL - cL * g, Uh - ch * g);
  T SR = dmax(UR + cR * g, Uh + ch * g);
  T Ss = (rR * UR * (SR - UR) - rL * UL * (SL - UL) + (pL - pR) * g2) / (rR * (SR - UR) - rL * (SL - UL));
  const T* W;
  T S, U, E, r, p;
  bool star;
  if (T(0) <= SL) { W = WL; S = T(0); U = UL; E = EL; r = rL; p = pL; star = false; }
  else if (T(0) <= Ss) { W = WL; S = SL; U = UL; E = EL; r = rL; p = pL; star = true; }
  else if (T(0) <= SR) { W = WR; S = SR; U = UR; E = ER; r = rR; p = pR; star = true; }
  else { W = WR; S = T(0); U = UR; E = ER; r = rR; p = pR; star = false; }
  // convective flux of the chosen side (Eq. 2)
  T FK[ND + 2];
  FK[0] = r * U;
#pragma unroll
  for (int m = 0; m < ND; ++m)
    FK[1 + m] = frame_nz(CART, ND, DIR, 0, m) ? r * W[1 + m] * U + xi[m] * p : r * W[1 + m] * U;
  FK[IP] = (E + p) * U;
  if (!star) {
#pragma unroll
    for (int v = 0; v < ND + 2; ++v) F[v] = FK[v];
    return;
  }
  T fac = r * (S - U) / (S - Ss);
  T d = Ss - U;
  F[0] = FK[0] + S * (fac - r);
#pragma unroll
  for (int m = 0; m < ND; ++m) {
    T qs = frame_nz(CART, ND, DIR, 0, m) ? fac * (W[1 + m] + xi[m] * d * ig2) : fac * W[1 + m];
    F[1 + m] = FK[1 + m] + S * (qs - r * W[1 + m]);
  }
  T qe = fac * (E / r + d * (Ss * ig2 + p / (r * (S - U))));
  F[IP] = FK[IP] + S * (qe - E);
}

// Flux at one interface i+1/2 from the stencil W_{i-2..i+3}, the gradients
// W'_{i,i+1}, second derivatives W''_{i,i+1}, whether the interface's sensor is
// above its threshold (disc) and the interface metrics.  Wave order: 0 = u_n - c, 1 = entropy, 2.. = shear,
// last = u_n + c.
template <int ND, bool CART, int DIR, typename T = double>
__device__ __forceinline__ void gbr_flux(const GbrCfg& q, const DevGrid& g, const T (&Wst)[6][ND + 2],
                                         const T (&Wd)[2][ND + 2], const T (&Wdd)[2][ND + 2], bool disc,
                                         const T* xi, T* F) {
  constexpr int NV = ND + 2, IP = ND + 1;
  const T c12 = T(1.0 / 12.0);
  const T gamma = gconst<T>(q.gamma, q.f_gamma), gm1 = gconst<T>(q.gm1, q.f_gm1),
          alpha = gconst<T>(q.alpha, q.f_alpha), eps = gconst<T>(q.eps, q.f_eps);
  Frame<ND, T> fr;
  T g2, gg, ig2;
  if (CART) {
    g2 = gconst<T>(g.cg2[DIR], g.f_cg2[DIR]);
    gg = gconst<T>(g.cg[DIR], g.f_cg[DIR]);
    ig2 = gconst<T>(g.cig2[DIR], g.f_cig2[DIR]);
#pragma unroll
    for (int m = 0; m < ND; ++m) {
      fr.n[m] = gconst<T>(g.cn[DIR][m], g.f_cn[DIR][m]);
      fr.t1[m] = gconst<T>(g.ct1[DIR][m], g.f_ct1[DIR][m]);
      fr.t2[m] = gconst<T>(g.ct2[DIR][m], g.f_ct2[DIR][m]);
    }
  } else {
    g2 = xi[0] * xi[0];
#pragma unroll
    for (int m = 1; m < ND; ++m) g2 = g2 + xi[m] * xi[m];
    gg = sqrt(g2);
    T ig = T(1.0) / gg;
    ig2 = T(1.0) / g2;
#pragma unroll
    for (int m = 0; m < ND; ++m) fr.n[m] = xi[m] * ig;
    tangents<ND, T>(fr.n, fr.t1, fr.t2);
  }
  T rb = T(0.5) * (Wst[2][0] + Wst[3][0]);
  T pb = T(0.5) * (Wst[2][IP] + Wst[3][IP]);
  fr.cb = sqrt(gamma * pb / rb);
  T ic = T(1.0) / fr.cb;
  fr.ic2 = ic * ic;
  fr.ha = T(0.5) * fr.ic2;
  fr.hb = T(0.5) * rb * ic;
  fr.cr = fr.cb / rb;

  T C[6][NV], Cd[2][NV], Cdd[2][NV];
#pragma unroll
  for (int j = 0; j < 6; ++j) to_char<ND, CART, DIR, T>(fr, Wst[j], C[j]);
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    to_char<ND, CART, DIR, T>(fr, Wd[j], Cd[j]);
    to_char<ND, CART, DIR, T>(fr, Wdd[j], Cdd[j]);
  }
  T CL[NV], CR[NV];
#pragma unroll
  for (int b = 0; b < NV; ++b) {
    T v0 = C[0][b], v1 = C[1][b], v2 = C[2][b], v3 = C[3][b], v4 = C[4][b], v5 = C[5][b];
    T cl = v2 + T(0.5) * Cd[0][b] + Cdd[0][b] * c12;
    T cr = v3 - T(0.5) * Cd[1][b] + Cdd[1][b] * c12;
    if (b == 0 || b == IP) {  // acoustic: sensor
      if (disc) {
        CL[b] = mp5(v0, v1, v2, v3, v4, alpha, eps);
        CR[b] = mp5(v5, v4, v3, v2, v1, alpha, eps);
      } else {
        CL[b] = cl;
        CR[b] = cr;
      }
    } else if (b == 1) {      // entropy: MP criterion
      T cc = T(0.5) * (cl + cr);
      T umpL = v2 + minmod2(v3 - v2, alpha * (v2 - v1));
      CL[b] = ((cl - v2) * (cl - umpL) > eps) ? mp5(v0, v1, v2, v3, v4, alpha, eps) : cc;
      T umpR = v3 + minmod2(v2 - v3, alpha * (v3 - v4));
      CR[b] = ((cr - v3) * (cr - umpR) > eps) ? mp5(v5, v4, v3, v2, v1, alpha, eps) : cc;
    } else {                  // shear: sensor
      if (disc) {
        CL[b] = mp5(v0, v1, v2, v3, v4, alpha, eps);
        CR[b] = mp5(v5, v4, v3, v2, v1, alpha, eps);
      } else {
        T cc = T(0.5) * (cl + cr);
        CL[b] = cc;
        CR[b] = cc;
      }
    }
  }
  T WL[NV], WR[NV];
  from_char<ND, CART, DIR, T>(fr, CL, WL);
  from_char<ND, CART, DIR, T>(fr, CR, WR);
  if (WL[0] <= T(0) || WL[IP] <= T(0) || WR[0] <= T(0) || WR[IP] <= T(0)) {
#pragma unroll
    for (int v = 0; v < NV; ++v) { WL[v] = Wst[2][v]; WR[v] = Wst[3][v]; }
  }
  T xl[3];
  if (CART) {
#pragma unroll
    for (int m = 0; m < ND; ++m) xl[m] = (m == DIR) ? gconst<T>(g.cxh[DIR], g.f_cxh[DIR]) : T(0);
  } else {
#pragma unroll
    for (int m = 0; m < ND; ++m) xl[m] = xi[m];
  }
  hllc<ND, CART, DIR, T>(gamma, gm1, WL, WR, xl, g2, gg, ig2, F);
}

// ---------------------------------------------------------------- FP64 form
// The same flux in FP64, value for value what gbr_flux gives, with fewer
// instructions on the FP64 pipe, which bounds the sweep (2 a clock an SM):
//   * divisions and square roots on the integer and FP32 pipes (cg_fp64.cuh);
//   * a product with a power of two is exact, so x - 2 y, x + y/2 and the like
//     are one fused multiply-add, and the factor 2 of the second derivatives
//     and of 1/c^2 = 2 (1/(2 c^2)) is carried along instead of multiplied;
//   * comparisons, minima and minmods on the bit patterns;
//   * the characteristic variables of the outer stencil nodes only where MP5
//     reads them (the acoustic and shear waves of a flagged interface, the
//     entropy wave where Eq. (8) limits it);
//   * products with a factor known to be in range on the integer pipes (IM);
//   * on a Cartesian grid whose unit normals are exactly 1 (UN) no
//     multiplication by them.
// Measured (triple point 1792 x 768, MEG6, with the staging and the epilogue):
// FP64 instructions an interface 569 -> 278 without the products on the integer
// pipes, 181 to 200 with them; the sweep 1.51 -> 0.76 -> 0.61 ms a launch, the
// whole step 9.98 -> 5.23 -> 4.19 ms.
// Returns false where an operand is out of the range of these forms (a state
// that is not positive, NaN, extreme magnitudes): the caller then repeats the
// interface, with plain products if it had them on the integer pipes, or with
// gbr_flux.
// (mp5's value; the range tests of its operands go to R)
__device__ __forceinline__ double mp5_f64(double um2, double um1, double u0, double up1, double up2, double alpha,
                                          double eps, F64Range& R) {
  // 60 = 1.875 2^5: B, 2^105 / B, 1 / 1.875 and the exponent word of div_by
  const Divisor sixty{0x001e000000000000ull, 0x0011111111111111ull, 0.53333333333f, 0x40400000u};
  double ul = __fma_rn(2.0, um2, -(13.0 * um1)) + 47.0 * u0 + 27.0 * up1 - 3.0 * up2;
  R.any0(ul);
  ul = div_by(ul, sixty);
  const double dm = u0 - um1, dp = up1 - u0, adm = alpha * dm;
  const double ump = u0 + minmod_f64(dp, adm);
  if (bits64((ul - u0) * (ul - ump)) <= bits64(eps)) return ul;
  const double dm1 = __fma_rn(-2.0, um1, um2) + u0;
  const double d0 = __fma_rn(-2.0, u0, um1) + up1;
  const double dp1 = __fma_rn(-2.0, up1, u0) + up2;
  const double dm4p = minmod_f64(minmod_f64(__fma_rn(4.0, d0, -dp1), __fma_rn(4.0, dp1, -d0)), minmod_f64(d0, dp1));
  const double dm4m = minmod_f64(minmod_f64(__fma_rn(4.0, d0, -dm1), __fma_rn(4.0, dm1, -d0)), minmod_f64(d0, dm1));
  const double uul = u0 + adm;
  const double umd = 0.5 * ((u0 + up1) - dm4p);
  const double ulc = __fma_rn(0.5, dm, u0) + (4.0 / 3.0) * dm4m;
  const long long k0 = order_key(u0), k1 = order_key(up1), kd = order_key(umd), kl = order_key(uul), kc = order_key(ulc);
  const double umin = from_key(kmax(kmin(kmin(k0, k1), kd), kmin(kmin(k0, kl), kc)));
  const double umax = from_key(kmin(kmax(kmax(k0, k1), kd), kmax(kmax(k0, kl), kc)));
  return ul + minmod_f64(umin - ul, umax - ul);
}

// The left and right MP5 states of one wave from its stencil v0..v5: a
// function of its own, so that the sweep holds its code once (few warps take
// it, and inlined for every wave and side it would crowd the instruction cache).
struct Mp5Pair {
  double L, R;
  unsigned worst;
};
static __device__ __noinline__ Mp5Pair mp5_pair_f64(double v0, double v1, double v2, double v3, double v4, double v5,
                                                    double alpha, double eps) {
  F64Range R;
  Mp5Pair o;
  o.L = mp5_f64(v0, v1, v2, v3, v4, alpha, eps, R);
  o.R = mp5_f64(v5, v4, v3, v2, v1, alpha, eps, R);
  o.worst = R.worst;
  return o;
}

// sum_m a[m] u[m] over the structurally non-zero a[m], in index order (sdot)
template <int ND, bool CART, int DIR, int VEC, class PR>
__device__ __forceinline__ double sdot_f64(const PR& P, const double* a, const double* u) {
  double s = 0.0;
  bool first = true;
#pragma unroll
  for (int m = 0; m < ND; ++m) {
    if (!frame_nz(CART, ND, DIR, VEC, m)) continue;
    const double t = CART ? P.kz(a[m], u[m]) : P.zz(a[m], u[m]);
    s = first ? t : s + t;
    first = false;
  }
  return s;
}

// characteristic variables of a primitive vector (to_char's values)
template <int ND, bool CART, int DIR, bool UN, class PR>
__device__ __forceinline__ void to_char_f64(const PR& P, const Frame<ND, double>& f, const double* w,
                                            double* c) {
  static_assert(!UN || ND <= 2, "exact unit normals: 1D and 2D");
  constexpr int IP = ND + 1;
  const double un = UN ? by_sign(f.n[DIR], w[1 + DIR]) : sdot_f64<ND, CART, DIR, 0>(P, f.n, w + 1);
  const double a = P.kz(f.ha, w[IP]), b = P.kz(f.hb, un);
  c[0] = a - b;
  c[1] = __fma_rn(-2.0, a, w[0]);
  c[IP] = a + b;
#pragma unroll
  for (int m = 0; m < ND; ++m)
    if (UN && ND >= 2 && frame_nz(CART, ND, DIR, 1, m)) c[2] = by_sign(f.t1[m], w[1 + m]);
  if (!UN && ND >= 2) c[2] = sdot_f64<ND, CART, DIR, 1>(P, f.t1, w + 1);
  if (!UN && ND == 3) c[3] = sdot_f64<ND, CART, DIR, 2>(P, f.t2, w + 1);
}

// from_char's values; cb2 = cb^2
template <int ND, bool CART, int DIR, bool UN, class PR>
__device__ __forceinline__ void from_char_f64(const PR& P, const Frame<ND, double>& f, double cb2,
                                              const double* c, double* w) {
  constexpr int IP = ND + 1;
  const double s = c[0] + c[IP];
  const double un = P.kz(f.cr, c[IP] - c[0]);
  w[0] = c[1] + s;
  w[IP] = P.kz(cb2, s);
#pragma unroll
  for (int m = 0; m < ND; ++m) {
    if (UN) {
      if (m == DIR) w[1 + m] = by_sign(f.n[m], un);
      else w[1 + m] = by_sign(f.t1[m], c[2]);
      continue;
    }
    auto t = [&](double a, double b) { return CART ? P.kz(a, b) : P.zz(a, b); };
    double u = 0.0;
    bool any = false;
    if (frame_nz(CART, ND, DIR, 0, m)) { u = t(f.n[m], un); any = true; }
    if (ND >= 2 && frame_nz(CART, ND, DIR, 1, m)) { u = any ? u + t(f.t1[m], c[2]) : t(f.t1[m], c[2]); any = true; }
    if (ND == 3 && frame_nz(CART, ND, DIR, 2, m)) { u = any ? u + t(f.t2[m], c[3]) : t(f.t2[m], c[3]); any = true; }
    w[1 + m] = u;
  }
}

template <int ND, bool CART, int DIR, class PR>
__device__ __forceinline__ void hllc_f64(const PR& P, const GbrCfg& q, const double* WL, const double* WR, const double* xi,
                                         double g2, double g, double ig2, double* F, F64Range& R) {
  constexpr int IP = ND + 1;
  auto xm = [&](double a, double b) { return CART ? P.kz(a, b) : P.zz(a, b); };  // by a metric component
  const double rL = WL[0], pL = WL[IP], rR = WR[0], pR = WR[IP];
  R.pos(rL);
  R.pos(pL);
  R.pos(rR);
  R.pos(pR);
  const double UL = sdot_f64<ND, CART, DIR, 0>(P, xi, WL + 1);
  const double UR = sdot_f64<ND, CART, DIR, 0>(P, xi, WR + 1);
  double SL, SR, EL, ER;
  {
    double qL = P.zz(WL[1], WL[1]), qR = P.zz(WR[1], WR[1]);
#pragma unroll
    for (int m = 1; m < ND; ++m) {
      qL = qL + P.zz(WL[1 + m], WL[1 + m]);
      qR = qR + P.zz(WR[1 + m], WR[1 + m]);
    }
    EL = __fma_rn(0.5, P.kz(rL, qL), div_by(pL, q.d_gm1));
    ER = __fma_rn(0.5, P.kz(rR, qR), div_by(pR, q.d_gm1));
    double cL, cR, HL, HR;
    {
      const Divisor D = divisor(rL);
      const double HN = EL + pL;
      R.any0(HN);
      cL = sqrt_ranged(div_by(P.kk(q.gamma, pL), D));
      HL = div_by(HN, D);
    }
    {
      const Divisor D = divisor(rR);
      const double HN = ER + pR;
      R.any0(HN);
      cR = sqrt_ranged(div_by(P.kk(q.gamma, pR), D));
      HR = div_by(HN, D);
    }
    const double sL = sqrt_ranged(rL), sR = sqrt_ranged(rR);
    const double iden = rcp_by(divisor(sL + sR));
    double uh[3];
#pragma unroll
    for (int m = 0; m < ND; ++m) uh[m] = P.kz(iden, P.kz(sL, WL[1 + m]) + P.kz(sR, WR[1 + m]));
    double qh = P.zz(uh[0], uh[0]);
#pragma unroll
    for (int m = 1; m < ND; ++m) qh = qh + P.zz(uh[m], uh[m]);
    const double Uh = sdot_f64<ND, CART, DIR, 0>(P, xi, uh);
    const double Hh = P.kz(iden, P.kz(sL, HL) + P.kz(sR, HR));
    const double c2 = P.kz(q.gm1, __fma_rn(-0.5, qh, Hh));
    R.pos(c2);
    const double chg = P.kk(g, sqrt_ranged(c2));
    SL = min_f64(UL - P.kk(g, cL), Uh - chg);
    SR = max_f64(UR + P.kk(g, cR), Uh + chg);
  }
  double Ss;
  {
    const double eR = SR - UR, eL = SL - UL;
    const double num = P.zz(P.kz(rR, UR), eR) - P.zz(P.kz(rL, UL), eL) + P.kz(g2, pL - pR),
                 den = P.kz(rR, eR) - P.kz(rL, eL);
    R.any0(num);
    R.any(den);
    Ss = div_by(num, divisor(den));
  }
  // the first of 0 <= SL, 0 <= S*, 0 <= SR that holds decides (S* may exceed SR
  // where gamma is near 1)
  const bool left = nonneg(SL) || nonneg(Ss);
  const bool star = !nonneg(SL) && (nonneg(Ss) || nonneg(SR));
  double W[ND];
#pragma unroll
  for (int m = 0; m < ND; ++m) W[m] = left ? WL[1 + m] : WR[1 + m];
  const double r = left ? rL : rR, p = left ? pL : pR, U = left ? UL : UR, E = left ? EL : ER, S = left ? SL : SR;
  double ru[ND];
  F[0] = P.kz(r, U);
#pragma unroll
  for (int m = 0; m < ND; ++m) {
    ru[m] = P.kz(r, W[m]);
    F[1 + m] = P.zz(ru[m], U);
    if (frame_nz(CART, ND, DIR, 0, m)) F[1 + m] = F[1 + m] + xm(xi[m], p);
  }
  F[IP] = P.zz(E + p, U);
  if (!star) return;
  const double SU = S - U, rSU = P.kz(r, SU), SS = S - Ss, d = Ss - U;
  R.any(rSU);
  R.any(SS);
  R.any0(E);
  const double fac = div_by(rSU, divisor(SS));
  F[0] = F[0] + P.zz(S, fac - r);
#pragma unroll
  for (int m = 0; m < ND; ++m) {
    const double qs =
        P.zz(fac, frame_nz(CART, ND, DIR, 0, m) ? W[m] + P.kz(ig2, xm(xi[m], d)) : W[m]);
    F[1 + m] = F[1 + m] + P.zz(S, qs - ru[m]);
  }
  const double qe = P.zz(fac, div_by(E, divisor(r)) + P.zz(d, P.kz(ig2, Ss) + div_by(p, divisor(rSU))));
  F[IP] = F[IP] + P.zz(S, qe - E);
}

template <class PR>
__device__ __forceinline__ PR make_products(F64Range& R) {
  if constexpr (std::is_same_v<PR, F64Products>) return F64Products{R};
  else return PR{};
}

// IM: products on the integer pipes (a contracting unit fuses them instead).
// W(j, w): the primitives of stencil node i-2+j (j = 0..5); Wd(j, w), Wh(j, w):
// first derivatives and halved second derivatives of node i+j (j = 0, 1).
template <int ND, bool CART, int DIR, bool UN, bool IM, class FW, class FD, class FH>
__device__ __forceinline__ bool gbr_flux_f64(const GbrCfg& q, const DevGrid& g, FW ldW, FD ldD, FH ldH, bool disc,
                                             const double* xi, double* F) {
  constexpr int NV = ND + 2, IP = ND + 1;
  if (!q.f64_fast) return false;  // at once: the caller's IEEE form is all that is paid
  F64Range R;
  using PR = std::conditional_t<IM, F64Products, PlainProducts>;
  const PR P = make_products<PR>(R);
  Frame<ND, double> fr;
  double g2, gg, ig2, xl[3];
  if (CART) {
    g2 = g.cg2[DIR];
    gg = g.cg[DIR];
    ig2 = g.cig2[DIR];
#pragma unroll
    for (int m = 0; m < ND; ++m) {
      fr.n[m] = g.cn[DIR][m];
      fr.t1[m] = g.ct1[DIR][m];
      fr.t2[m] = g.ct2[DIR][m];
      xl[m] = m == DIR ? g.cxh[DIR] : 0.0;
    }
  } else {
#pragma unroll
    for (int m = 0; m < ND; ++m) xl[m] = xi[m];
    g2 = xi[0] * xi[0];
#pragma unroll
    for (int m = 1; m < ND; ++m) g2 = g2 + xi[m] * xi[m];
    R.pos(g2);
    gg = sqrt_ranged(g2);
    const double ig = rcp_by(divisor(gg));
    ig2 = rcp_by(divisor(g2));
#pragma unroll
    for (int m = 0; m < ND; ++m) fr.n[m] = xi[m] * ig;
    if (ND == 2) {
      fr.t1[0] = -fr.n[1];
      fr.t1[1] = fr.n[0];
    } else if (ND == 3) {  // tangents(): t1 from the two largest components of n, t2 = n x t1
      const double* n = fr.n;
      int s = 0;
      if (order_key(fabs(n[1])) < order_key(fabs(n[0]))) s = 1;
      if (order_key(fabs(n[2])) < order_key(fabs(s == 1 ? n[1] : n[0]))) s = 2;
      const double na = s == 0 ? n[1] : (s == 1 ? n[2] : n[0]), nb = s == 0 ? n[2] : (s == 1 ? n[0] : n[1]);
      const double r = rcp_by(divisor(sqrt_ranged(na * na + nb * nb)));
      const double ta = -nb * r, tb = na * r;
      fr.t1[0] = s == 0 ? 0.0 : (s == 1 ? tb : ta);
      fr.t1[1] = s == 0 ? ta : (s == 1 ? 0.0 : tb);
      fr.t1[2] = s == 0 ? tb : (s == 1 ? ta : 0.0);
      fr.t2[0] = n[1] * fr.t1[2] - n[2] * fr.t1[1];
      fr.t2[1] = n[2] * fr.t1[0] - n[0] * fr.t1[2];
      fr.t2[2] = n[0] * fr.t1[1] - n[1] * fr.t1[0];
    }
  }
  double w2[NV], w3[NV];
  ldW(2, w2);
  ldW(3, w3);
  double cb2;
  {
    const double rs = w2[0] + w3[0], ps = w2[IP] + w3[IP];  // twice the averaged density and pressure
    R.pos(rs);
    R.pos(ps);
    const Divisor D = divisor(rs);
    fr.cb = sqrt_ranged(div_by(P.kk(q.gamma, ps), D));
    const double ic = rcp_by(divisor(fr.cb));
    fr.ic2 = P.kk(ic, ic);
    fr.ha = scale2<-1>(fr.ic2);
    fr.hb = scale2<-2>(P.kk(rs, ic));
    fr.cr = scale2<1>(div_by(fr.cb, D));
    cb2 = P.kk(fr.cb, fr.cb);
    R.any(fr.ha);
    R.any(fr.hb);
    R.any(fr.cr);
    R.any(cb2);
  }
  double CL[NV], CR[NV], C2[NV], C3[NV];
  to_char_f64<ND, CART, DIR, UN>(P, fr, w2, C2);
  to_char_f64<ND, CART, DIR, UN>(P, fr, w3, C3);
  const double c6 = 2.0 * (1.0 / 12.0);
  {
    double w[NV], c[NV];
    ldD(0, w);
    to_char_f64<ND, CART, DIR, UN>(P, fr, w, c);
#pragma unroll
    for (int b = 0; b < NV; ++b) CL[b] = __fma_rn(0.5, c[b], C2[b]);
    ldH(0, w);
    to_char_f64<ND, CART, DIR, UN>(P, fr, w, c);
#pragma unroll
    for (int b = 0; b < NV; ++b) CL[b] = CL[b] + P.kz(c6, c[b]);
    ldD(1, w);
    to_char_f64<ND, CART, DIR, UN>(P, fr, w, c);
#pragma unroll
    for (int b = 0; b < NV; ++b) CR[b] = __fma_rn(-0.5, c[b], C3[b]);
    ldH(1, w);
    to_char_f64<ND, CART, DIR, UN>(P, fr, w, c);
#pragma unroll
    for (int b = 0; b < NV; ++b) CR[b] = CR[b] + P.kz(c6, c[b]);
  }
  {  // entropy wave: MP criterion
    auto entropy = [&](int j) {
      double w[NV];
      ldW(j, w);
      return __fma_rn(-2.0, P.kz(fr.ha, w[IP]), w[0]);
    };
    const double v1 = entropy(1), v2 = C2[1], v3 = C3[1], v4 = entropy(4);
    const double cl = CL[1], cr = CR[1], cc = 0.5 * (cl + cr), dv = v3 - v2;
    const double umpL = v2 + minmod_f64(dv, P.zz(q.alpha, v2 - v1));
    const double umpR = v3 + minmod_f64(-dv, P.zz(q.alpha, v3 - v4));
    const double tL = P.zz(cl - v2, cl - umpL), tR = P.zz(cr - v3, cr - umpR);
    // finite and above eps
    const bool limL = bits64(tL) > bits64(q.eps) && __double2hiint(tL) < 0x7ff00000;
    const bool limR = bits64(tR) > bits64(q.eps) && __double2hiint(tR) < 0x7ff00000;
    CL[1] = cc;
    CR[1] = cc;
    if (limL || limR) {
      const Mp5Pair m = mp5_pair_f64(entropy(0), v1, v2, v3, v4, entropy(5), q.alpha, q.eps);
      R.see(m.worst);
      if (limL) CL[1] = m.L;
      if (limR) CR[1] = m.R;
    }
  }
  if (!disc) {  // acoustic waves upwind, shear waves central
#pragma unroll
    for (int b = 2; b < IP; ++b) {
      const double cc = 0.5 * (CL[b] + CR[b]);
      CL[b] = cc;
      CR[b] = cc;
    }
  } else {
    double C0[NV], C1[NV], C4[NV], C5[NV], w[NV];
    ldW(0, w);
    to_char_f64<ND, CART, DIR, UN>(P, fr, w, C0);
    ldW(1, w);
    to_char_f64<ND, CART, DIR, UN>(P, fr, w, C1);
    ldW(4, w);
    to_char_f64<ND, CART, DIR, UN>(P, fr, w, C4);
    ldW(5, w);
    to_char_f64<ND, CART, DIR, UN>(P, fr, w, C5);
#pragma unroll
    for (int b = 0; b < NV; ++b) {
      if (b == 1) continue;
      const Mp5Pair m = mp5_pair_f64(C0[b], C1[b], C2[b], C3[b], C4[b], C5[b], q.alpha, q.eps);
      R.see(m.worst);
      CL[b] = m.L;
      CR[b] = m.R;
    }
  }
  double WL[NV], WR[NV];
  from_char_f64<ND, CART, DIR, UN>(P, fr, cb2, CL, WL);
  from_char_f64<ND, CART, DIR, UN>(P, fr, cb2, CR, WR);
  hllc_f64<ND, CART, DIR>(P, q, WL, WR, xl, g2, gg, ig2, F, R);
  return R.ok();
}

}  // namespace cgk
