// recon64.cuh -- the 2D FP64 reconstruction of one field (Sec. 2.2 Steps 1-3, Eq. 2.23), shared
// by the FP64 kernels of every equation (stage2d_char64.cuh, stage2d_comp64.cuh), in the
// arithmetic of f64_ops.cuh and arranged for few FP64 operations:
//  * the constant term of the combined polynomial from its cell average (which every p_m
//    shares, Eq. 2.5): c_{0,0} is never formed;
//  * coefficients scaled by (sqrt(15)/10)^degree, so that the interior Gauss points lie at -1,
//    0, 1 and are sums of coefficients, the edges' taken from shared even and odd parts;
//  * beta_0 of Eq. 2.20 completed to squares by parity class, where most cross terms vanish:
//    34 operations instead of 46 (the same quadratic form, still a sum of squares);
//  * the weights as the four sums of b_m that the slopes of the combined polynomial need.
#pragma once
#include "f64_ops.cuh"
#include "hweno_device.cuh"

namespace hw {

namespace c64 {

constexpr double S1 = 0.38729833462074168852;  // sqrt(15)/10, the outer Gauss node
constexpr double S2 = 0.15, S3 = S1 * 0.15, S4 = 0.0225;

// S1 .. S4 are those of the coordinates: scaled here, 1 in namespace plain
#define HW_C64_CONSTANTS(X)                                                                   \
  X(ONE, 1.0) X(MZERO, -0.0)                                                                  \
  /* beta_0 */                                                                                \
  X(B_A8, S1 / (12.0 * S3)) X(B_A6, S1 / (4.0 * S3)) X(B_W1, 1.0 / S2)                        \
  X(B_W6, 781.0 / (20.0 * S3 * S3)) X(B_W8, 47.0 / (10.0 * S3 * S3))                          \
  X(B_C12, S2 / (12.0 * S4)) X(B_C10, 63.0 * S2 / (130.0 * S4))                               \
  X(B_W3, 13.0 / (3.0 * S2 * S2)) X(B_W10, 1421461.0 / (2275.0 * S4 * S4))                    \
  X(B_W12, 5083.0 * 144.0 / (270.0 * S2 * S2)) X(B_E, 17.0 * S2 / (70.0 * S4))                \
  X(B_W4, 7.0 / (6.0 * S2 * S2)) X(B_WP, 710728.0 / (33600.0 * S4 * S4))                      \
  X(B_WM, 710730.0 / (33600.0 * S4 * S4))                                                     \
  /* weights */                                                                               \
  X(W_TAU, 25.0 / 16.0) X(MTWO, -2.0)                                                         \
  /* evaluation */                                                                            \
  X(M12, -25.0 / 81.0) X(MX, -5.0 / 9.0) X(V8, 1.0 / (144.0 * S3)) X(V6, 1.0 / (80.0 * S3))   \
  X(V1, 1.0 / (12.0 * S1)) X(H1, 0.5 / S1) X(H2, 0.25 / S2) X(H3, 0.125 / S3)                 \
  X(H4, 0.0625 / S4)                                                                          \
  /* the Appendix coefficients */                                                             \
  X(MFOUR, -4.0) X(A1X, S1 / 48.0) X(A1E, -397.0 / 456.0 * S1) X(A1V, -75.0 / 19.0 * S1)      \
  X(A6E, 5.0 / 19.0 * S3) X(A6V, 60.0 / 19.0 * S3) X(A8X, -0.25 * S3) X(A8E, 0.5 * S3)        \
  X(A4X, -7.0 / 22.0 * S2) X(A4V, 75.0 / 11.0 * S2) X(A11X, 5.0 / 22.0 * S4)                  \
  X(A11V, -60.0 / 11.0 * S4) X(A3R, -S2 / 48.0) X(A3Q, S2 / 24.0) X(A3P, 71.0 / 48.0 * S2)    \
  X(A3V, -45.0 / 8.0 * S2) X(A10P, -5.0 / 8.0 * S4) X(A10V, 15.0 / 4.0 * S4)                  \
  X(A12R, 0.25 * S4) X(A12P, -0.5 * S4)                                                       \
  /* cell, volume and faces */                                                                \
  X(HALF, 0.5) X(WC, 25.0 / 324.0) X(WE, 10.0 / 81.0) X(WM, 16.0 / 81.0)                      \
  X(RS2, 0.375) X(THREEQ, 0.75) X(QUARTER, 0.25) X(THIRD, 1.0 / 3.0) X(TWOTHIRD, 2.0 / 3.0)
enum Const : int {
#define X(name, value) k##name,
  HW_C64_CONSTANTS(X)
#undef X
  kStatic,             // from here on: values of the problem, written at the start of an item
  kEPS = kStatic, kGLO, kG0, kSGLO, kGM1, kHGM1, kGAM, kAX, kAY, kIDX, kFX0, kFX1, kFX2, kIDY,
  kFY0, kFY1, kFY2, kCount
};
static __constant__ double c64_constants[kStatic] = {
#define X(name, value) (value),
    HW_C64_CONSTANTS(X)
#undef X
};
// the same in unscaled coordinates, for the FP32-bulk kernels, whose smoothness indicators and
// weights are evaluated in FP64 by the functions below
namespace plain {
constexpr double S1 = 1.0, S2 = 1.0, S3 = 1.0, S4 = 1.0;
static __constant__ double constants[kStatic] = {
#define X(name, value) (value),
    HW_C64_CONSTANTS(X)
#undef X
};
}  // namespace plain
constexpr int kTable = (kCount + 7) / 8 * 8;  // doubles of shared memory

#define K(name) o.k<c64::k##name>()

// the table of an item (visible after the caller's next __syncthreads)
template <bool SCALED = true>
__device__ __forceinline__ void fill_table(double* tab, const KProblem& P) {
  const int t = threadIdx.x;
  for (int n = t; n < kStatic; n += blockDim.x)
    tab[n] = SCALED ? c64_constants[n] : plain::constants[n];
  if (t == 0) {
    tab[kEPS] = 25.0 * P.eps;  // d_m is scaled by 25, the squared divisor of u_ave
    tab[kGLO] = P.glo;
    tab[kG0] = P.g0[1];
    tab[kSGLO] = (SCALED ? S1 : 1.0) * P.glo;
    tab[kGM1] = P.gm1;
    tab[kHGM1] = -0.5 * P.gm1;
    tab[kGAM] = P.gam;
    tab[kAX] = P.ax;
    tab[kAY] = P.ay;
    // Gauss moments of a face from twice its flux, divided by the cell size
    tab[kIDX] = P.inv_dx;
    tab[kFX0] = 5.0 / 36.0 * P.inv_dx;
    tab[kFX1] = 2.0 / 9.0 * P.inv_dx;
    tab[kFX2] = 5.0 / 36.0 * S1 * P.inv_dx;
    tab[kIDY] = P.inv_dy;
    tab[kFY0] = 5.0 / 36.0 * P.inv_dy;
    tab[kFY1] = 2.0 / 9.0 * P.inv_dy;
    tab[kFY2] = 5.0 / 36.0 * S1 * P.inv_dy;
  }
}

// beta_0 of Eq. 2.20 from the scaled coefficients c[1..14]
__device__ __forceinline__ double beta0(const Ops& o, const double (&c)[15]) {
  // odd in one coordinate: (c1 + c6/4 + c8/12)^2 + 781/20 c6^2 + 47/10 c8^2, and c2, c9, c7
  const double k8 = K(B_A8), k6 = K(B_A6);
  const double ta = fma(k8, c[8], fma(k6, c[6], c[1]));
  const double tb = fma(k8, c[7], fma(k6, c[9], c[2]));
  double b = o.mul(K(B_W1), fma(tb, tb, o.mul(ta, ta)));
  b = fma(K(B_W6), fma(c[9], c[9], o.mul(c[6], c[6])), b);
  b = fma(K(B_W8), fma(c[7], c[7], o.mul(c[8], c[8])), b);
  // even in both: 13/3 (c3 + 63/130 c10 + c12/12)^2 + 1421461/2275 c10^2, c5, c14, and c12^2
  const double c12 = o.mul(K(B_C12), c[12]), k10 = K(B_C10);
  const double tc = fma(k10, c[10], o.add(c[3], c12));
  const double td = fma(k10, c[14], o.add(c[5], c12));
  b = fma(K(B_W3), fma(td, td, o.mul(tc, tc)), b);
  b = fma(K(B_W10), fma(c[14], c[14], o.mul(c[10], c[10])), b);
  b = fma(o.mul(K(B_W12), c12), c12, b);
  // odd in both: 7/6 (c4 + 17/70 (c11 + c13))^2 + 42.3.. (c11^2 + c13^2) - c11 c13 / 8400
  const double p = o.add(c[11], c[13]), m = o.sub(c[11], c[13]);
  const double te = fma(K(B_E), p, c[4]);
  b = fma(o.mul(K(B_W4), te), te, b);
  b = fma(o.mul(K(B_WP), p), p, b);
  b = fma(o.mul(K(B_WM), m), m, b);
  return b;
}

// The factors of the combined polynomial (Eq. 2.23): a0 of p_0 and, for the slopes of p_1..p_4
// (el, er: u5 - u4, u6 - u5; eb, et: u5 - u2, u8 - u5; in scaled coordinates), the sums
// b1 + b3 (of el), b2 + b4 (er), b1 + b2 (eb), b3 + b4 (et), b_m = omega_m - a0 gamma_m.
struct Factors {
  double a0, l, r, b, t;
};

// the sum of |averages| of cells 2, 4, 5, 6, 8 (5 sqrt(u_ave)) from the cell's own, w5, and the
// one-sided differences; w5 = 0 where ZERO_MEAN
template <bool ZERO_MEAN>
__device__ __forceinline__ double average_sum(const Ops& o, const double (&e)[4], double w5) {
  if constexpr (ZERO_MEAN)
    return o.add(o.add(fabs(e[0]), fabs(e[1])), o.add(fabs(e[2]), fabs(e[3])));
  else
    return o.add(o.add(o.add(fabs(o.sub(w5, e[0])), fabs(o.add(w5, e[1]))),
                       o.add(fabs(o.sub(w5, e[2])), fabs(o.add(w5, e[3])))), fabs(w5));
}

// Eq. 2.20-2.22 from beta_0, the one-sided differences e = {el, er, eb, et} and a, the average
// sum: the product form of hweno_device.cuh's nonlinear_weights_fast with d_m scaled by 25 (the
// squared divisor of u_ave), as far as its users share it.
struct Products {
  double b1, b2, b3, b4;  // beta_m of the linear polynomials
  double D0, A, B, d1, d2, d3, d4;  // D_1 = A d2, D_2 = A d1, D_3 = B d4, D_4 = B d3
  double N0, inv, tau;                       // a0 = N0 inv
  bool ok;  // the products stay in the double range

  // q = D_1 + .. + D_4 by sum(*this); INT: the reciprocal on integers
  template <bool INT, class Sum>
  __device__ __forceinline__ void set(const Ops& o, double bt0, const double (&e)[4], double a,
                                      const KProblem& P, Sum sum) {
    const double el2 = o.mul(e[0], e[0]), er2 = o.mul(e[1], e[1]), eb2 = o.mul(e[2], e[2]),
                 et2 = o.mul(e[3], e[3]);
    b1 = o.add(el2, eb2);
    b2 = o.add(er2, eb2);
    b3 = o.add(el2, et2);
    b4 = o.add(er2, et2);
    const double s = o.add(o.add(fabs(o.sub(bt0, b1)), fabs(o.sub(bt0, b2))),
                           o.add(fabs(o.sub(bt0, b3)), fabs(o.sub(bt0, b4))));
    tau = o.mul(o.mul(K(W_TAU), s), s);  // 25 tau
    double ua = o.mul(a, a);             // 25 u_ave
    if (P.wmode == 1) ua = 25.0;
    const double eps = K(EPS);
    const double d0 = fma(bt0, ua, eps);
    d1 = fma(b1, ua, eps);
    d2 = fma(b2, ua, eps);
    d3 = fma(b3, ua, eps);
    d4 = fma(b4, ua, eps);
    const double p12 = o.mul(d1, d2), p34 = o.mul(d3, d4);
    D0 = o.mul(p12, p34);
    const double D = o.mul(D0, d0);
    A = o.mul(d0, p34);
    B = o.mul(d0, p12);
    const double q = sum(*this);
    N0 = fma(tau, D0, D);
    const double S = fma(tau, fma(K(GLO), q, o.mul(K(G0), D0)), D);
    const int eD = (__double2hiint(D) >> 20) & 0x7ff, eS = (__double2hiint(S) >> 20) & 0x7ff;
    ok = eD > 64 && eD < 2047 - 64 && eS > 64 && eS < 2047 - 64;
    inv = INT ? rcp_in_range(S) : rcp_in_range(o, S);
  }
};

// The factors; false where the products left the double range and the direct formula was used.
__device__ __forceinline__ bool factors(const Ops& o, double bt0, const double (&e)[4], double a,
                                        const KProblem& P, Factors& F) {
  Products p;
  double q12, q34, q13, q24;
  p.set<true>(o, bt0, e, a, P, [&](const Products& x) {
    q12 = o.mul(x.A, o.add(x.d1, x.d2));
    q34 = o.mul(x.B, o.add(x.d3, x.d4));
    q13 = fma(x.A, x.d2, o.mul(x.B, x.d4));
    q24 = fma(x.A, x.d1, o.mul(x.B, x.d3));
    return o.add(q12, q34);
  });
  const bool lin = P.wmode == 2;
  const double k = o.mul(K(SGLO), o.mul(p.tau, p.inv));
  const double k0 = o.mul(K(MTWO), o.mul(k, p.D0));
  F.a0 = lin ? 1.0 : o.mul(p.N0, p.inv);
  F.l = lin ? 0.0 : fma(k, q13, k0);
  F.r = lin ? 0.0 : fma(k, q24, k0);
  F.b = lin ? 0.0 : fma(k, q12, k0);
  F.t = lin ? 0.0 : fma(k, q34, k0);
  if (p.ok || lin) return true;
  const double beta[5] = {bt0, p.b1, p.b2, p.b3, p.b4};
  double bm[5];
  nonlinear_weights_direct<5>(beta, 0.04 * (a * a), P, F.a0, bm);
  F.l = S1 * (bm[1] + bm[3]);
  F.r = S1 * (bm[2] + bm[4]);
  F.b = S1 * (bm[1] + bm[2]);
  F.t = S1 * (bm[3] + bm[4]);
  return false;
}
// The same as a0 and the single b_1..b_4, in unscaled coordinates.
__device__ __forceinline__ bool weights(const Ops& o, double bt0, const double (&e)[4], double a,
                                        const KProblem& P, double& a0, double (&b)[5]) {
  Products p;
  double D1, D2, D3, D4;
  p.set<false>(o, bt0, e, a, P, [&](const Products& x) {
    D1 = o.mul(x.A, x.d2);
    D2 = o.mul(x.A, x.d1);
    D3 = o.mul(x.B, x.d4);
    D4 = o.mul(x.B, x.d3);
    return o.add(o.add(D1, D2), o.add(D3, D4));
  });
  const bool lin = P.wmode == 2;
  const double k = o.mul(K(GLO), o.mul(p.tau, p.inv)), k0 = -o.mul(k, p.D0);
  a0 = lin ? 1.0 : o.mul(p.N0, p.inv);
  b[1] = lin ? 0.0 : fma(k, D1, k0);
  b[2] = lin ? 0.0 : fma(k, D2, k0);
  b[3] = lin ? 0.0 : fma(k, D3, k0);
  b[4] = lin ? 0.0 : fma(k, D4, k0);
  if (p.ok || lin) return true;
  const double beta[5] = {bt0, p.b1, p.b2, p.b3, p.b4};
  nonlinear_weights_direct<5>(beta, 0.04 * (a * a), P, a0, b);
  return false;
}

// The 14 stencil combinations that the Appendix coefficients of one component are formed from:
//  0 X1, 1 Va, 2 X2, 3 Wa, 4 X3, 5 v8 - v2, 6 w6 - w4, 7 corners - 4 u5, 8 Vd, 9 Wd,
//  10 u5 - u4, 11 u6 - u5, 12 u5 - u2, 13 u8 - u5
// from the component's window rows below, at and above the cell (m0, m1, m2 at the column left of
// it; its x and y first moments WC and 2 WC further on).
template <int WC, class Out>
__device__ __forceinline__ void combinations(const Ops& o, const double* m0, const double* m1,
                                             const double* m2, Out s) {
  const double u1 = m0[0], u3 = m0[2], u7 = m2[0], u9 = m2[2];
  const double sb = o.add(u1, u3), st = o.add(u7, u9), db = o.sub(u1, u3), dt = o.sub(u7, u9);
  s(0, o.add(db, dt));
  s(2, o.sub(sb, st));
  s(4, o.sub(db, dt));
  const double u5 = m1[1];
  s(7, fma(K(MFOUR), u5, o.add(sb, st)));
  s(10, o.sub(u5, m1[0]));
  s(11, o.sub(m1[2], u5));
  s(12, o.sub(u5, m0[1]));
  s(13, o.sub(m2[1], u5));
  const double v4 = m1[WC], v6 = m1[WC + 2];
  s(1, o.add(v4, v6));
  s(8, o.sub(v6, v4));
  s(5, o.sub(m2[WC + 1], m0[WC + 1]));
  const double z2 = m0[2 * WC + 1], z8 = m2[2 * WC + 1];
  s(3, o.add(z2, z8));
  s(9, o.sub(z8, z2));
  s(6, o.sub(m1[2 * WC + 2], m1[2 * WC]));
}
// The scaled Appendix coefficients from combinations 0..9 (s(n)) and the differences e of 10..13.
template <class In>
__device__ __forceinline__ void coefficients(const Ops& o, In s, const double (&e)[4],
                                             double (&C)[15]) {
  {
    const double X1 = s(0), Va = s(1), ex = -o.add(e[0], e[1]);
    const double X2 = s(2), Wa = s(3), ey = -o.add(e[2], e[3]);
    const double kx = K(A1X), ke = K(A1E), kv = K(A1V);
    C[1] = fma(kv, Va, fma(ke, ex, o.mul(kx, X1)));
    C[2] = fma(kv, Wa, fma(ke, ey, o.mul(kx, X2)));
    const double k6 = K(A6E), k6v = K(A6V);
    C[6] = fma(k6v, Va, o.mul(k6, ex));
    C[9] = fma(k6v, Wa, o.mul(k6, ey));
    const double k8 = K(A8X), k8e = K(A8E);
    C[8] = fma(k8e, ex, o.mul(k8, X1));
    C[7] = fma(k8e, ey, o.mul(k8, X2));
  }
  {
    const double X3 = s(4), v82 = s(5), w64 = s(6);
    C[4] = fma(K(A4X), X3, o.mul(K(A4V), o.add(v82, w64)));
    const double x = o.mul(K(A11X), X3), kv = K(A11V);
    C[11] = fma(kv, v82, x);
    C[13] = fma(kv, w64, x);
  }
  {
    const double r = s(7), Vd = s(8), Wd = s(9);
    const double p = o.sub(e[1], e[0]), q = o.sub(e[3], e[2]);
    const double rr = o.mul(K(A3R), r), kq = K(A3Q), kp = K(A3P), kv = K(A3V);
    C[3] = fma(kv, Vd, fma(kp, p, fma(kq, q, rr)));
    C[5] = fma(kv, Wd, fma(kp, q, fma(kq, p, rr)));
    const double k10 = K(A10P), k10v = K(A10V);
    C[10] = fma(k10v, Vd, o.mul(k10, p));
    C[14] = fma(k10v, Wd, o.mul(k10, q));
    const double k12 = K(A12P);
    C[12] = fma(k12, q, fma(k12, p, o.mul(K(A12R), r)));
  }
}

// Index of the coefficient that plays the role of n when the coordinates change places.
template <int DIR>
__device__ __forceinline__ constexpr int role(int n) {
  return DIR == 0 ? n
                  : (n == 1 ? 2 : n == 2 ? 1 : n == 3 ? 5 : n == 5 ? 3 : n == 6 ? 9 : n == 9 ? 6
                     : n == 7 ? 8 : n == 8 ? 7 : n == 10 ? 14 : n == 14 ? 10 : n == 11 ? 13
                     : n == 13 ? 11 : n);
}

// the constant term of the polynomial with cell average `mean`
__device__ __forceinline__ double constant_term(const Ops& o, const double (&C)[15], double mean) {
  return fma(K(M12), C[12], fma(K(MX), o.add(o.add(C[3], C[10]), o.add(C[5], C[14])), mean));
}
// the first-moment modification of direction DIR
template <int DIR>
__device__ __forceinline__ double vhat(const Ops& o, const double (&C)[15]) {
  return fma(K(V8), C[role<DIR>(8)], fma(K(V6), C[role<DIR>(6)], o.mul(K(V1), C[role<DIR>(1)])));
}
// values on the two edges normal to direction DIR, at the three Gauss points along them
// (C[0] set): lo = {(-1/2, -s), (-1/2, 0), (-1/2, s)}, hi the same at +1/2
template <int DIR>
__device__ __forceinline__ void edges(const Ops& o, const double (&C)[15], double (&lo)[3],
                                      double (&hi)[3]) {
#define CC(n) C[role<DIR>(n)]
  const double h = K(H1), h2 = K(H2), h3 = K(H3);
  const double E0 = fma(K(H4), CC(10), fma(h2, CC(3), C[0]));
  const double O0 = fma(h3, CC(6), o.mul(h, CC(1)));
  const double Ev = o.add(E0, fma(h2, CC(12), o.add(CC(5), CC(14))));
  const double Od = fma(h, CC(8), O0);
  const double Eo = o.add(fma(h2, CC(7), CC(2)), CC(9));
  const double Oo = fma(h3, CC(11), o.mul(h, o.add(CC(4), CC(13))));
#undef CC
  const double Pp = o.add(Ev, Oo), Pm = o.sub(Ev, Oo), Qp = o.add(Od, Eo), Qm = o.sub(Od, Eo);
  hi[2] = o.add(Pp, Qp);   // (+, +): even + odd-even + even-odd + odd-odd
  lo[0] = o.sub(Pp, Qp);   // (-, -)
  hi[0] = o.add(Pm, Qm);   // (+, -)
  lo[2] = o.sub(Pm, Qm);   // (-, +)
  hi[1] = o.add(E0, O0);
  lo[1] = o.sub(E0, O0);
}
// values at the nine interior Gauss points, index 3 (1 + xi/s) + (1 + eta/s)
__device__ __forceinline__ void interior(const Ops& o, const double (&C)[15], double (&in)[9]) {
  const double ex = o.add(C[3], C[10]), ey = o.add(C[5], C[14]);
  const double EX = o.add(C[0], ex), EY = o.add(C[0], ey);
  const double EE = o.add(o.add(EX, ey), C[12]);
  const double ox = o.add(C[1], C[6]), oy = o.add(C[2], C[9]);
  const double OE = o.add(ox, C[8]), EO = o.add(oy, C[7]);
  const double OO = o.add(C[4], o.add(C[11], C[13]));
  const double Pp = o.add(EE, OO), Pm = o.sub(EE, OO), Qp = o.add(OE, EO), Qm = o.sub(OE, EO);
  in[8] = o.add(Pp, Qp);
  in[0] = o.sub(Pp, Qp);
  in[6] = o.add(Pm, Qm);
  in[2] = o.sub(Pm, Qm);
  in[7] = o.add(EX, ox);
  in[1] = o.sub(EX, ox);
  in[5] = o.add(EY, oy);
  in[3] = o.sub(EY, oy);
  in[4] = C[0];
}

// hweno_device.cuh's euler_speeds<2> in these operations: false where the average is not
// admissible.
__device__ __forceinline__ bool speeds(const Ops& o, const double (&u)[4], double& s0, double& s1) {
  const double ir = rcp_any(u[0]);
  const double vx = o.mul(u[1], ir), vy = o.mul(u[2], ir);
  const double e = fma(-K(HALF), fma(u[1], vx, o.mul(u[2], vy)), u[3]);
  const double c2 = o.mul(o.mul(o.mul(K(GAM), K(GM1)), e), ir);
  const double c = sqrt_any(o, c2, K(HALF), K(RS2));
  s0 = o.add(fabs(vx), c);
  s1 = o.add(fabs(vy), c);
  return u[0] > 0.0 && e > 0.0 && finite_bits(e);
}

}  // namespace c64

}  // namespace hw
