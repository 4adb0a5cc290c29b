// stage2d_char64.cuh -- one work item of the fused 2D stage for the Euler equations with the
// local characteristic decomposition in FP64 (Sec. 2.2, Remark 2.2, Eq. 2.16, 2.23, 2.13):
// the same decomposition into bands and row chunks as stage2d_item.cuh, with the arithmetic
// arranged for the fewest FP64 operations, which bound it.
//
// What the arrangement uses, all exact identities of the scheme's formulas:
//  * the cell's own Galilean frame.  With q = m - u rho and E' = E - u.q - u^2 rho / 2 (u the
//    velocity of the cell's average), the characteristic variables are X/2 -+ q_n/(2c),
//    W1 = rho - X and q_t, X = (gamma-1)/c^2 E'.  The frame is linear in the state, so it is
//    applied to the 14 stencil combinations the Appendix coefficients are formed from, once
//    for both passes; and W1 (the entropy field) is the same field in both passes, so it is
//    reconstructed once per cell: seven fields instead of eight;
//  * the constant term of the combined polynomial from its cell average (which every p_m
//    shares, Eq. 2.5): c_{0,0} is never formed;
//  * coefficients scaled by (sqrt(15)/10)^degree, so that the interior Gauss points lie at -1,
//    0, 1 and are sums of coefficients, the edges' taken from shared even and odd parts;
//  * beta_0 of Eq. 2.20 completed to squares by parity class, where most cross terms vanish:
//    34 operations instead of 46 (the same quadratic form, still a sum of squares);
//  * the volume integrals of f and g in the cell's frame: the Gauss rule integrates the linear
//    parts exactly (the polynomial's average is the cell average), so only the sums of
//    q_n^2/rho, q_n q_t/rho, ... over the nine points are left, and the frame is undone once
//    per cell instead of per point.
#pragma once
#include "hweno_device.cuh"

namespace hw {

namespace c64 {

constexpr double S1 = 0.38729833462074168852;  // sqrt(15)/10, the outer Gauss node
constexpr double S2 = 0.15, S3 = S1 * 0.15, S4 = 0.0225;

// The FP64 unit takes 16 clocks per warp for a DFMA whose three operands are vector registers
// and 19 for a DADD, a DMUL or a DFMA with a constant or uniform operand (measured: 2.00 and
// 1.68 lanes per clock and SM, whatever the number of warps).  So every operation here is a
// three-register DFMA: a + b = a 1 + b, a b = a b + (-0), both exact, with 1 and -0 held in
// registers, and the constants are read from shared memory into registers at each use, through
// an address that depends on the thread (a provably uniform one would be loaded into a uniform
// register).  2048^2 stage: 21.2 ms with plain operators, 18.8 ms so.
#define HW_C64_CONSTANTS(X)                                                                   \
  X(ONE, 1.0) X(NZERO, -0.0)                                                                  \
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
  X(THREEQ, 0.75) X(QUARTER, 0.25) X(THIRD, 1.0 / 3.0) X(TWOTHIRD, 2.0 / 3.0)
enum Const : int {
#define X(name, value) k##name,
  HW_C64_CONSTANTS(X)
#undef X
  kStatic,             // from here on: values of the problem, written at the start of an item
  kEPS = kStatic, kGLO, kG0, kSGLO, kGM1, kHGM1, kGAM, kIDX, kFX0, kFX1, kFX2, kFY0, kFY1, kFY2,
  kIDY, kCount
};
static __constant__ double c64_constants[kStatic] = {
#define X(name, value) (value),
    HW_C64_CONSTANTS(X)
#undef X
};
constexpr int kTable = (kCount + 7) / 8 * 8;  // doubles of shared memory

struct Ops {
  double one, nz;
  unsigned tab;  // shared address of the table (+ 0 for every thread, which no pass can prove)
  template <int I>
  __device__ __forceinline__ double k() const {
    double v;  // volatile: a constant is loaded where it is used, not kept in registers
    asm volatile("ld.shared.f64 %0, [%1+%2];" : "=d"(v) : "r"(tab), "n"(8 * I));
    return v;
  }
  __device__ __forceinline__ double add(double a, double b) const { return fma(a, one, b); }
  __device__ __forceinline__ double sub(double a, double b) const { return fma(-b, one, a); }
  __device__ __forceinline__ double mul(double a, double b) const { return fma(a, b, nz); }
};
#define K(name) o.k<k##name>()

// the table of an item (visible after the caller's next __syncthreads)
__device__ __forceinline__ void fill_table(double* tab, const KProblem& P) {
  const int t = threadIdx.x;
  static_assert(kStatic <= 64, "one entry per thread of the narrowest block");
  if (t < kStatic) tab[t] = c64_constants[t];
  if (t == 0) {
    tab[kEPS] = 25.0 * P.eps;  // d_m is scaled by 25, the squared divisor of u_ave
    tab[kGLO] = P.glo;
    tab[kG0] = P.g0[1];
    tab[kSGLO] = S1 * P.glo;
    tab[kGM1] = P.gm1;
    tab[kHGM1] = -0.5 * P.gm1;
    tab[kGAM] = P.gam;
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

// 1/x of a normal double with exponent field in [1, 2044]: the hardware's 20-bit reciprocal,
// refined by one third-order step y + y (e + e^2), e = 1 - x y (the new residual e^3 < 2^-59).
__device__ __forceinline__ double rcp_in_range(const Ops& o, double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, o.one);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rcp_any(const Ops& o, double x) {
  const int eb = (int)(((unsigned long long)__double_as_longlong(x) >> 52) & 0x7ff);
  if (eb < 1 || eb > 2044) return 1.0 / x;
  return rcp_in_range(o, x);
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

// Eq. 2.20-2.22 from beta_0 and the one-sided differences e = {el, er, eb, et}; w5 the field's
// cell average (zero where ZERO_MEAN).  The product form of hweno_device.cuh's
// nonlinear_weights_fast, in the sums the combination needs and with d_m scaled by 25 (the
// squared divisor of u_ave); the direct formula where the products leave the double range.
template <bool ZERO_MEAN>
__device__ __forceinline__ bool factors(const Ops& o, double bt0, const double (&e)[4], double w5,
                                        const KProblem& P, Factors& F) {
  const double el2 = o.mul(e[0], e[0]), er2 = o.mul(e[1], e[1]), eb2 = o.mul(e[2], e[2]),
               et2 = o.mul(e[3], e[3]);
  const double b1 = o.add(el2, eb2), b2 = o.add(er2, eb2), b3 = o.add(el2, et2),
               b4 = o.add(er2, et2);
  const double s = o.add(o.add(fabs(o.sub(bt0, b1)), fabs(o.sub(bt0, b2))),
                         o.add(fabs(o.sub(bt0, b3)), fabs(o.sub(bt0, b4))));
  const double tau = o.mul(o.mul(K(W_TAU), s), s);  // 25 tau
  double a;
  if constexpr (ZERO_MEAN)
    a = o.add(o.add(fabs(e[0]), fabs(e[1])), o.add(fabs(e[2]), fabs(e[3])));
  else
    a = o.add(o.add(o.add(fabs(o.sub(w5, e[0])), fabs(o.add(w5, e[1]))),
                    o.add(fabs(o.sub(w5, e[2])), fabs(o.add(w5, e[3])))), fabs(w5));
  double ua = o.mul(a, a);  // 25 u_ave
  if (P.wmode == 1) ua = 25.0;
  const double eps = K(EPS);
  const double d0 = fma(bt0, ua, eps), d1 = fma(b1, ua, eps), d2 = fma(b2, ua, eps),
               d3 = fma(b3, ua, eps), d4 = fma(b4, ua, eps);
  const double p12 = o.mul(d1, d2), p34 = o.mul(d3, d4);
  const double D0 = o.mul(p12, p34), D = o.mul(D0, d0);
  const double A = o.mul(d0, p34), B = o.mul(d0, p12);  // D1 = A d2, D2 = A d1, D3 = B d4, D4 = B d3
  const double q12 = o.mul(A, o.add(d1, d2)), q34 = o.mul(B, o.add(d3, d4));
  const double q13 = fma(A, d2, o.mul(B, d4));
  const double q = o.add(q12, q34), q24 = o.sub(q, q13);
  const double N0 = fma(tau, D0, D);
  const double S = fma(tau, fma(K(GLO), q, o.mul(K(G0), D0)), D);
  const long long eD = (__double_as_longlong(D) >> 52) & 0x7ff;
  const long long eS = (__double_as_longlong(S) >> 52) & 0x7ff;
  const bool ok = eD > 64 && eD < 2047 - 64 && eS > 64 && eS < 2047 - 64;
  const bool lin = P.wmode == 2;
  const double inv = rcp_in_range(o, S);
  const double k = o.mul(K(SGLO), o.mul(tau, inv));
  const double k0 = o.mul(K(MTWO), o.mul(k, D0));
  F.a0 = lin ? 1.0 : o.mul(N0, inv);
  F.l = lin ? 0.0 : fma(k, q13, k0);
  F.r = lin ? 0.0 : fma(k, q24, k0);
  F.b = lin ? 0.0 : fma(k, q12, k0);
  F.t = lin ? 0.0 : fma(k, q34, k0);
  if (ok || lin) return true;
  const double beta[5] = {bt0, b1, b2, b3, b4};
  double bm[5];
  nonlinear_weights_direct<5>(beta, 0.04 * (a * a), P, F.a0, bm);
  F.l = S1 * (bm[1] + bm[3]);
  F.r = S1 * (bm[2] + bm[4]);
  F.b = S1 * (bm[1] + bm[2]);
  F.t = S1 * (bm[3] + bm[4]);
  return false;
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

}  // namespace c64

// Shared memory of a block, in doubles per thread column (and 36 more for the two columns the
// row window adds): the window [3 rows][12][BW + 2]; the x-face exchange [12][BW] (f - a1 u of
// each cell's left trace, then the Gauss moments of the face's flux); g + a2 u of the top
// traces carried to the next row [12][BW]; the coefficients of X/2, q_x, q_y [42][BW]; the
// entropy field's point values and modifications [23][BW]; and the table of constants.
template <int BW>
constexpr size_t smem_bytes_char64() {
  return sizeof(double) * (36 * (BW + 2) + (12 + 12 + 42 + 23) * BW + c64::kTable);
}

template <int BW>
__device__ __forceinline__ void stage2d_char64_item(const KProblem& P, const KStage& S, int band,
                                                    int j0, int j1, int wout, double* smem,
                                                    double (*red)[BW / 32]) {
  using namespace c64;
  constexpr int NC = 4, NA = 12, WC = BW + 2;
  const int t = threadIdx.x;
  double* win = smem;
  double* xch = win + 3 * NA * WC;
  double* car = xch + 12 * BW + t;       // this thread's column
  double* cf = xch + 24 * BW + t;        // this thread's column: X/2 (0-13), q_x, q_y
  double* w1p = cf + 42 * BW;            // this thread's column: W1 on x edges, y edges, inside
  double* tab = xch + (24 + 42 + 23) * BW;
  fill_table(tab, P);
  const int nx = P.nx, ny = P.ny;
  const size_t plane = (size_t)nx * ny;
  const int i0 = band * wout;
  const int i = i0 - 1 + t;
  const bool need = (t <= wout + 1) && (i <= nx);
  const bool outc = (t >= 1 && t <= wout && i < nx);
  const double a1 = S.alpha_in[0], a2 = S.alpha_in[1];
  const double dt = *S.dt;

  // window column t of a row is loaded by thread t, the two last columns by threads 0..23
  int fx0, fx1;
  const int ii0 = bc_map(i0 - 2 + t, nx, P.bc[0], P.bc[1], fx0);
  const int ii1 = bc_map(i0 - 2 + BW + t / NA, nx, P.bc[0], P.bc[1], fx1);
  auto load_row = [&](int r) {
    int fy;
    const int rr = bc_map(r, ny, P.bc[2], P.bc[3], fy);
    double* dst = win + ((r + 3) % 3) * NA * WC;  // r >= -2
    const double* src = S.Uin + (size_t)rr * nx;
    double v[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) v[a] = src[(size_t)a * plane + ii0];
    const int a1_ = t % NA;
    double v1 = 0.0;
    if (t < 2 * NA) v1 = src[(size_t)a1_ * plane + ii1];
    if (fx0 | fy) {
#pragma unroll
      for (int a = 0; a < NA; ++a) v[a] *= mirror_sign<EQ_EULER, 2>(a / 3, a % 3, fx0, fy);
    }
    if (t < 2 * NA && (fx1 | fy)) v1 *= mirror_sign<EQ_EULER, 2>(a1_ / 3, a1_ % 3, fx1, fy);
#pragma unroll
    for (int a = 0; a < NA; ++a) dst[a * WC + t] = v[a];
    if (t < 2 * NA) dst[a1_ * WC + BW + t / NA] = v1;
  };
#pragma unroll 1
  for (int r = j0 - 2; r <= j0; ++r) load_row(r);
  __syncthreads();
  Ops o;
  o.tab = (unsigned)__cvta_generic_to_shared(tab) + (unsigned)((S.k >> 2) * t);  // k <= 3: + 0
  o.one = K(ONE);
  o.nz = K(NZERO);

  double pend[NC][3];              // F^1..F^3 of (i, j-1) without its top face
  double pvh[NC], pwh[NC];         // v-hat, w-hat of (i, j-1)
#pragma unroll
  for (int c = 0; c < NC; ++c) pend[c][0] = pend[c][1] = pend[c][2] = pvh[c] = pwh[c] = 0.0;
  double wmax0 = 0.0, wmax1 = 0.0;
  bool fast = true;

#pragma unroll 1
  for (int j = j0 - 1; j <= j1; ++j) {
    const double* wm = win + ((j + 2) % 3) * NA * WC;  // j >= -1
    const double* w0 = win + ((j + 3) % 3) * NA * WC;
    const double* wp = win + ((j + 4) % 3) * NA * WC;
    const bool xrow = (j >= j0 && j < j1);

    // the cell's frame
    double vx = 0.0, vy = 0.0, q2h = 0.0, p5 = 0.0, c2 = 0.0, c = 0.0, h = 0.0, hic = 0.0, X5 = 0.0;
    double dX[4], dqx[4], dqy[4];  // X/2, q_x, q_y of u5 - u4, u6 - u5, u5 - u2, u8 - u5
    if (need) {
      double b1h;
      {
        const double U0 = w0[0 * WC + t + 1], U1 = w0[3 * WC + t + 1], U2 = w0[6 * WC + t + 1],
                     U3 = w0[9 * WC + t + 1];
        const double ir = rcp_any(o, U0);
        vx = o.mul(U1, ir);
        vy = o.mul(U2, ir);
        q2h = o.mul(K(HALF), fma(vx, vx, o.mul(vy, vy)));
        p5 = o.mul(K(GM1), fma(-U0, q2h, U3));
        c2 = o.mul(o.mul(K(GAM), p5), ir);
        const double rc = rsqrt(c2);
        c = o.mul(c2, rc);
        h = fma(o.add(U3, p5), ir, -q2h);
        hic = o.mul(K(HALF), rc);
        const double rc2 = o.mul(rc, rc);
        b1h = -o.mul(K(HGM1), rc2);
        X5 = o.mul(p5, rc2);
      }
      // the 14 stencil combinations of the conserved components
      //  0 X1, 1 Va, 2 X2, 3 Wa, 4 X3, 5 v82, 6 w64, 7 corners - 4 u5, 8 Vd, 9 Wd,
      //  10 u5 - u4, 11 u6 - u5, 12 u5 - u2, 13 u8 - u5
#pragma unroll
      for (int a = 0; a < NC; ++a) {
        double* s = a == 0 ? w1p : cf + (a == 3 ? 0 : 14 * a) * BW;
        const double* m0 = wm + 3 * a * WC + t;
        const double* m1 = w0 + 3 * a * WC + t;
        const double* m2 = wp + 3 * a * WC + t;
        const double u1 = m0[0], u3 = m0[2], u7 = m2[0], u9 = m2[2];
        const double sb = o.add(u1, u3), st = o.add(u7, u9), db = o.sub(u1, u3),
                     dtp = o.sub(u7, u9);
        s[0 * BW] = o.add(db, dtp);
        s[2 * BW] = o.sub(sb, st);
        s[4 * BW] = o.sub(db, dtp);
        const double u5 = m1[1];
        s[7 * BW] = fma(K(MFOUR), u5, o.add(sb, st));
        s[10 * BW] = o.sub(u5, m1[0]);
        s[11 * BW] = o.sub(m1[2], u5);
        s[12 * BW] = o.sub(u5, m0[1]);
        s[13 * BW] = o.sub(m2[1], u5);
        const double v4 = m1[WC], v6 = m1[WC + 2];
        s[1 * BW] = o.add(v4, v6);
        s[8 * BW] = o.sub(v6, v4);
        s[5 * BW] = o.sub(m2[WC + 1], m0[WC + 1]);
        const double z2 = m0[2 * WC + 1], z8 = m2[2 * WC + 1];
        s[3 * BW] = o.add(z2, z8);
        s[9 * BW] = o.sub(z8, z2);
        s[6 * BW] = o.sub(m1[2 * WC + 2], m1[2 * WC]);
      }
      // into the frame, in place: (rho, m_x, m_y, E) -> (W1, q_x, q_y, X/2)
      double dW[4];
      const double bx = o.mul(b1h, vx), by = o.mul(b1h, vy), bq = o.mul(b1h, q2h);
      const double m2 = K(MTWO);
#pragma unroll
      for (int n = 0; n < 14; ++n) {
        const double r = w1p[n * BW];
        const double qx = fma(-vx, r, cf[(14 + n) * BW]), qy = fma(-vy, r, cf[(28 + n) * BW]);
        const double xh = fma(-bq, r, fma(-by, qy, fma(-bx, qx, o.mul(b1h, cf[n * BW]))));
        const double w1 = fma(m2, xh, r);
        if (n >= 10) {
          dX[n - 10] = xh;
          dqx[n - 10] = qx;
          dqy[n - 10] = qy;
          dW[n - 10] = w1;
        } else {
          cf[n * BW] = xh;
          cf[(14 + n) * BW] = qx;
          cf[(28 + n) * BW] = qy;
          w1p[n * BW] = w1;
        }
      }
      // the Appendix coefficients (scaled) of one variable from its combinations
      auto coefficients = [&](const double* s, const double (&e)[4], double (&C)[15]) {
        {
          const double X1 = s[0 * BW], Va = s[1 * BW], ex = -o.add(e[0], e[1]);
          const double X2 = s[2 * BW], Wa = s[3 * BW], ey = -o.add(e[2], e[3]);
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
          const double X3 = s[4 * BW], v82 = s[5 * BW], w64 = s[6 * BW];
          C[4] = fma(K(A4X), X3, o.mul(K(A4V), o.add(v82, w64)));
          const double x = o.mul(K(A11X), X3), kv = K(A11V);
          C[11] = fma(kv, v82, x);
          C[13] = fma(kv, w64, x);
        }
        {
          const double r = s[7 * BW], Vd = s[8 * BW], Wd = s[9 * BW];
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
      };
      // X/2, q_x, q_y: their coefficients replace their combinations
#pragma unroll 1
      for (int v = 0; v < 3; ++v) {
        double* s = cf + 14 * v * BW;
        double C[15], e[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) e[n] = v == 0 ? dX[n] : (v == 1 ? dqx[n] : dqy[n]);
        coefficients(s, e, C);
#pragma unroll
        for (int n = 0; n < 14; ++n) s[n * BW] = C[n + 1];
      }
      // the entropy field: reconstructed here for both passes
      {
        double C[15];
        coefficients(w1p, dW, C);
        Factors F;
        const double mean = o.sub(w0[0 * WC + t + 1], X5);
        fast &= factors<false>(o, beta0(o, C), dW, mean, P, F);
#pragma unroll
        for (int n = 1; n < 15; ++n) C[n] = o.mul(C[n], F.a0);
        C[1] = fma(F.r, dW[1], fma(F.l, dW[0], C[1]));
        C[2] = fma(F.t, dW[3], fma(F.b, dW[2], C[2]));
        C[0] = constant_term(o, C, mean);
        double lo[3], hi[3];
        edges<1>(o, C, lo, hi);
#pragma unroll
        for (int g = 0; g < 3; ++g) {
          w1p[(6 + g) * BW] = lo[g];
          w1p[(9 + g) * BW] = hi[g];
        }
        if (xrow) {
          edges<0>(o, C, lo, hi);
#pragma unroll
          for (int g = 0; g < 3; ++g) {
            w1p[g * BW] = lo[g];
            w1p[(3 + g) * BW] = hi[g];
          }
          double in[9];
          interior(o, C, in);
#pragma unroll
          for (int g = 0; g < 9; ++g) w1p[(12 + g) * BW] = in[g];
          w1p[21 * BW] = vhat<0>(o, C);
          w1p[22 * BW] = vhat<1>(o, C);
        }
      }
    }

    double rx[NC][3];                // x-face and volume part of the RHS of (i, j)
    double vh[NC], wh[NC];
#pragma unroll
    for (int a = 0; a < NC; ++a) rx[a][0] = rx[a][1] = rx[a][2] = vh[a] = wh[a] = 0.0;
    double gb[3][NC];                // g - a2 u of the bottom traces
    double gt[3][NC];                // g + a2 u of the top traces

    // two passes: x (edge points of the x faces, the volume sum of f, v-hat), then y
#pragma unroll
    for (int dir = 0; dir < 2; ++dir) {
      if (dir == 0 && !xrow) continue;
      double glo[3][NC], ghi[3][NC];  // flux -+ a u of the low and high traces, 2 LF halves
      double vol[NC], mod[NC];
      if (need) {
        const double un = dir == 0 ? vx : vy, ut = dir == 0 ? vy : vx;
        const double* cX = cf;
        const double* cN = cf + (dir == 0 ? 14 : 28) * BW;   // normal momentum
        const double* cT = cf + (dir == 0 ? 28 : 14) * BW;   // tangential momentum
        const double(&eN)[4] = dir == 0 ? dqx : dqy;
        const double(&eT)[4] = dir == 0 ? dqy : dqx;
        double PX[15], PQ[15], PT[15];
        // the acoustic fields X/2 -+ q_n/(2c), then X = W0 + W3 and q_n = c (W3 - W0)
        {
          Factors F0, F3;
          const double w5 = o.mul(K(HALF), X5);
          double s0x, s0y, s3x, s3y;
          {
            double C[15], e[4];
#pragma unroll
            for (int n = 1; n < 15; ++n) C[n] = fma(-hic, cN[(n - 1) * BW], cX[(n - 1) * BW]);
#pragma unroll
            for (int n = 0; n < 4; ++n) e[n] = fma(-hic, eN[n], dX[n]);
            fast &= factors<false>(o, beta0(o, C), e, w5, P, F0);
            s0x = fma(F0.r, e[1], o.mul(F0.l, e[0]));
            s0y = fma(F0.t, e[3], o.mul(F0.b, e[2]));
          }
          {
            double C[15], e[4];
#pragma unroll
            for (int n = 1; n < 15; ++n) C[n] = fma(hic, cN[(n - 1) * BW], cX[(n - 1) * BW]);
#pragma unroll
            for (int n = 0; n < 4; ++n) e[n] = fma(hic, eN[n], dX[n]);
            fast &= factors<false>(o, beta0(o, C), e, w5, P, F3);
            s3x = fma(F3.r, e[1], o.mul(F3.l, e[0]));
            s3y = fma(F3.t, e[3], o.mul(F3.b, e[2]));
          }
          const double ap = o.add(F0.a0, F3.a0), am = o.sub(F3.a0, F0.a0);
          const double xq = o.mul(hic, am), qx = o.mul(c, am), qq = o.mul(K(HALF), ap);
#pragma unroll
          for (int n = 1; n < 15; ++n) {
            const double x = cX[(n - 1) * BW], q = cN[(n - 1) * BW];
            PX[n] = fma(xq, q, o.mul(ap, x));
            PQ[n] = fma(qq, q, o.mul(qx, x));
          }
          PX[1] = o.add(PX[1], o.add(s0x, s3x));
          PX[2] = o.add(PX[2], o.add(s0y, s3y));
          PQ[1] = fma(c, o.sub(s3x, s0x), PQ[1]);
          PQ[2] = fma(c, o.sub(s3y, s0y), PQ[2]);
          PX[0] = constant_term(o, PX, X5);
          PQ[0] = constant_term(o, PQ, o.nz);
        }
        // the shear field: the tangential momentum in the cell's frame
        {
#pragma unroll
          for (int n = 1; n < 15; ++n) PT[n] = cT[(n - 1) * BW];
          Factors F;
          fast &= factors<true>(o, beta0(o, PT), eT, 0.0, P, F);
#pragma unroll
          for (int n = 1; n < 15; ++n) PT[n] = o.mul(PT[n], F.a0);
          PT[1] = fma(F.r, eT[1], fma(F.l, eT[0], PT[1]));
          PT[2] = fma(F.t, eT[3], fma(F.b, eT[2], PT[2]));
          PT[0] = constant_term(o, PT, o.nz);
        }
        // conserved components of the frame variables (rho, q_n, q_t, X)
        auto conserved = [&](double r, double q, double s, double x, double& mn, double& mt,
                             double& E) {
          mn = fma(un, r, q);
          mt = fma(ut, r, s);
          E = fma(q2h, r, fma(ut, s, fma(un, q, o.mul(h, x))));
        };
        // traces and their fluxes
        {
          double X[2][3], Q[2][3], T[2][3];
          if (dir == 0) {
            edges<0>(o, PX, X[0], X[1]);
            edges<0>(o, PQ, Q[0], Q[1]);
            edges<0>(o, PT, T[0], T[1]);
          } else {
            edges<1>(o, PX, X[0], X[1]);
            edges<1>(o, PQ, Q[0], Q[1]);
            edges<1>(o, PT, T[0], T[1]);
          }
          const double a = dir == 0 ? a1 : a2, gm1 = K(GM1), hg = K(HGM1);
#pragma unroll
          for (int side = 0; side < 2; ++side)
#pragma unroll
            for (int g = 0; g < 3; ++g) {
              const double r = o.add(w1p[(6 * dir + 3 * side + g) * BW], X[side][g]);
              double mn, mt, E;
              conserved(r, Q[side][g], T[side][g], X[side][g], mn, mt, E);
              const double ir = rcp_any(o, r);
              const double vn = o.mul(mn, ir);
              const double kin = o.mul(fma(mn, mn, o.mul(mt, mt)), ir);
              const double p = fma(hg, kin, o.mul(gm1, E));
              const double fn = fma(mn, vn, p), ft = o.mul(mt, vn), fE = o.mul(o.add(E, p), vn);
              double(&f)[NC] = side == 0 ? glo[g] : ghi[g];
              const double as = side == 0 ? -a : a;
              f[0] = fma(as, r, mn);
              f[dir == 0 ? 1 : 2] = fma(as, mn, fn);
              f[dir == 0 ? 2 : 1] = fma(as, mt, ft);
              f[3] = fma(as, E, fE);
            }
        }
        // volume sum and first-moment modification
        if (xrow) {
          double X[9], Q[9], T[9];
          interior(o, PX, X);
          interior(o, PQ, Q);
          interior(o, PT, T);
          double Z = o.nz, A = o.nz, B = o.nz, G1 = o.nz, G2 = o.nz;
          const double wc = K(WC), we = K(WE), wm_ = K(WM);
#pragma unroll
          for (int g = 0; g < 9; ++g) {
            const double r = o.add(w1p[(12 + g) * BW], X[g]);
            const double ir = rcp_any(o, r);
            const double wir = o.mul(g == 4 ? wm_ : ((g & 1) ? we : wc), ir);
            const double qa = o.mul(Q[g], wir);
            const double z = fma(Q[g], Q[g], o.mul(T[g], T[g]));
            Z = fma(wir, z, Z);
            A = fma(Q[g], qa, A);
            B = fma(T[g], qa, B);
            G1 = fma(X[g], qa, G1);
            G2 = fma(o.mul(qa, ir), z, G2);
          }
          const double hg = K(HGM1);
          const double pm = fma(hg, Z, p5);
          const double mn = w0[(dir == 0 ? 3 : 6) * WC + t + 1];
          const double mt = w0[(dir == 0 ? 6 : 3) * WC + t + 1];
          const double E = w0[9 * WC + t + 1];
          vol[0] = mn;
          vol[dir == 0 ? 1 : 2] = fma(mn, un, o.add(A, pm));
          vol[dir == 0 ? 2 : 1] = fma(mt, un, B);
          vol[3] = fma(un, o.add(E, pm),
                       fma(ut, B, fma(un, A, fma(o.add(h, c2), G1, o.mul(hg, G2)))));
          const double Xv = dir == 0 ? vhat<0>(o, PX) : vhat<1>(o, PX);
          const double Qv = dir == 0 ? vhat<0>(o, PQ) : vhat<1>(o, PQ);
          const double Tv = dir == 0 ? vhat<0>(o, PT) : vhat<1>(o, PT);
          mod[0] = o.add(w1p[(21 + dir) * BW], Xv);
          conserved(mod[0], Qv, Tv, Xv, mod[dir == 0 ? 1 : 2], mod[dir == 0 ? 2 : 1], mod[3]);
        }
      }
      if (dir == 0) {
        // x faces: twice the LF flux of a face is (f + a u) of the left cell's trace plus
        // (f - a u) of the right cell's; each face formed once, by the thread left of it
        if (need) {
#pragma unroll
          for (int g = 0; g < 3; ++g)
#pragma unroll
            for (int a = 0; a < NC; ++a) xch[(a * 3 + g) * BW + t] = glo[g][a];
        }
        __syncthreads();
        if (need && t <= wout && i < nx) {
          const double k0 = K(FX0), k1 = K(FX1), k2 = K(FX2);
#pragma unroll
          for (int a = 0; a < NC; ++a) {
            double* x = xch + a * 3 * BW + t + 1;
            const double F0 = o.add(ghi[0][a], x[0]), F1 = o.add(ghi[1][a], x[BW]),
                         F2 = o.add(ghi[2][a], x[2 * BW]);
            x[0] = fma(k1, F1, o.mul(k0, o.add(F0, F2)));  // the slots' only reader
            x[BW] = o.mul(k2, o.sub(F2, F0));
          }
        }
        __syncthreads();
        if (outc) {
          const double idx = K(IDX), half = K(HALF);
#pragma unroll
          for (int a = 0; a < NC; ++a) {
            const double* x = xch + a * 3 * BW + t;
            const double Lw = x[0], Rw = x[1];
            rx[a][0] = o.sub(Lw, Rw);
            rx[a][1] = fma(vol[a], idx, -o.mul(half, o.add(Lw, Rw)));
            rx[a][2] = o.sub(x[BW], x[BW + 1]);
          }
        }
        if (need) {
#pragma unroll
          for (int a = 0; a < NC; ++a) vh[a] = mod[a];
        }
      } else if (need) {
#pragma unroll
        for (int g = 0; g < 3; ++g)
#pragma unroll
          for (int a = 0; a < NC; ++a) {
            gb[g][a] = glo[g][a];
            gt[g][a] = ghi[g][a];
          }
        if (xrow) {
          const double idy = K(IDY);
#pragma unroll
          for (int a = 0; a < NC; ++a) {
            wh[a] = mod[a];
            rx[a][2] = fma(vol[a], idy, rx[a][2]);
          }
        }
      }
    }

    // y face j-1/2 between (i, j-1) (its top traces' part carried) and (i, j): Eq. 2.16
    if (need && j > j0 - 1) {
      const double k0 = K(FY0), k1 = K(FY1), k2 = K(FY2), half = K(HALF);
#pragma unroll
      for (int a = 0; a < NC; ++a) {
        const double G0 = o.add(car[(a * 3 + 0) * BW], gb[0][a]),
                     G1 = o.add(car[(a * 3 + 1) * BW], gb[1][a]),
                     G2 = o.add(car[(a * 3 + 2) * BW], gb[2][a]);
        const double sw = fma(k1, G1, o.mul(k0, o.add(G0, G2)));
        const double sm = o.mul(k2, o.sub(G2, G0));
        pend[a][0] = o.sub(pend[a][0], sw);
        pend[a][1] = o.sub(pend[a][1], sm);
        pend[a][2] = fma(-half, sw, pend[a][2]);
        rx[a][0] = o.add(rx[a][0], sw);
        rx[a][1] = o.add(rx[a][1], sm);
        rx[a][2] = fma(-half, sw, rx[a][2]);
      }
      // stage update of (i, j-1): Eq. 2.13
      if (outc && j - 1 >= j0) {
        const size_t q = (size_t)(j - 1) * nx + i;
        double ua[NC];
        bool bad = false;
#pragma unroll
        for (int a = 0; a < NC; ++a) {
          const double own[3] = {wm[(a * 3) * WC + t + 1], pvh[a], pwh[a]};
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            const size_t qa = (size_t)(a * 3 + m) * plane + q;
            double base;
            if (S.k == 1) {
              base = own[m];
              if (m > 0) S.Vh[(size_t)(a * 2 + m - 1) * plane + q] = own[m];
            } else {
              base = (m == 0) ? S.Un[qa] : S.Vh[(size_t)(a * 2 + m - 1) * plane + q];
            }
            const double adv = fma(dt, pend[a][m], own[m]);
            double out;
            if (S.k == 1) out = adv;
            else if (S.k == 2) out = fma(K(THREEQ), base, o.mul(K(QUARTER), adv));
            else out = fma(K(THIRD), base, o.mul(K(TWOTHIRD), adv));
            S.Uout[qa] = out;
            bad |= !finite_bits(out);
            if (m == 0) ua[a] = out;
          }
        }
        double s0, s1;
        bad |= !euler_speeds<2>(P, ua, s0, s1);
        if (!bad) {
          wmax0 = fmax(wmax0, s0);
          wmax1 = fmax(wmax1, s1);
        } else {
          atomicOr(S.status, kStatusNonphysical);
        }
      }
    }
    // carry row j to the next iteration
    if (need) {
#pragma unroll
      for (int g = 0; g < 3; ++g)
#pragma unroll
        for (int a = 0; a < NC; ++a) car[(a * 3 + g) * BW] = gt[g][a];
#pragma unroll
      for (int a = 0; a < NC; ++a) {
        pend[a][0] = rx[a][0];
        pend[a][1] = rx[a][1];
        pend[a][2] = rx[a][2];
        pvh[a] = vh[a];
        pwh[a] = wh[a];
      }
    }
    __syncthreads();                       // every read of row j-1 is done
    if (j + 2 <= j1 + 1) load_row(j + 2);  // into the slot of row j-1
    __syncthreads();
  }

  // block maxima of the output wave speeds -> one atomic per block and direction
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    wmax0 = fmax(wmax0, __shfl_xor_sync(0xffffffffu, wmax0, o));
    wmax1 = fmax(wmax1, __shfl_xor_sync(0xffffffffu, wmax1, o));
  }
  if ((t & 31) == 0) {
    red[0][t >> 5] = wmax0;
    red[1][t >> 5] = wmax1;
  }
  const int any_direct = __syncthreads_or(fast ? 0 : 1);
  if (t == 0) {
    // informational status bit: some cell of the block needed the direct-formula weights
    if (any_direct) atomicOr(S.status, kStatusDirectWeights);
    double m0 = red[0][0], m1 = red[1][0];
#pragma unroll
    for (int w = 1; w < BW / 32; ++w) {
      m0 = fmax(m0, red[0][w]);
      m1 = fmax(m1, red[1][w]);
    }
    atomic_max_nonneg(&S.alpha_out[0], m0);
    atomic_max_nonneg(&S.alpha_out[1], m1);
  }
  __syncthreads();  // the block may start another item in the same shared memory
}

#undef K

}  // namespace hw
