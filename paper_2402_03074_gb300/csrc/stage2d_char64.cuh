// stage2d_char64.cuh -- the reconstruction of one cell of the 2D Euler equations with the local
// characteristic decomposition in FP64 (Sec. 2.2, Remark 2.2), for the tiles of
// stage2d_tile64.cuh: traces, volume sums and first-moment modifications of both passes.
//
// On top of recon64.cuh, the cell's own Galilean frame.  With q = m - u rho and E' = E - u.q -
// u^2 rho / 2 (u the velocity of the cell's average), the characteristic variables are
// X/2 -+ q_n/(2c), W1 = rho - X and q_t, X = (gamma-1)/c^2 E'.
//  * The frame is linear in the state, so it is applied to the 14 stencil combinations the
//    Appendix coefficients are formed from, once for both passes; and W1 (the entropy field) is
//    the same field in both passes, so it is reconstructed once per cell: seven fields instead
//    of eight.
//  * The volume integrals of f and g are taken in the frame: the Gauss rule integrates the linear
//    parts exactly (the polynomial's average is the cell average), so only the sums of
//    q_n^2/rho, q_n q_t/rho, ... over the nine points are left, and the frame is undone once
//    per cell instead of per point.
// Against the field-by-field evaluation in the conserved variables (eight fields, points
// unprojected one by one; the same bands and blocks), 2048^2, 96-thread blocks: 29.0 -> 21.2 ms
// per stage; 18.8 ms on the three-register FMAs of f64_ops.cuh.
#pragma once
#include "recon64.cuh"

namespace hw {

// T: threads of the block (the stride of a thread's column in shared memory); WC: columns of the
// row window.
template <int T, int WC>
struct Char64Cell {
  static constexpr int NC = 4;
  static constexpr int kCols = 65;  // the coefficients of X/2, q_x, q_y; 21 values and both
                                    // modifications of W1
  const KProblem& P;
  const Ops& o;
  const double *wm, *w0, *wp;  // window rows below, at, above the cell, at the column left of it
  double* cf;                  // this thread's column: X/2 (0-13), q_x, q_y
  double* w1p;                 // W1 on the x edges, the y edges, inside; its modifications
  double vx, vy, q2h, p5, c2, c, h, hic, X5;  // the cell's frame
  double dX[4], dqx[4], dqy[4];  // X/2, q_x, q_y of u5 - u4, u6 - u5, u5 - u2, u8 - u5

  __device__ __forceinline__ Char64Cell(const KProblem& P_, const Ops& o_, const double* wm_,
                                        const double* w0_, const double* wp_, double* col)
      : P(P_), o(o_), wm(wm_), w0(w0_), wp(wp_), cf(col), w1p(col + 42 * T) {}

  // What both passes share; xrow: the cell is in an output row (not in a ring row, of which only
  // the y traces are used).  Returns false where the direct-formula weights were needed.
  __device__ __forceinline__ bool begin(bool xrow) {
    using namespace c64;
    bool fast = true;
    double b1h;
    {
      const double U0 = w0[0 * WC + 1], U1 = w0[3 * WC + 1], U2 = w0[6 * WC + 1],
                   U3 = w0[9 * WC + 1];
      const double ir = rcp_any(U0);
      vx = o.mul(U1, ir);
      vy = o.mul(U2, ir);
      q2h = o.mul(K(HALF), fma(vx, vx, o.mul(vy, vy)));
      p5 = o.mul(K(GM1), fma(-U0, q2h, U3));
      c2 = o.mul(o.mul(K(GAM), p5), ir);
      const double rc = rsqrt_any(o, c2, K(HALF), K(RS2));
      c = o.mul(c2, rc);
      h = fma(o.add(U3, p5), ir, -q2h);
      hic = o.mul(K(HALF), rc);
      const double rc2 = o.mul(rc, rc);
      b1h = -o.mul(K(HGM1), rc2);
      X5 = o.mul(p5, rc2);
    }
    // the stencil combinations of the conserved components
#pragma unroll
    for (int a = 0; a < NC; ++a) {
      double* s = a == 0 ? w1p : cf + (a == 3 ? 0 : 14 * a) * T;
      combinations<WC>(o, wm + 3 * a * WC, w0 + 3 * a * WC, wp + 3 * a * WC,
                       [s](int n, double v) { s[n * T] = v; });
    }
    // into the frame, in place: (rho, m_x, m_y, E) -> (W1, q_x, q_y, X/2)
    double dW[4];
    const double bx = o.mul(b1h, vx), by = o.mul(b1h, vy), bq = o.mul(b1h, q2h);
    const double m2 = K(MTWO);
#pragma unroll
    for (int n = 0; n < 14; ++n) {
      const double r = w1p[n * T];
      const double qx = fma(-vx, r, cf[(14 + n) * T]), qy = fma(-vy, r, cf[(28 + n) * T]);
      const double xh = fma(-bq, r, fma(-by, qy, fma(-bx, qx, o.mul(b1h, cf[n * T]))));
      const double w1 = fma(m2, xh, r);
      if (n >= 10) {
        dX[n - 10] = xh;
        dqx[n - 10] = qx;
        dqy[n - 10] = qy;
        dW[n - 10] = w1;
      } else {
        cf[n * T] = xh;
        cf[(14 + n) * T] = qx;
        cf[(28 + n) * T] = qy;
        w1p[n * T] = w1;
      }
    }
    // X/2, q_x, q_y: their coefficients replace their combinations
#pragma unroll 1
    for (int v = 0; v < 3; ++v) {
      double* s = cf + 14 * v * T;
      double C[15], e[4];
#pragma unroll
      for (int n = 0; n < 4; ++n) e[n] = v == 0 ? dX[n] : (v == 1 ? dqx[n] : dqy[n]);
      coefficients(o, [s](int n) { return s[n * T]; }, e, C);
#pragma unroll
      for (int n = 0; n < 14; ++n) s[n * T] = C[n + 1];
    }
    // the entropy field: reconstructed here for both passes
    {
      double C[15];
      coefficients(o, [this](int n) { return w1p[n * T]; }, dW, C);
      Factors F;
      const double mean = o.sub(w0[0 * WC + 1], X5);
      fast &= factors(o, beta0(o, C), dW, average_sum<false>(o, dW, mean), P, F);
#pragma unroll
      for (int n = 1; n < 15; ++n) C[n] = o.mul(C[n], F.a0);
      C[1] = fma(F.r, dW[1], fma(F.l, dW[0], C[1]));
      C[2] = fma(F.t, dW[3], fma(F.b, dW[2], C[2]));
      C[0] = constant_term(o, C, mean);
      double lo[3], hi[3];
      edges<1>(o, C, lo, hi);
#pragma unroll
      for (int g = 0; g < 3; ++g) {
        w1p[(6 + g) * T] = lo[g];
        w1p[(9 + g) * T] = hi[g];
      }
      if (xrow) {
        edges<0>(o, C, lo, hi);
#pragma unroll
        for (int g = 0; g < 3; ++g) {
          w1p[g * T] = lo[g];
          w1p[(3 + g) * T] = hi[g];
        }
        double in[9];
        interior(o, C, in);
#pragma unroll
        for (int g = 0; g < 9; ++g) w1p[(12 + g) * T] = in[g];
        w1p[21 * T] = vhat<0>(o, C);
        w1p[22 * T] = vhat<1>(o, C);
      }
    }
    return fast;
  }

  // The pass of direction DIR: flux - a u on the low edge and flux + a u on the high edge at the
  // three Gauss points, and in output rows the volume sum and the first-moment modification.
  template <int DIR>
  __device__ __forceinline__ bool pass(bool xrow, double a, double (&lo)[3][NC],
                                       double (&hi)[3][NC], double (&vol)[NC], double (&mod)[NC]) {
    using namespace c64;
    bool fast = true;
    const double un = DIR == 0 ? vx : vy, ut = DIR == 0 ? vy : vx;
    const double* cX = cf;
    const double* cN = cf + (DIR == 0 ? 14 : 28) * T;   // normal momentum
    const double* cT = cf + (DIR == 0 ? 28 : 14) * T;   // tangential momentum
    const double(&eN)[4] = DIR == 0 ? dqx : dqy;
    const double(&eT)[4] = DIR == 0 ? dqy : dqx;
    double PX[15], PQ[15], PT[15];
    // the acoustic fields X/2 -+ q_n/(2c), then X = W0 + W3 and q_n = c (W3 - W0)
    {
      Factors F0, F3;
      const double w5 = o.mul(K(HALF), X5);
      double s0x, s0y, s3x, s3y;
      {
        double C[15], e[4];
#pragma unroll
        for (int n = 1; n < 15; ++n) C[n] = fma(-hic, cN[(n - 1) * T], cX[(n - 1) * T]);
#pragma unroll
        for (int n = 0; n < 4; ++n) e[n] = fma(-hic, eN[n], dX[n]);
        fast &= factors(o, beta0(o, C), e, average_sum<false>(o, e, w5), P, F0);
        s0x = fma(F0.r, e[1], o.mul(F0.l, e[0]));
        s0y = fma(F0.t, e[3], o.mul(F0.b, e[2]));
      }
      {
        double C[15], e[4];
#pragma unroll
        for (int n = 1; n < 15; ++n) C[n] = fma(hic, cN[(n - 1) * T], cX[(n - 1) * T]);
#pragma unroll
        for (int n = 0; n < 4; ++n) e[n] = fma(hic, eN[n], dX[n]);
        fast &= factors(o, beta0(o, C), e, average_sum<false>(o, e, w5), P, F3);
        s3x = fma(F3.r, e[1], o.mul(F3.l, e[0]));
        s3y = fma(F3.t, e[3], o.mul(F3.b, e[2]));
      }
      const double ap = o.add(F0.a0, F3.a0), am = o.sub(F3.a0, F0.a0);
      const double xq = o.mul(hic, am), qx = o.mul(c, am), qq = o.mul(K(HALF), ap);
#pragma unroll
      for (int n = 1; n < 15; ++n) {
        const double x = cX[(n - 1) * T], q = cN[(n - 1) * T];
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
      for (int n = 1; n < 15; ++n) PT[n] = cT[(n - 1) * T];
      Factors F;
      fast &= factors(o, beta0(o, PT), eT, average_sum<true>(o, eT, 0.0), P, F);
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
      double X[2][3], Q[2][3], Y[2][3];
      edges<DIR>(o, PX, X[0], X[1]);
      edges<DIR>(o, PQ, Q[0], Q[1]);
      edges<DIR>(o, PT, Y[0], Y[1]);
      const double gm1 = K(GM1), hg = K(HGM1);
#pragma unroll
      for (int side = 0; side < 2; ++side)
#pragma unroll
        for (int g = 0; g < 3; ++g) {
          const double r = o.add(w1p[(6 * DIR + 3 * side + g) * T], X[side][g]);
          double mn, mt, E;
          conserved(r, Q[side][g], Y[side][g], X[side][g], mn, mt, E);
          const double ir = rcp_any(r);
          const double vn = o.mul(mn, ir);
          const double kin = o.mul(fma(mn, mn, o.mul(mt, mt)), ir);
          const double p = fma(hg, kin, o.mul(gm1, E));
          const double fn = fma(mn, vn, p), ft = o.mul(mt, vn), fE = o.mul(o.add(E, p), vn);
          double(&f)[NC] = side == 0 ? lo[g] : hi[g];
          const double as = side == 0 ? -a : a;
          f[0] = fma(as, r, mn);
          f[DIR == 0 ? 1 : 2] = fma(as, mn, fn);
          f[DIR == 0 ? 2 : 1] = fma(as, mt, ft);
          f[3] = fma(as, E, fE);
        }
    }
    // volume sum and first-moment modification
    if (xrow) {
      double X[9], Q[9], Y[9];
      interior(o, PX, X);
      interior(o, PQ, Q);
      interior(o, PT, Y);
      double Z = o.nz, A = o.nz, B = o.nz, G1 = o.nz, G2 = o.nz;
      const double wc = K(WC), we = K(WE), wm_ = K(WM);
#pragma unroll
      for (int g = 0; g < 9; ++g) {
        const double r = o.add(w1p[(12 + g) * T], X[g]);
        const double ir = rcp_any(r);
        const double wir = o.mul(g == 4 ? wm_ : ((g & 1) ? we : wc), ir);
        const double qa = o.mul(Q[g], wir);
        const double z = fma(Q[g], Q[g], o.mul(Y[g], Y[g]));
        Z = fma(wir, z, Z);
        A = fma(Q[g], qa, A);
        B = fma(Y[g], qa, B);
        G1 = fma(X[g], qa, G1);
        G2 = fma(o.mul(qa, ir), z, G2);
      }
      const double hg = K(HGM1);
      const double pm = fma(hg, Z, p5);
      const double mn = w0[(DIR == 0 ? 3 : 6) * WC + 1];
      const double mt = w0[(DIR == 0 ? 6 : 3) * WC + 1];
      const double E = w0[9 * WC + 1];
      vol[0] = mn;
      vol[DIR == 0 ? 1 : 2] = fma(mn, un, o.add(A, pm));
      vol[DIR == 0 ? 2 : 1] = fma(mt, un, B);
      vol[3] = fma(un, o.add(E, pm),
                   fma(ut, B, fma(un, A, fma(o.add(h, c2), G1, o.mul(hg, G2)))));
      const double Xv = vhat<DIR>(o, PX);
      const double Qv = vhat<DIR>(o, PQ);
      const double Tv = vhat<DIR>(o, PT);
      mod[0] = o.add(w1p[(21 + DIR) * T], Xv);
      conserved(mod[0], Qv, Tv, Xv, mod[DIR == 0 ? 1 : 2], mod[DIR == 0 ? 2 : 1], mod[3]);
    }
    return fast;
  }
};
}  // namespace hw
