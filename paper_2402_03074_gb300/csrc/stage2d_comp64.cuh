// stage2d_comp64.cuh -- the reconstruction of one cell in FP64, component by component (scalar
// laws, and Euler without the characteristic decomposition), for the tiles of
// stage2d_tile64.cuh.  One reconstruction of a component serves both passes, so every point is
// evaluated once; the volume sums of f and g are taken together over the same nine points (one
// reciprocal of rho each), and the parts the Gauss rule integrates exactly (the mass fluxes, the
// kinetic part of the mean pressure's linear terms, all of advection) come from the averages.
#pragma once
#include "recon64.cuh"

namespace hw {

template <int EQ, int T, int WC>
struct Comp64Cell {
  static constexpr int NC = EQ == EQ_EULER ? 4 : 1;
  static constexpr int kCols = 15 * NC;  // the combined polynomial of every component
  const KProblem& P;
  const Ops& o;
  const double *wm, *w0, *wp;  // window rows below, at, above the cell, at the column left of it
  double* col;
  double vg[NC];  // the volume sum of g, formed with that of f

  __device__ __forceinline__ Comp64Cell(const KProblem& P_, const Ops& o_, const double* wm_,
                                        const double* w0_, const double* wp_, double* col_)
      : P(P_), o(o_), wm(wm_), w0(w0_), wp(wp_), col(col_) {}

  __device__ __forceinline__ void polynomial(int a, double (&C)[15]) const {
#pragma unroll
    for (int n = 0; n < 15; ++n) C[n] = col[(15 * a + n) * T];
  }

  __device__ __forceinline__ bool begin(bool) {
    using namespace c64;
    bool fast = true;
#pragma unroll 1
    for (int a = 0; a < NC; ++a) {
      double s[14], C[15];
      combinations<WC>(o, wm + 3 * a * WC, w0 + 3 * a * WC, wp + 3 * a * WC,
                       [&s](int n, double v) { s[n] = v; });
      const double e[4] = {s[10], s[11], s[12], s[13]};
      coefficients(o, [&s](int n) { return s[n]; }, e, C);
      const double mean = w0[3 * a * WC + 1];
      Factors F;
      fast &= factors(o, beta0(o, C), e, average_sum<false>(o, e, mean), P, F);
#pragma unroll
      for (int n = 1; n < 15; ++n) C[n] = o.mul(C[n], F.a0);
      C[1] = fma(F.r, e[1], fma(F.l, e[0], C[1]));
      C[2] = fma(F.t, e[3], fma(F.b, e[2], C[2]));
      C[0] = constant_term(o, C, mean);
#pragma unroll
      for (int n = 0; n < 15; ++n) col[(15 * a + n) * T] = C[n];
    }
    return fast;
  }

  // flux of direction DIR at the state u
  template <int DIR>
  __device__ __forceinline__ void flux(const double (&u)[NC], double (&f)[NC]) const {
    using namespace c64;
    if constexpr (EQ == EQ_ADV) {
      f[0] = o.mul(DIR == 0 ? K(AX) : K(AY), u[0]);
    } else if constexpr (EQ == EQ_BURG) {
      f[0] = o.mul(o.mul(K(HALF), u[0]), u[0]);
    } else {
      constexpr int n = 1 + DIR, t = 2 - DIR;
      const double ir = rcp_any(u[0]);
      const double vn = o.mul(u[n], ir);
      const double kin = o.mul(fma(u[n], u[n], o.mul(u[t], u[t])), ir);
      const double p = fma(K(HGM1), kin, o.mul(K(GM1), u[3]));
      f[0] = u[n];
      f[n] = fma(u[n], vn, p);
      f[t] = o.mul(u[t], vn);
      f[3] = o.mul(o.add(u[3], p), vn);
    }
  }

  // The pass of direction DIR: flux - a u on the low edge and flux + a u on the high edge at the
  // three Gauss points, and in output rows the volume sum and the first-moment modification.
  template <int DIR>
  __device__ __forceinline__ bool pass(bool xrow, double a, double (&lo)[3][NC],
                                       double (&hi)[3][NC], double (&vol)[NC], double (&mod)[NC]) {
    using namespace c64;
    {
      double tr[2][3][NC];
#pragma unroll
      for (int b = 0; b < NC; ++b) {
        double C[15], l[3], h[3];
        polynomial(b, C);
        edges<DIR>(o, C, l, h);
        if (xrow) mod[b] = vhat<DIR>(o, C);
#pragma unroll
        for (int g = 0; g < 3; ++g) {
          tr[0][g][b] = l[g];
          tr[1][g][b] = h[g];
        }
      }
#pragma unroll
      for (int side = 0; side < 2; ++side)
#pragma unroll
        for (int g = 0; g < 3; ++g) {
          double f[NC];
          flux<DIR>(tr[side][g], f);
#pragma unroll
          for (int b = 0; b < NC; ++b)
            (side == 0 ? lo : hi)[g][b] = fma(side == 0 ? -a : a, tr[side][g][b], f[b]);
        }
    }
    if (!xrow) return true;
    if constexpr (DIR == 1) {
#pragma unroll
      for (int b = 0; b < NC; ++b) vol[b] = vg[b];
    } else if constexpr (EQ == EQ_ADV) {
      const double u = w0[1];
      vol[0] = o.mul(K(AX), u);
      vg[0] = o.mul(K(AY), u);
    } else if constexpr (EQ == EQ_BURG) {
      double C[15], u[9];
      polynomial(0, C);
      interior(o, C, u);
      const double sc = fma(u[8], u[8], fma(u[6], u[6], fma(u[2], u[2], o.mul(u[0], u[0]))));
      const double se = fma(u[7], u[7], fma(u[5], u[5], fma(u[3], u[3], o.mul(u[1], u[1]))));
      const double s = fma(K(WC), sc, fma(K(WE), se, o.mul(o.mul(K(WM), u[4]), u[4])));
      vol[0] = vg[0] = o.mul(K(HALF), s);
    } else {
      double u[4][9];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        double C[15];
        polynomial(b, C);
        interior(o, C, u[b]);
      }
      // means of m_x^2/rho, m_x m_y/rho, m_y^2/rho, (E + p) m_x/rho, (E + p) m_y/rho
      double xx = o.nz, xy = o.nz, yy = o.nz, hx = o.nz, hy = o.nz;
      const double wc = K(WC), we = K(WE), wm_ = K(WM), gm1 = K(GM1), hg = K(HGM1);
#pragma unroll
      for (int g = 0; g < 9; ++g) {
        const double ir = rcp_any(u[0][g]);
        const double wir = o.mul(g == 4 ? wm_ : ((g & 1) ? we : wc), ir);
        const double wx = o.mul(u[1][g], wir), wy = o.mul(u[2][g], wir);
        const double kin = o.mul(fma(u[1][g], u[1][g], o.mul(u[2][g], u[2][g])), ir);
        const double H = o.add(u[3][g], fma(hg, kin, o.mul(gm1, u[3][g])));
        xx = fma(u[1][g], wx, xx);
        xy = fma(u[2][g], wx, xy);
        yy = fma(u[2][g], wy, yy);
        hx = fma(H, wx, hx);
        hy = fma(H, wy, hy);
      }
      const double p = fma(hg, o.add(xx, yy), o.mul(gm1, w0[9 * WC + 1]));  // the mean pressure
      vol[0] = w0[3 * WC + 1];
      vol[1] = o.add(xx, p);
      vol[2] = xy;
      vol[3] = hx;
      vg[0] = w0[6 * WC + 1];
      vg[1] = xy;
      vg[2] = o.add(yy, p);
      vg[3] = hy;
    }
    return true;
  }
};

}  // namespace hw
