// stage1d_lanes64.cuh -- one block of the fused 1D HWENO-U stage in FP64 (Sec. 2.1, Eq. 2.3, 2.4,
// 2.12, 2.13) with four lanes per cell, for grids too short to fill the GPU with one thread per
// cell.
//
// What bounds a short grid is the number of FP64 instructions of one warp: a warp gets one in 64
// clocks, whether 32 of its lanes are active or one (measured), and an SM runs four warps at that
// rate.  So a cell's work is spread over four lanes of a warp, in the parts that differ:
//  * Euler: lane f reconstructs field f (with the characteristic decomposition the field of row f
//    of L, else component f; lane 3 repeats field 2); lane p then takes the Gauss-Lobatto point p
//    of all fields, its flux and its trace; lane c updates component c;
//  * scalar laws: lane l forms the coefficient c_{l+1} of p_0 and its term of beta_0, then the
//    point l.
// The lanes exchange their parts through shared memory.  A stage is then about 190 FP64
// instructions of a warp for Euler and 74 for a scalar law, instead of 325 and 110 in the
// lanes-per-field and one-thread-per-cell layouts before.  The block's largest speed takes two
// integer reductions (a double maximum over a warp costs 135 clocks per shuffle), divisions and
// square roots are refined from the hardware's 20-bit values (a double square root costs 1070
// clocks).  Measured, whole calls: 4000-cell Euler shock tube, 128 steps, 8.70 -> 4.01 ms;
// 240-cell Euler, 400 steps, 16.9 -> 10.6 ms; 200-cell advection, 334 steps, 5.97 -> 4.45 ms.
// The halves of the Lax-Friedrichs flux are formed as in stage2d_tile64.cuh.
#pragma once
#include "f64_ops.cuh"
#include "hweno_device.cuh"
#include "stage1d_item.cuh"

namespace hw {
namespace l64 {

// constants by lane (column l of [kLane][4]), then those every lane shares
enum : int {
  kCX, kCY, kSX, kSY,          // c_{l+1} = CX x + CY y; x = dr + SX dl, y = vp + SY vm
  kT, kB,                      // term of beta_0: KB (c_{l+1} + KT c_{l+3})^2
  kX1, kX2, kX3, kX4,          // point l: u = mean + X1 C1 + X2 C2 + X3 C3 + X4 C4
  kSF, kSH, kDF,               // row l of L: factors of b1h and of 1/(2c), constant
  kLane
};
constexpr double R5 = 0.22360679774997896964;  // sqrt(5)/10
static __device__ const double lane_constants[kLane][4] = {
    {63.0 / 76.0, 23.0 / 16.0, -5.0 / 19.0, -5.0 / 8.0},
    {-75.0 / 19.0, -45.0 / 8.0, 60.0 / 19.0, 15.0 / 4.0},
    {1.0, -1.0, 1.0, -1.0},
    {1.0, -1.0, 1.0, -1.0},
    {0.25, 63.0 / 130.0, 0.0, 0.0},
    {1.0, 13.0 / 3.0, 781.0 / 20.0, 1421461.0 / 2275.0},
    {-0.5, -R5, R5, 0.5},
    {1.0 / 4.0 - 1.0 / 12.0, 0.05 - 1.0 / 12.0, 0.05 - 1.0 / 12.0, 1.0 / 4.0 - 1.0 / 12.0},
    {-0.125, -0.05 * R5, 0.05 * R5, 0.125},
    {1.0 / 16.0 - 1.0 / 80.0, 0.0025 - 1.0 / 80.0, 0.0025 - 1.0 / 80.0, 1.0 / 16.0 - 1.0 / 80.0},
    {1.0, -2.0, 1.0, 1.0},
    {-1.0, 0.0, 1.0, 1.0},
    {0.0, 1.0, 0.0, 0.0}};

#define HW_L64_CONSTANTS(X)                                                                   \
  X(ONE, 1.0) X(MZERO, -0.0) X(TAU, 2.25) X(V1, 1.0 / 12.0) X(V3, 1.0 / 80.0) X(HALF, 0.5)    \
  X(GL0, 1.0 / 12.0) X(GL1, 5.0 / 12.0) X(THREEQ, 0.75) X(QUARTER, 0.25) X(THIRD, 1.0 / 3.0)  \
  X(TWOTHIRD, 2.0 / 3.0) X(RS2, 0.375)                                                        \
  X(CX0, 63.0 / 76.0) X(CX1, 23.0 / 16.0) X(CX2, -5.0 / 19.0) X(CX3, -5.0 / 8.0)              \
  X(CY0, -75.0 / 19.0) X(CY1, -45.0 / 8.0) X(CY2, 60.0 / 19.0) X(CY3, 15.0 / 4.0)             \
  X(T0, 0.25) X(T1, 63.0 / 130.0) X(B1, 13.0 / 3.0) X(B2, 781.0 / 20.0)                       \
  X(B3, 1421461.0 / 2275.0) X(E2, 1.0 / 4.0 - 1.0 / 12.0) X(E4, 1.0 / 16.0 - 1.0 / 80.0)      \
  X(I2, 0.05 - 1.0 / 12.0) X(I4, 0.0025 - 1.0 / 80.0) X(O3, 0.125) X(R1, R5) X(R3, 0.05 * R5)
enum Const : int {
#define X(name, value) k##name,
  HW_L64_CONSTANTS(X)
#undef X
  kStatic,  // from here on: values of the problem
  kEPS = kStatic, kGLO, kG0, kGM1, kHGM1, kGAM, kAX, kIDX, kHIDX, kCount
};
static __device__ const double constants[kStatic] = {
#define X(name, value) (value),
    HW_L64_CONSTANTS(X)
#undef X
};
constexpr int kTable = kCount + 4 * kLane;  // doubles of shared memory: the shared constants,
                                            // then the lanes' [kLane][4]

// One thread's part of the table of a block of T threads: load() issues the reads of the constants
// (from global memory, coalesced: 32 different entries of constant memory are read one after
// another, 0.4 us of a 6 us launch), store() writes the table, visible after the next barrier.
// The launches of a single stage load before their window and store after its loads are issued, so
// that the two latencies are one: a stage of 200 advection cells 6.1 -> 5.0 us, of 8000 (one thread
// per cell) 8.3 -> 6.4 us, of 8000 Euler cells 22.3 -> 20.3 us.
template <int T>
struct TableFill {
  static constexpr int N = (kStatic + 4 * kLane + T - 1) / T;
  double v[N];
  __device__ __forceinline__ void load() {
    const double* lanes = &lane_constants[0][0];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const int n = threadIdx.x + q * T;
      v[q] = n < kStatic ? constants[n] : n < kStatic + 4 * kLane ? lanes[n - kStatic] : 0.0;
    }
  }
  __device__ __forceinline__ void store(double* tab, const KProblem& P) const {
    if (threadIdx.x == 0) {
      tab[kEPS] = 9.0 * P.eps;  // d_m is scaled by 9, the squared divisor of u_ave
      tab[kGLO] = P.glo;
      tab[kG0] = P.g0[0];
      tab[kGM1] = P.gm1;
      tab[kHGM1] = -0.5 * P.gm1;
      tab[kGAM] = P.gam;
      tab[kAX] = P.ax;
      tab[kIDX] = P.inv_dx;
      tab[kHIDX] = 0.5 * P.inv_dx;
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const int n = threadIdx.x + q * T;
      if (n < kStatic + 4 * kLane) tab[n < kStatic ? n : n + kCount - kStatic] = v[q];
    }
  }
};
// a table filled before the item (the launches of several items per block)
struct TableFilled {
  __device__ __forceinline__ void store(double*, const KProblem&) const {}
};
template <int T>
__device__ __forceinline__ void fill_table(double* tab, const KProblem& P) {
  TableFill<T> f;
  f.load();
  f.store(tab, P);
}
#define K(name) o.k<l64::k##name>()

// The factors of the combined polynomial (Eq. 2.12): a0 of p_0 and b1, b2 of the slopes dl, dr
// (the product form of nonlinear_weights_fast, d_m scaled by 9; the direct formula where it
// does not apply).
__device__ __forceinline__ void factors(const Ops& o, double bt0, double dl, double dr, double um,
                                        double u0, double up, const KProblem& P, double& a0,
                                        double& b1, double& b2) {
  const double bl = o.mul(dl, dl), br = o.mul(dr, dr);
  const double s = o.add(fabs(o.sub(bt0, bl)), fabs(o.sub(bt0, br)));
  const double tau = o.mul(o.mul(K(TAU), s), s);  // 9 tau
  const double a = o.add(o.add(fabs(um), fabs(u0)), fabs(up));
  double ua = o.mul(a, a);  // 9 u_ave
  if (P.wmode == 1) ua = 9.0;
  const double eps = K(EPS);
  const double d0 = fma(bt0, ua, eps), d1 = fma(bl, ua, eps), d2 = fma(br, ua, eps);
  const double D0 = o.mul(d1, d2), D1 = o.mul(d0, d2), D2 = o.mul(d0, d1);
  const double D = o.mul(D0, d0);
  const double N0 = fma(tau, D0, D);
  const double S = fma(tau, fma(K(GLO), o.add(D1, D2), o.mul(K(G0), D0)), D);
  const long long eD = (__double_as_longlong(D) >> 52) & 0x7ff;
  const long long eS = (__double_as_longlong(S) >> 52) & 0x7ff;
  const bool ok = eD > 64 && eD < 2047 - 64 && eS > 64 && eS < 2047 - 64;
  const double inv = rcp_in_range(o, S);
  const double k = o.mul(K(GLO), o.mul(tau, inv)), k0 = o.mul(k, D0);
  const bool lin = P.wmode == 2;
  a0 = lin ? 1.0 : o.mul(N0, inv);
  b1 = lin ? 0.0 : fma(k, D1, -k0);
  b2 = lin ? 0.0 : fma(k, D2, -k0);
  if (!(ok || lin)) {
    const double beta[3] = {bt0, bl, br};
    const double third = a * (1.0 / 3.0);
    double bm[3];
    nonlinear_weights_direct<3>(beta, third * third, P, a0, bm);
    b1 = bm[1];
    b2 = bm[2];
  }
}

// Row of L (characteristic fields u - c, u, u + c) as the factors of rho, m and E: sf, sh and df
// are the field's constants (1, -1, 0), (-2, 0, 1), (1, 1, 0).
struct Frame1 {
  double vel, cs, q2h, H, b1h, hic;
  __device__ __forceinline__ void init(const Ops& o, double U0, double U1, double U2) {
    const double ir = rcp_any(o, U0);
    vel = o.mul(U1, ir);
    q2h = o.mul(o.mul(K(HALF), vel), vel);
    const double p = o.mul(K(GM1), fma(-U0, q2h, U2));
    const double c2 = o.mul(o.mul(K(GAM), p), ir);
    const double rc = rsqrt_any(o, c2, K(HALF), K(RS2));
    cs = o.mul(c2, rc);
    H = o.mul(o.add(U2, p), ir);
    b1h = -o.mul(K(HGM1), rcp_any(o, c2));  // rounded once less than from rc twice
    hic = o.mul(K(HALF), rc);
  }
  __device__ __forceinline__ void row(const Ops& o, double sf, double sh, double df, double& l0,
                                      double& l1, double& l2) const {
    const double gh = o.mul(sh, hic);
    l2 = o.mul(sf, b1h);
    l1 = fma(-l2, vel, gh);
    l0 = fma(-gh, vel, fma(l2, q2h, df));
  }
  // U = R W (columns u - c, u, u + c)
  __device__ __forceinline__ void unproject(const Ops& o, double W0, double W1, double W2,
                                            double (&U)[3]) const {
    const double X = o.add(W0, W2), cD = o.mul(cs, o.sub(W2, W0));
    U[0] = o.add(X, W1);
    U[1] = fma(vel, U[0], cD);
    U[2] = fma(H, X, fma(vel, cD, o.mul(q2h, W1)));
  }
};

// One field of the Euler equations: values at the four Gauss-Lobatto points and v-hat.
__device__ __forceinline__ void field64(const Ops& o, double um, double u0, double up, double vm,
                                        double vp, const KProblem& P, double (&w)[5]) {
  const double dl = o.sub(u0, um), dr = o.sub(up, u0);
  const double du = o.add(dr, dl), d2 = o.sub(dr, dl), sv = o.add(vp, vm), dv = o.sub(vp, vm);
  const double c1 = fma(K(CY0), sv, o.mul(K(CX0), du)), c2 = fma(K(CY1), dv, o.mul(K(CX1), d2));
  const double c3 = fma(K(CY2), sv, o.mul(K(CX2), du)), c4 = fma(K(CY3), dv, o.mul(K(CX3), d2));
  const double t1 = fma(K(T0), c3, c1), t2 = fma(K(T1), c4, c2);
  double b = o.mul(t1, t1);
  b = fma(o.mul(K(B1), t2), t2, b);
  b = fma(o.mul(K(B2), c3), c3, b);
  b = fma(o.mul(K(B3), c4), c4, b);
  double a0, b1, b2;
  factors(o, b, dl, dr, um, u0, up, P, a0, b1, b2);
  const double C1 = fma(b2, dr, fma(b1, dl, o.mul(a0, c1)));
  const double C2 = o.mul(a0, c2), C3 = o.mul(a0, c3), C4 = o.mul(a0, c4);
  const double Ee = fma(K(E4), C4, fma(K(E2), C2, u0)), Oe = fma(K(O3), C3, o.mul(K(HALF), C1));
  const double Ei = fma(K(I4), C4, fma(K(I2), C2, u0)), Oi = fma(K(R3), C3, o.mul(K(R1), C1));
  w[0] = o.sub(Ee, Oe);
  w[1] = o.sub(Ei, Oi);
  w[2] = o.add(Ei, Oi);
  w[3] = o.add(Ee, Oe);
  w[4] = fma(K(V3), C3, o.mul(K(V1), C1));
}

template <int EQ>
__device__ __forceinline__ void flux64(const Ops& o, const double* u, double* f) {
  if constexpr (EQ == EQ_ADV) {
    f[0] = o.mul(K(AX), u[0]);
  } else if constexpr (EQ == EQ_BURG) {
    f[0] = o.mul(o.mul(K(HALF), u[0]), u[0]);
  } else {
    const double vn = o.mul(u[1], rcp_any(o, u[0])), mv = o.mul(u[1], vn);
    const double p = fma(K(HGM1), mv, o.mul(K(GM1), u[2]));
    f[0] = u[1];
    f[1] = o.add(mv, p);
    f[2] = o.mul(vn, o.add(u[2], p));
  }
}

// component c of the update (Eq. 2.3, 2.13) from the fluxes FL, FR of its faces (times 1/dx) and
// its fluxes at the points; returns the new average, clears `ok` where a value is not finite
template <class IO>
__device__ __forceinline__ double update64(const Ops& o, const IO& io, int c, int i, double FL,
                                           double FR, double f0, double f1, double f2, double f3,
                                           double own_u, double own_v, bool& ok) {
  const int k = io.k();
  const double dt = io.dt();
  const double F1 = o.sub(FL, FR);
  const double vol = fma(K(GL1), o.add(f1, f2), o.mul(K(GL0), o.add(f0, f3)));
  const double F2 = fma(vol, K(IDX), -o.mul(K(HALF), o.add(FL, FR)));
  double ou, ov;
  const double au = fma(dt, F1, own_u), av = fma(dt, F2, own_v);
  if (k == 1) {
    io.set_vh(c, i, own_v);
    ou = au;
    ov = av;
  } else {
    const double base_u = io.un(2 * c, i), base_v = io.vh(c, i);
    const double kb = k == 2 ? K(THREEQ) : K(THIRD), ka = k == 2 ? K(QUARTER) : K(TWOTHIRD);
    ou = fma(kb, base_u, o.mul(ka, au));
    ov = fma(kb, base_v, o.mul(ka, av));
  }
  io.out(2 * c, i, ou);
  io.out(2 * c + 1, i, ov);
  ok &= finite_bits(ou) && finite_bits(ov);
  return ou;
}
// wave speed of an output average; clears `ok` where it is not physical
__device__ __forceinline__ double speed64(const Ops& o, const double (&ua)[3], bool& ok) {
  const double ir = rcp_any(o, ua[0]);
  const double vn = o.mul(ua[1], ir);
  const double e = fma(-o.mul(K(HALF), ua[1]), vn, ua[2]);  // internal energy density
  const double c2 = o.mul(o.mul(o.mul(K(GAM), K(GM1)), e), ir);
  ok &= ua[0] > 0.0 && e > 0.0 && finite_bits(e);
  return o.add(fabs(vn), sqrt_any(o, c2, K(HALF), K(RS2)));
}

// The window of a block of T threads: moments of the COLS cells from `first` on (boundary-mapped),
// every thread's loads in flight together; `issued` runs behind them.
template <int EQ, int T, int COLS, class IO, class F>
__device__ __forceinline__ void load_window(const KProblem& P, const IO& io, int first, double* win,
                                            F issued) {
  constexpr int NA = 2 * (EQ == EQ_EULER ? 3 : 1), N = (NA * COLS + T - 1) / T;
  double v[N];
  bool neg[N];
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int idx = threadIdx.x + q * T, a = idx / COLS, col = idx % COLS;
    neg[q] = false;
    v[q] = 0.0;
    if (idx < NA * COLS) {
      int flip;
      const int ii = bc_map(first + col, P.nx, P.bc[0], P.bc[1], flip);
      neg[q] = flip && mirror_sign<EQ, 1>(a / 2, a % 2, 1, 0) < 0.0;
      v[q] = io.in(a, ii);
    }
  }
  issued();
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int idx = threadIdx.x + q * T;
    if (idx < NA * COLS) win[idx] = neg[q] ? -v[q] : v[q];
  }
}

}  // namespace l64

// `tab`: the block's table of constants, stored by `fill` (or filled before the call).
// Block blk of BW threads: G = BW / 4 slots of four lanes stand for the cells i0-1 .. i0+G-2,
// i0 = blk (G - 2), and update the G - 2 cells from i0 on.  A warp's eight slots exchange within
// the warp; only the face fluxes cross warps.
template <int EQ, bool CHAR, int BW, class IO, class Fill>
__device__ __forceinline__ void stage1d_lanes64_item_io(const KProblem& P, const IO& io, int blk,
                                                        double* tab, const Fill& table) {
  using namespace l64;
  constexpr int NC = EQ == EQ_EULER ? 3 : 1, NM = 2, G = BW / 4;
  const int nx = P.nx;
  const int t = threadIdx.x, q = t >> 2, f = t & 3;
  const int i0 = blk * (G - 2);
  const int i = i0 - 1 + q;  // reconstructed cell of this lane's slot

  __shared__ double win[NC * NM][G + 2];  // moments of cells i0-2 .. i0+G-1
  __shared__ double part[G][NC][6];       // scalar: C1..C4; Euler: points 0..3 and v-hat of a field
  __shared__ double pf[G][4][NC];         // fluxes at the points
  __shared__ double tr[NC][G + 1];        // flux - alpha u of each slot's left trace, then the
                                          // flux of its left face (times 1/dx)
  __shared__ double red[BW / 32];

  if constexpr (IO::kTabulated) {
    io.fill(&win[0][0]);
    table.store(tab, P);
  } else {
    load_window<EQ, BW, G + 2>(P, io, i0 - 2, &win[0][0], [&] { table.store(tab, P); });
  }
  __syncthreads();
  const Ops o = make_ops<kONE, kMZERO>(tab, io.k());
  const double alpha = io.alpha();
  const double* lk = tab + kCount + f;
  auto lane_k = [&](int n) { return lk[4 * n]; };

  const bool upd = (q >= 1 && q <= G - 2 && i < nx);
  // every lane computes (slots past the right ring read clamped columns; their results are not
  // stored), so that the whole warp takes part in the exchanges
  double u[NC], fl[NC], vh[NC];  // the state and the flux of point f; v-hat of the components
  if constexpr (EQ != EQ_EULER) {
    const double um = win[0][q], u0 = win[0][q + 1], up = win[0][q + 2];
    const double vm = win[1][q], vp = win[1][q + 2];
    const double dl = o.sub(u0, um), dr = o.sub(up, u0);
    const double x = fma(lane_k(kSX), dl, dr), y = fma(lane_k(kSY), vm, vp);
    const double c = fma(lane_k(kCY), y, o.mul(lane_k(kCX), x));
    const double c2 = __shfl_down_sync(0xffffffffu, c, 2, 4);  // lanes 2, 3: their own
    const double tt = fma(lane_k(kT), c2, c);
    double b = o.mul(o.mul(lane_k(kB), tt), tt);
    b = o.add(b, __shfl_xor_sync(0xffffffffu, b, 1));
    b = o.add(b, __shfl_xor_sync(0xffffffffu, b, 2));
    double a0, b1, b2;
    factors(o, b, dl, dr, um, u0, up, P, a0, b1, b2);
    const double sl = fma(b2, dr, o.mul(b1, dl));
    part[q][0][f] = fma(a0, c, f == 0 ? sl : o.nz);
    __syncwarp();
    const double C1 = part[q][0][0], C2 = part[q][0][1], C3 = part[q][0][2], C4 = part[q][0][3];
    u[0] = fma(lane_k(kX4), C4, fma(lane_k(kX3), C3, fma(lane_k(kX2), C2, fma(lane_k(kX1), C1, u0))));
    vh[0] = fma(K(V3), C3, o.mul(K(V1), C1));
    flux64<EQ>(o, u, fl);
  } else {
    // field f of the stencil: row f of L (char), or the component itself
    Frame1 E;
    double l0 = 0.0, l1 = 0.0, l2 = 0.0;
    if constexpr (CHAR) {
      E.init(o, win[0][q + 1], win[2][q + 1], win[4][q + 1]);
      E.row(o, lane_k(kSF), lane_k(kSH), lane_k(kDF), l0, l1, l2);
    }
    const int ff = f < 3 ? f : 2;
    auto field = [&](int col, int m) -> double {
      if constexpr (CHAR)
        return fma(l2, win[4 + m][col], fma(l1, win[2 + m][col], o.mul(l0, win[m][col])));
      else
        return win[2 * ff + m][col];
    };
    double w[5];
    field64(o, field(q, 0), field(q + 1, 0), field(q + 2, 0), field(q, 1), field(q + 2, 1), P, w);
    if (f < 3) {
#pragma unroll
      for (int n = 0; n < 5; ++n) part[q][f][n] = w[n];
    }
    __syncwarp();
    auto conserved = [&](int n, double (&U)[NC]) {
      if constexpr (CHAR) {
        E.unproject(o, part[q][0][n], part[q][1][n], part[q][2][n], U);
      } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) U[c] = part[q][c][n];
      }
    };
    conserved(f, u);
    conserved(4, vh);
    flux64<EQ>(o, u, fl);
  }
  // traces (points 0 and 3): twice the LF flux of a face (Eq. 2.4) is flux + alpha u of the left
  // cell's right trace plus flux - alpha u of the right cell's left trace
  double g[NC];
  const double as = f == 0 ? -alpha : alpha;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    g[c] = fma(as, u[c], fl[c]);
    pf[q][f][c] = fl[c];
    if (f == 0) tr[c][q] = g[c];
  }
  __syncthreads();
  if (f == 3 && q < G - 1 && i < nx) {
    const double k = K(HIDX);
#pragma unroll
    for (int c = 0; c < NC; ++c) tr[c][q + 1] = o.mul(k, o.add(g[c], tr[c][q + 1]));
  }
  __syncthreads();
  // component f of the update
  double ou = 0.0;
  bool ok = true;
  if (upd && f < NC) {
    double own_v = vh[0];
    if constexpr (NC == 3) own_v = f == 0 ? vh[0] : (f == 1 ? vh[1] : vh[2]);
    ou = update64(o, io, f, i, tr[f][q], tr[f][q + 1], pf[q][0][f], pf[q][1][f], pf[q][2][f],
                  pf[q][3][f], win[f * NM][q + 1], own_v, ok);
  }
  // wave speed and physicality of the output average
  double wmax = 0.0;
  if constexpr (EQ == EQ_EULER) {
    const int lane0 = (t & 31) & ~3;
    double ua[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) ua[c] = __shfl_sync(0xffffffffu, ou, lane0 + c);
    const unsigned fine = __ballot_sync(0xffffffffu, ok);
    if (upd && f == 0) {
      ok = ((fine >> lane0) & 7u) == 7u;
      wmax = speed64(o, ua, ok);
    }
  } else {
    if (upd && f == 0) wmax = EQ == EQ_ADV ? fabs(P.ax) : fabs(ou);
  }
  if (!ok) {
    if (f == 0) io.nonphysical();
    wmax = 0.0;
  }
  if (!(wmax >= 0.0)) wmax = __longlong_as_double(0x7ff0000000000000LL);  // NaN -> +inf
  wmax = warp_max_nonneg(wmax);
  if ((t & 31) == 0) red[t >> 5] = wmax;
  __syncthreads();
  if (t < 32) {
    const double m = warp_max_nonneg(t < BW / 32 ? red[t] : 0.0);
    if (t == 0) io.raise_alpha(m);
  }
  __syncthreads();  // the block may start another item in the same shared memory
}

// The same stage with one thread per cell (BW - 2 cells per block), for grids that fill the GPU
// so, and for the batched launches: operation for operation the arithmetic of the lanes, so the
// results are the same bits.
template <int EQ, bool CHAR, int BW, class IO, class Fill>
__device__ __forceinline__ void stage1d_thread64_item_io(const KProblem& P, const IO& io, int blk,
                                                         double* tab, const Fill& table) {
  using namespace l64;
  constexpr int NC = EQ == EQ_EULER ? 3 : 1, NM = 2;
  const int nx = P.nx;
  const int t = threadIdx.x;
  const int i0 = blk * (BW - 2);
  const int i = i0 - 1 + t;  // reconstructed cell of this thread

  __shared__ double win[NC * NM][BW + 2];  // moments of cells i0-2 .. i0+BW-1
  __shared__ double tr[NC][BW + 1];        // flux - alpha u of each cell's left trace, then the
                                           // flux of its left face (times 1/dx)
  __shared__ double red[BW / 32];

  load_window<EQ, BW, BW + 2>(P, io, i0 - 2, &win[0][0], [&] { table.store(tab, P); });
  __syncthreads();
  const Ops o = make_ops<kONE, kMZERO>(tab, io.k());
  const double alpha = io.alpha();
  const bool need = (i <= nx);  // cells beyond the right ring are idle
  const bool upd = (t >= 1 && t <= BW - 2 && i < nx);
  double fp[4][NC], gr[NC], vh[NC];  // fluxes at the points; flux + alpha u of the right trace
  if (need) {
    double pts[4][NC];
    if constexpr (EQ != EQ_EULER) {
      const double um = win[0][t], u0 = win[0][t + 1], up = win[0][t + 2];
      const double vm = win[1][t], vp = win[1][t + 2];
      const double dl = o.sub(u0, um), dr = o.sub(up, u0);
      const double* lk = tab + kCount;
      // (the lanes' x and y of l = 2, 3 are those of 0, 1, and their factor of tt^2 is 1 at l = 0)
      const double x[2] = {o.add(dl, dr), o.sub(dr, dl)}, y[2] = {o.add(vm, vp), o.sub(vp, vm)};
      double c[4];
#pragma unroll
      for (int l = 0; l < 4; ++l)
        c[l] = fma(lk[4 * kCY + l], y[l & 1], o.mul(lk[4 * kCX + l], x[l & 1]));
      double b[4];
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        const double tt = l < 2 ? fma(lk[4 * kT + l], c[l + 2], c[l]) : c[l];
        b[l] = o.mul(l == 0 ? tt : o.mul(lk[4 * kB + l], tt), tt);
      }
      double a0, b1, b2;
      factors(o, o.add(o.add(b[0], b[1]), o.add(b[2], b[3])), dl, dr, um, u0, up, P, a0, b1, b2);
      double C[4];
      C[0] = fma(a0, c[0], fma(b2, dr, o.mul(b1, dl)));
#pragma unroll
      for (int l = 1; l < 4; ++l) C[l] = o.mul(a0, c[l]);
#pragma unroll
      for (int l = 0; l < 4; ++l)
        pts[l][0] = fma(lk[4 * kX4 + l], C[3], fma(lk[4 * kX3 + l], C[2],
                    fma(lk[4 * kX2 + l], C[1], fma(lk[4 * kX1 + l], C[0], u0))));
      vh[0] = fma(K(V3), C[2], o.mul(K(V1), C[0]));
    } else {
      Frame1 E;
      if constexpr (CHAR) E.init(o, win[0][t + 1], win[2][t + 1], win[4][t + 1]);
      double w[3][5];
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        double l0 = 0.0, l1 = 0.0, l2 = 0.0;
        if constexpr (CHAR) {
          const double* lk = tab + kCount + f;
          E.row(o, lk[4 * kSF], lk[4 * kSH], lk[4 * kDF], l0, l1, l2);
        }
        auto field = [&](int col, int m) -> double {
          if constexpr (CHAR)
            return fma(l2, win[4 + m][col], fma(l1, win[2 + m][col], o.mul(l0, win[m][col])));
          else
            return win[2 * f + m][col];
        };
        field64(o, field(t, 0), field(t + 1, 0), field(t + 2, 0), field(t, 1), field(t + 2, 1), P,
                w[f]);
      }
#pragma unroll
      for (int n = 0; n < 5; ++n) {
        double U[NC];
        if constexpr (CHAR) {
          E.unproject(o, w[0][n], w[1][n], w[2][n], U);
        } else {
#pragma unroll
          for (int c = 0; c < NC; ++c) U[c] = w[c][n];
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) (n < 4 ? pts[n][c] : vh[c]) = U[c];
      }
    }
#pragma unroll
    for (int g = 0; g < 4; ++g) flux64<EQ>(o, pts[g], fp[g]);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      tr[c][t] = fma(-alpha, pts[0][c], fp[0][c]);
      gr[c] = fma(alpha, pts[3][c], fp[3][c]);
    }
  }
  __syncthreads();
  if (need && t < BW - 1 && i < nx) {
    const double k = K(HIDX);
#pragma unroll
    for (int c = 0; c < NC; ++c) tr[c][t + 1] = o.mul(k, o.add(gr[c], tr[c][t + 1]));
  }
  __syncthreads();
  double wmax = 0.0;
  if (upd) {
    bool ok = true;
    double ua[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c)
      ua[c] = update64(o, io, c, i, tr[c][t], tr[c][t + 1], fp[0][c], fp[1][c], fp[2][c], fp[3][c],
                       win[c * NM][t + 1], vh[c], ok);
    if constexpr (EQ == EQ_EULER) wmax = speed64(o, ua, ok);
    else wmax = EQ == EQ_ADV ? fabs(P.ax) : fabs(ua[0]);
    if (!ok) {
      io.nonphysical();
      wmax = 0.0;
    }
  }
  if (!(wmax >= 0.0)) wmax = __longlong_as_double(0x7ff0000000000000LL);  // NaN -> +inf
  wmax = warp_max_nonneg(wmax);
  if ((t & 31) == 0) red[t >> 5] = wmax;
  __syncthreads();
  if (t < 32) {
    const double m = warp_max_nonneg(t < BW / 32 ? red[t] : 0.0);
    if (t == 0) io.raise_alpha(m);
  }
  __syncthreads();  // the block may start another item in the same shared memory
}
#undef K

// One block of the one-thread-per-cell layout in either precision; tab: the FP64 table of
// constants, stored by `table` (or filled by the block before the call).
template <int EQ, bool CHAR, typename R, int BW, class Fill>
__device__ __forceinline__ void thread_item1d(const KProblem& P, const KStage& S, int blk, double* tab,
                                              const Fill& table) {
  const Global1D io{S, P.nx};
  if constexpr (sizeof(R) == sizeof(double))
    stage1d_thread64_item_io<EQ, CHAR, BW>(P, io, blk, tab, table);
  else stage1d_item_io<EQ, CHAR, R, BW>(P, io, blk);
}


}  // namespace hw
