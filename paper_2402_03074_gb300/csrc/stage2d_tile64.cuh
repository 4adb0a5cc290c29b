// stage2d_tile64.cuh -- one work item of the fused 2D HWENO-U stage in FP64 (Sec. 2.2, Eq. 2.16,
// 2.23, 2.13), every equation; shared by the single-solve kernel (stage2d_impl.cuh) and the
// batched ones (batch.cu, static_batch.cu).
//
// Decomposition: a block owns a band of wout <= BX-2 output columns and a chunk of output rows
// [j0, j1).  Its BX x BY threads stand for the columns i0-1 .. i0+wout (the band plus one ring
// column on each side) of BY consecutive rows, and sweep the rows j0-1 .. j1 BY at a time.  Every
// thread reconstructs its cell from a row window of the stage input in shared memory; the x-face
// fluxes of a row are formed once per face by the row's own threads, the y-face fluxes once per
// face by the threads above the face, from the traces below it (those of the tile's last row
// carried to the next step).  A row is complete once the face above it is: the tile's last row
// one step later.  Redundant work is the two ring columns per band and the y traces of the two
// ring rows per chunk.
//
// Why BY rows at once: an SM needs six to eight warps to keep its FP64 unit busy (a warp alone gets
// one FP64 instruction in 64 clocks, the SM one in 16), and a chunk of r rows costs r + 0.9 rows
// of work (the ring rows' y passes).  With one row at a time, six warps are two 96-column blocks
// each with its own ring rows, and a grid of 240^2 cells in chunks of 3 rows spends a quarter of
// its work on ring rows and idle lanes; one block of 32 x 8 covers 13 rows in 30 columns.
// Measured (whole calls; before: characteristic Euler one row at a time in two 96-thread blocks
// per SM, the other classes in 128-thread blocks of the field-by-field arithmetic; then the tiles
// of six or seven warps; then the present ones, with their reciprocals on integers): 240^2 Euler,
// 12 steps, 17.3, 11.9, 10.05 ms; 40^2 Euler, 24 steps, 13.6, 7.27, 7.32 ms; 517 x 389 Euler, one
// step, 3.33, 3.27, 3.15 ms; 2048^2 Euler, one step, 56.5, 56.4, 54.5 ms; 240^2 Burgers, 48 steps,
// 17.0, 8.05, 7.01 ms; 768^2 component-wise Euler, one step, 8.39, 5.50, 5.19 ms.
//
// The Lax-Friedrichs flux.  Twice the flux of a face is f(uL) + f(uR) - a (uR - uL) (Eq. 2.4); each
// cell forms its half alone, f(u) - a u on its low edges and f(u) + a u on its high ones, so that one
// number per point and component crosses the face and not two (the second set would not fit the
// shared memory of the 64 x 4 tile).  The halves are rounded at the scale of a u, which the jump does
// not have: the first moments of a uniform flow at 1e-6 of the sound speed come out as 4e-18 of the
// average and not as 1e-24.  On waves and Riemann data it does not show: the stages' rms errors
// against an evaluation in long double (tests/test_gpu_rounding.py) are 4.1e-17 to 7.1e-17 of the
// scale (averages) and 0.8e-17 to 1.7e-17 (first moments), 4 to 33 % below those of the kernels
// before, which formed the jump first, and within 6 % of those with u measured from the average of
// the cell below the edge, which both its cells know and which makes the subtraction as good as the
// jump's.  That form costs 48 FP64 operations per cell: 2048^2 54.5 -> 55.7 ms, 768^2 component-wise
// 5.19 -> 5.34 ms, 240^2 Burgers 6.98 -> 7.18 ms.
#pragma once
#include "stage2d_char64.cuh"
#include "stage2d_comp64.cuh"

namespace hw {

template <int EQ, bool CHAR, int T, int WC>
struct Cell64 {
  using type = Comp64Cell<EQ, T, WC>;
};
template <int T, int WC>
struct Cell64<EQ_EULER, true, T, WC> {
  using type = Char64Cell<T, WC>;
};

// Shared memory of a block: the row window [BY + 2][NA][BX + 2]; per thread the x-face exchange
// (3 NC: flux - a u of the low trace, then the Gauss moments of the face's flux), the high y
// traces (3 NC, and BX columns more: the tile's last row in turns), the y-face moments (2 NC)
// and the cell's column; and the table of constants.  In the Euler tiles of eight warps the y-face
// moments lie in the exchange (kSharedFaces; one more barrier between steps): it would be 235 KB.
template <int EQ, int BX, int BY>
constexpr bool kSharedFaces = EQ == EQ_EULER && BX * BY == 256;
template <int EQ, bool CHAR, int BX, int BY>
constexpr size_t smem_bytes_tile64() {
  using Cell = typename Cell64<EQ, CHAR, BX * BY, BX + 2>::type;
  constexpr int NC = Cell::NC;
  return sizeof(double) * ((BY + 2) * 3 * NC * (BX + 2) +
                           ((kSharedFaces<EQ, BX, BY> ? 6 : 8) * NC + Cell::kCols) * BX * BY +
                           3 * NC * BX + c64::kTable);
}

template <int EQ, bool CHAR, int BX, int BY>
__device__ __forceinline__ void stage2d_tile64_item(const KProblem& P, const KStage& S, int band,
                                                    int j0, int j1, int wout, double* smem,
                                                    double (*red)[BX * BY / 32]) {
  using namespace c64;
  constexpr int T = BX * BY, WC = BX + 2;
  using Cell = typename Cell64<EQ, CHAR, T, WC>::type;
  constexpr int NC = Cell::NC, NA = 3 * NC, NR = BY + 2;
  static_assert(BX % 32 == 0 && 2 * NA <= BX, "a warp is in one row; the window's last columns");
  const int t = threadIdx.x;
  const int tx = t % BX, ty = t / BX;  // ty is uniform over a warp
  double* win = smem;
  double* xch = win + NR * NA * WC + t;        // [3 NC][T], this thread's column
  double* car = win + NR * NA * WC + NA * T;   // [BY + 1][3 NC][BX]
  double* fm = kSharedFaces<EQ, BX, BY> ? win + NR * NA * WC : car + (BY + 1) * NA * BX;  // [2 NC][T]
  double* col = car + (BY + 1) * NA * BX + (kSharedFaces<EQ, BX, BY> ? 0 : 2 * NC * T);   // [kCols][T]
  double* tab = col + Cell::kCols * T;
  fill_table(tab, P);
  const int nx = P.nx, ny = P.ny;
  const size_t plane = (size_t)nx * ny;
  const int i0 = band * wout;
  const int i = i0 - 1 + tx;
  const bool lane = (tx <= wout + 1) && (i <= nx);
  const bool outc = (tx >= 1 && tx <= wout && i < nx);
  const double a1 = S.alpha_in[0], a2 = S.alpha_in[1];
  const double dt = *S.dt;

  // window column tx of a row is loaded by thread tx of a row group, the two last columns by
  // threads 0 .. 2 NA - 1
  int fx0, fx1;
  const int ii0 = bc_map(i0 - 2 + tx, nx, P.bc[0], P.bc[1], fx0);
  const int ii1 = bc_map(i0 - 2 + BX + tx / NA, nx, P.bc[0], P.bc[1], fx1);
  auto load_row = [&](int r) {
    int fy;
    const int rr = bc_map(r, ny, P.bc[2], P.bc[3], fy);
    double* dst = win + ((r - j0 + 2) % NR) * NA * WC;  // r >= j0 - 2
    const double* src = S.Uin + (size_t)rr * nx;
    double v[NA], v1 = 0.0;
    const int a1_ = tx % NA;
#pragma unroll
    for (int a = 0; a < NA; ++a) v[a] = src[(size_t)a * plane + ii0];
    if (tx < 2 * NA) v1 = src[(size_t)a1_ * plane + ii1];
    if (fx0 | fy) {
#pragma unroll
      for (int a = 0; a < NA; ++a) v[a] *= mirror_sign<EQ, 2>(a / 3, a % 3, fx0, fy);
    }
    if (tx < 2 * NA && (fx1 | fy)) v1 *= mirror_sign<EQ, 2>(a1_ / 3, a1_ % 3, fx1, fy);
#pragma unroll
    for (int a = 0; a < NA; ++a) dst[a * WC + tx] = v[a];
    if (tx < 2 * NA) dst[a1_ * WC + BX + tx / NA] = v1;
  };
#pragma unroll 1
  for (int r = j0 - 2 + ty; r <= j0 - 1 + BY && r <= j1 + 1; r += BY) load_row(r);
  __syncthreads();
  const Ops o = make_ops<kONE, kMZERO>(tab, S.k);
  // the threads of a row wait for each other (named barrier of the row; a warp on its own)
  auto row_sync = [&]() {
    if constexpr (BX == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + ty), "n"(BX) : "memory");
  };

  // the row waiting for the face above it (used by the threads of the tile's last row)
  double pend[NC][3], pvh[NC], pwh[NC];
#pragma unroll
  for (int a = 0; a < NC; ++a) pend[a][0] = pend[a][1] = pend[a][2] = pvh[a] = pwh[a] = 0.0;
  double wmax0 = 0.0, wmax1 = 0.0;
  bool fast = true;

#pragma unroll 1
  for (int step = 0;; ++step) {
    const int jb = j0 - 1 + step * BY;
    if (jb > j1) break;  // uniform over the block
    const int j = jb + ty;
    const bool xrow = (j >= j0 && j < j1);   // uniform over a row group, as j <= j1
    const bool need = lane && j <= j1;
    const int slot = step * BY + ty;         // of the row below
    const double* wm = win + (slot % NR) * NA * WC + tx;
    const double* w0 = win + ((slot + 1) % NR) * NA * WC + tx;
    const double* wp = win + ((slot + 2) % NR) * NA * WC + tx;
    // the high y traces of row ty; the last row's alternate between two slots
    double* cmine = car + (ty < BY - 1 ? ty : BY - 1 + (step & 1)) * NA * BX + tx;
    const double* cbelow = car + (ty > 0 ? ty - 1 : BY - 1 + ((step + 1) & 1)) * NA * BX + tx;

    double rx[NC][3];                // right-hand side of (i, j) without its top face
    double vh[NC], wh[NC];
    double gb[3][NC];                // g - a2 u of the bottom traces
#pragma unroll
    for (int a = 0; a < NC; ++a) rx[a][0] = rx[a][1] = rx[a][2] = vh[a] = wh[a] = 0.0;
    {
      Cell cell(P, o, wm, w0, wp, col + t);
      if (need) fast &= cell.begin(xrow);
      if (xrow) {
        double glo[3][NC], ghi[3][NC], vol[NC];
        if (need) {
          fast &= cell.template pass<0>(xrow, a1, glo, ghi, vol, vh);
          // x faces: twice the LF flux of a face is f + a u of the left cell's high trace plus
          // f - a u of the right cell's low trace; formed once, by the thread left of the face
#pragma unroll
          for (int g = 0; g < 3; ++g)
#pragma unroll
            for (int a = 0; a < NC; ++a) xch[(a * 3 + g) * T] = glo[g][a];
        }
        row_sync();
        if (need && tx <= wout && i < nx) {
          const double k0 = K(FX0), k1 = K(FX1), k2 = K(FX2);
#pragma unroll
          for (int a = 0; a < NC; ++a) {
            double* x = xch + a * 3 * T + 1;  // the right neighbour's column
            const double F0 = o.add(ghi[0][a], x[0]), F1 = o.add(ghi[1][a], x[T]),
                         F2 = o.add(ghi[2][a], x[2 * T]);
            x[0] = fma(k1, F1, o.mul(k0, o.add(F0, F2)));  // this thread is its only reader
            x[T] = o.mul(k2, o.sub(F2, F0));
          }
        }
        row_sync();
        if (outc) {
          const double idx = K(IDX), half = K(HALF);
#pragma unroll
          for (int a = 0; a < NC; ++a) {
            const double* x = xch + a * 3 * T;
            const double Lw = x[0], Rw = x[1];
            rx[a][0] = o.sub(Lw, Rw);
            rx[a][1] = fma(vol[a], idx, -o.mul(half, o.add(Lw, Rw)));
            rx[a][2] = o.sub(x[T], x[T + 1]);
          }
        }
      }
      if (need) {
        double gt[3][NC], vol[NC];
        fast &= cell.template pass<1>(xrow, a2, gb, gt, vol, wh);
#pragma unroll
        for (int g = 0; g < 3; ++g)
#pragma unroll
          for (int a = 0; a < NC; ++a) cmine[(a * 3 + g) * BX] = gt[g][a];
        if (xrow) {
          const double idy = K(IDY);
#pragma unroll
          for (int a = 0; a < NC; ++a) rx[a][2] = fma(vol[a], idy, rx[a][2]);
        }
      }
    }
    __syncthreads();  // the step's traces are in place and nothing reads the window any more

    // the y face below row j (Eq. 2.16), formed once, by the threads above it
    if (need && j > j0 - 1) {
      const double k0 = K(FY0), k1 = K(FY1), k2 = K(FY2), half = K(HALF);
#pragma unroll
      for (int a = 0; a < NC; ++a) {
        const double G0 = o.add(cbelow[(a * 3 + 0) * BX], gb[0][a]),
                     G1 = o.add(cbelow[(a * 3 + 1) * BX], gb[1][a]),
                     G2 = o.add(cbelow[(a * 3 + 2) * BX], gb[2][a]);
        const double sw = fma(k1, G1, o.mul(k0, o.add(G0, G2)));
        const double sm = o.mul(k2, o.sub(G2, G0));
        fm[(2 * a) * T + t] = sw;
        fm[(2 * a + 1) * T + t] = sm;
        rx[a][0] = o.add(rx[a][0], sw);
        rx[a][1] = o.add(rx[a][1], sm);
        rx[a][2] = fma(-half, sw, rx[a][2]);
      }
    }
    // the window's next BY rows, into the slots of the rows no longer needed
    if (j + BY + 1 <= j1 + 1) load_row(j + BY + 1);
    __syncthreads();

    // the row whose top face is now known: this thread's row j, or in the tile's last row the
    // one it processed a step ago (row j takes its place)
    const bool last = ty == BY - 1;
    const int jc = last ? j - BY : j;
    const double* face = fm + (last ? tx : t + BX);
    if (last) {
#pragma unroll
      for (int a = 0; a < NC; ++a) {
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const double x = rx[a][m];
          rx[a][m] = pend[a][m];
          pend[a][m] = x;
        }
        const double x = vh[a], y = wh[a];
        vh[a] = pvh[a];
        wh[a] = pwh[a];
        pvh[a] = x;
        pwh[a] = y;
      }
    }
    if (outc && jc >= j0 && jc < j1) {
      // its stage update: Eq. 2.13
      const size_t q = (size_t)jc * nx + i;
      const double half = K(HALF);
      double ua[NC];
      bool bad = false;
#pragma unroll
      for (int a = 0; a < NC; ++a) {
        const double sw = face[(2 * a) * T], sm = face[(2 * a + 1) * T];
        const double F[3] = {o.sub(rx[a][0], sw), o.sub(rx[a][1], sm), fma(-half, sw, rx[a][2])};
        const double own[3] = {S.Uin[(size_t)(a * 3) * plane + q], vh[a], wh[a]};
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
          const double adv = fma(dt, F[m], own[m]);
          double out;
          if (S.k == 1) out = adv;
          else if (S.k == 2) out = fma(K(THREEQ), base, o.mul(K(QUARTER), adv));
          else out = fma(K(THIRD), base, o.mul(K(TWOTHIRD), adv));
          S.Uout[qa] = out;
          bad |= !finite_bits(out);
          if (m == 0) ua[a] = out;
        }
      }
      if constexpr (EQ == EQ_EULER) {
        double s0, s1;
        bad |= !speeds(o, ua, s0, s1);
        if (!bad) {
          wmax0 = fmax(wmax0, s0);
          wmax1 = fmax(wmax1, s1);
        }
      } else {
        wmax0 = fmax(wmax0, Phys<EQ, double>::speed(P, 0, ua));
        wmax1 = fmax(wmax1, Phys<EQ, double>::speed(P, 1, ua));
      }
      if (bad) atomicOr(S.status, kStatusNonphysical);
    }
    if constexpr (kSharedFaces<EQ, BX, BY>)
      if (jb + BY <= j1) __syncthreads();  // the faces' place is written next (uniform)
  }

  // block maxima of the output wave speeds -> one atomic per block and direction
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    wmax0 = fmax(wmax0, __shfl_xor_sync(0xffffffffu, wmax0, d));
    wmax1 = fmax(wmax1, __shfl_xor_sync(0xffffffffu, wmax1, d));
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
    for (int w = 1; w < T / 32; ++w) {
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
