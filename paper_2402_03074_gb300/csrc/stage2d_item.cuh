// stage2d_item.cuh -- one work item of the fused 2D HWENO-U stage (Sec. 2.2, Eq. 2.16, 2.23,
// 2.13), shared by the single-solve kernel (stage2d_impl.cuh) and the batched ones (batch.cu,
// static_batch.cu): the tile of a class, and the item in FP32-bulk arithmetic (the FP64 item:
// stage2d_tile64.cuh).
//
// Decomposition, as in FP64: a block owns a band of wout <= BX-2 output columns and a chunk of
// output rows [j0, j1).  Its BX x BY threads stand for the columns i0-1 .. i0+wout (the band plus
// one ring column on each side) of BY consecutive rows, and sweep the rows j0-1 .. j1 BY at a
// time.  Every thread reconstructs its cell (i, j) once from a (BY + 2)-row shared-memory window
// of the stage input; the x-face fluxes of a row are formed once per face through shared memory
// by the row's threads, the y-face fluxes once per face by the threads above the face from the
// traces below it (those of the tile's last row carried to the next step).  A row is complete
// once the face above it is (the tile's last row one step later): its stage update is written
// and the wave speed of the output is folded into a block maximum.  Redundant work is the two
// ring columns per band and the two ring rows per chunk (x pass skipped on ring rows).
#pragma once
#include "geometry.h"
#include "hweno_device.cuh"
#include "stage2d_tile64.cuh"

namespace hw {

// Tile of a block: bands of at most BW - 2 columns, kTileRows rows at once (geometry.h).
template <typename R, int BW>
constexpr int kTileRows = sizeof(R) == sizeof(double) ? tile_rows64(BW) : tile_rows32(BW);
template <typename R, int BW>
constexpr int kThreads2D = BW * kTileRows<R, BW>;

// Resident blocks per SM the 2D stage kernels are compiled for: the FP64 Euler kernels take the
// register file and the shared memory with one block of 256 threads, the
// scalar FP64 ones two; the FP32-bulk kernels twelve warps (at most 168 registers per thread),
// which hides more of the FP64 latency of their weight evaluation.
template <int EQ, typename R, int BW>
constexpr int kMinBlocks2D =
    sizeof(R) == sizeof(double) ? (EQ == EQ_EULER ? 1 : 2) : 384 / kThreads2D<R, BW>;

// Gauss weights on [-1/2, 1/2] (sum 1) and nodes
#define GW0 (5.0 / 18.0)
#define GW1 (4.0 / 9.0)

template <int EQ, typename R>
__device__ __forceinline__ void flux_dir(const KProblem& P, int dir, const R* u, R* f) {
  if constexpr (EQ == EQ_EULER) euler_flux<2, R>(P, dir, u, f);
  else Phys<EQ, R>::flux(P, dir, u, f);
}

// sum_g sum_h w_g w_h f(u(xi_g, eta_h)) over the 3x3 interior points (index 3g+h)
template <int EQ, int NC, typename R>
__device__ __forceinline__ void volume_sum(const KProblem& P, int dir, const R (&in)[9][NC],
                                           R (&vol)[NC]) {
  const R wc = R(GW0 * GW0), we = R(GW0 * GW1), wm = R(GW1 * GW1);
#pragma unroll
  for (int c = 0; c < NC; ++c) vol[c] = R(0);
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    R f[NC];
    flux_dir<EQ, R>(P, dir, in[p], f);
    const int g = p / 3, h = p % 3;
    const R wgt = (g == 1 && h == 1) ? wm : ((g == 1 || h == 1) ? we : wc);
#pragma unroll
    for (int c = 0; c < NC; ++c) vol[c] += wgt * f[c];
  }
}

// One work item: band `band` (output columns band*wout .. +wout-1) and the output rows
// [j0, j1) of one stage of one solve, processed by a whole block.
// smem: dynamic shared memory of smem_bytes2d<EQ, CHAR, R, BW>(); red: two doubles per warp.
// In FP32-bulk the row window holds the stage input in the bulk precision (converted once per
// value when a row is loaded), and the FP64 update reads the cell's own averages from global
// memory.

// Shared memory of a block, FP32-bulk: the table of constants, the (BY + 2)-row window, the
// x-face exchange, the y-face moments and the top traces (in shared memory rather than in
// registers: fewer spills, stages 2 % faster).
template <int EQ, bool CHAR, typename R, int BW>
constexpr size_t smem_bytes2d() {
  constexpr int NC = (EQ == EQ_EULER) ? 4 : 1;
  if constexpr (sizeof(R) == sizeof(double))
    return smem_bytes_tile64<EQ, CHAR, BW, kTileRows<R, BW>>();
  constexpr int BY = kTileRows<R, BW>;
  return sizeof(double) * c64::kTable +
         sizeof(R) * ((BY + 2) * 3 * NC * (BW + 2) + (6 + 2) * NC * BW * BY +
                      6 * NC * BW * (BY + 1));
}

// Steps 2 and 3 of one field in FP64 from its FP32 Appendix coefficients c and averages u (of
// cells 2, 4, 5, 6, 8 are read), by the operations of recon64.cuh in unscaled coordinates: beta_0
// as in the FP64 kernels, the weights in the product form.  On return c is the combined
// polynomial (Eq. 2.23) a0 p_0 + sum_m b_m p_m, formed in FP32 from the rounded a0, 1 - a0
// and b_m.  Returns false where the direct formula was needed.
//
// These operations bound the FP32-bulk kernels (the SM takes an FP64 instruction of a warp in 16
// clocks, FP32 ones in a quarter).  93 per field as three-register FMAs (f64_ops.cuh) instead of
// 117 in plain operators: 2048^2 step 24.6 -> 22.1 ms.  One evaluation of the entropy field for
// both passes would take 20.3 ms, but the passes' FP32 coefficients of it round differently, and
// the results would move by that.
template <typename R>
__device__ __forceinline__ bool weigh_field(const Ops& o, const R (&u)[9], const KProblem& P,
                                            R (&c)[15]) {
  double d[15];
#pragma unroll
  for (int n = 1; n < 15; ++n) d[n] = to_f64(c[n]);
  const double e[4] = {to_f64(u[4] - u[3]), to_f64(u[5] - u[4]), to_f64(u[4] - u[1]),
                       to_f64(u[7] - u[4])};
  const double a = o.add(o.add(o.add(to_f64(fabs(u[1])), to_f64(fabs(u[3]))),
                               o.add(to_f64(fabs(u[4])), to_f64(fabs(u[5])))),
                         to_f64(fabs(u[7])));
  double a0, bm[5];
  const bool fast = c64::weights(o, c64::beta0(o, d), e, a, P, a0, bm);
  const R f0 = from_f64<R>(a0), om = from_f64<R>(o.sub(o.one, a0));
  const R b1 = from_f64<R>(bm[1]), b2 = from_f64<R>(bm[2]), b3 = from_f64<R>(bm[3]),
          b4 = from_f64<R>(bm[4]);
  combine2d<R>(c, u, f0, om, b1, b2, b3, b4, c);
  return fast;
}

template <int EQ, bool CHAR, typename R, int BX, int BY>
__device__ __forceinline__ void stage2d_mixed_item(const KProblem& P, const KStage& S, int band,
                                                   int j0, int j1, int wout, double* smem,
                                                   double (*red)[BX * BY / 32]) {
  constexpr int NC = (EQ == EQ_EULER) ? 4 : 1;
  constexpr int NM = 3;
  constexpr int NA = NC * NM, T = BX * BY, NR = BY + 2;
  constexpr int WC = BX + 2;  // window columns: global columns i0-2 .. i0+BX-1
  const int t = threadIdx.x;
  const int tx = t % BX, ty = t / BX;  // ty is uniform over a warp
  // rows of the stage input for the reconstruction of the tile's rows, row r in slot
  // (r - j0 + 2) mod NR
  c64::fill_table<false>(smem, P);
  R* win = reinterpret_cast<R*>(smem + c64::kTable);    // [NR][NA][WC]
  // x-face exchange of the thread's row, [NC][3][2][BX]: the left trace u and its flux f of every
  // thread's cell; the face flux at the left face of thread x's cell then overwrites the u
  // slot x (its only reader, thread x - 1, has read it by then)
  R* trL = win + NR * NA * WC + ty * NC * 3 * 2 * BX;
  auto fhx = [&](int cg, int x) -> R& { return trL[(cg * 2 + 0) * BX + x]; };
  // the rows' top traces and g of them, [BY + 1][2][3][NC][BX] (the tile's last row alternates
  // between two slots, as it is read a step later)
  R* car = win + NR * NA * WC + NC * 3 * 2 * T;
  // Gauss moments of the face below each row, [2 NC][T]
  R* fm = car + (BY + 1) * 6 * NC * BX;

  const int nx = P.nx, ny = P.ny;
  const size_t plane = (size_t)nx * ny;
  const int i0 = band * wout;   // wout <= BX - 2 output columns per band
  const int i = i0 - 1 + tx;
  const bool lane = (tx <= wout + 1) && (i <= nx);
  const bool outc = (tx >= 1 && tx <= wout && i < nx);
  const R a1 = (R)S.alpha_in[0], a2 = (R)S.alpha_in[1];
  const double dt = *S.dt;
  const R idx = kconst<R>(P.inv_dx, P.inv_dxf), idy = kconst<R>(P.inv_dy, P.inv_dyf);
  const R s15 = R(HW_S15);

  // window column tx of a row is loaded by thread tx of a row's threads, the two last columns by
  // threads 0 .. 2 NA - 1
  int fx0, fx1;
  const int ii0 = bc_map(i0 - 2 + tx, nx, P.bc[0], P.bc[1], fx0);
  const int ii1 = bc_map(i0 - 2 + BX + tx / NA, nx, P.bc[0], P.bc[1], fx1);
  auto load_row = [&](int r) {
    int fy;
    const int rr = bc_map(r, ny, P.bc[2], P.bc[3], fy);
    R* dst = win + ((r - j0 + 2) % NR) * NA * WC;  // r >= j0 - 2
    const double* src = S.Uin + (size_t)rr * nx;
    double v[NA], v1 = 0.0;
    const int a1_ = tx % NA;
#pragma unroll
    for (int a = 0; a < NA; ++a) v[a] = src[(size_t)a * plane + ii0];
    if (tx < 2 * NA) v1 = src[(size_t)a1_ * plane + ii1];
    if (fx0 | fy) {
#pragma unroll
      for (int a = 0; a < NA; ++a) v[a] *= mirror_sign<EQ, 2>(a / NM, a % NM, fx0, fy);
    }
    if (tx < 2 * NA && (fx1 | fy)) v1 *= mirror_sign<EQ, 2>(a1_ / NM, a1_ % NM, fx1, fy);
#pragma unroll
    for (int a = 0; a < NA; ++a) dst[a * WC + tx] = from_f64<R>(v[a]);
    if (tx < 2 * NA) dst[a1_ * WC + BX + tx / NA] = from_f64<R>(v1);
  };
#pragma unroll 1
  for (int r = j0 - 2 + ty; r <= j0 - 1 + BY && r <= j1 + 1; r += BY) load_row(r);
  __syncthreads();
  const Ops o = make_ops<c64::kONE, c64::kMZERO>(smem, S.k);
  // the threads of a row wait for each other (named barrier of the row; a warp on its own)
  auto row_sync = [&]() {
    if constexpr (BX == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + ty), "n"(BX) : "memory");
  };

  // the row waiting for the face above it (used by the threads of the tile's last row)
  R pend[NC][3];
  R pvh[NC], pwh[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) pend[c][0] = pend[c][1] = pend[c][2] = pvh[c] = pwh[c] = R(0);
  double wmax0 = 0.0, wmax1 = 0.0;
  bool fast_weights = true;        // cleared where the direct-formula weights were needed

#pragma unroll 1
  for (int step = 0;; ++step) {
    const int jb = j0 - 1 + step * BY;
    if (jb > j1) break;  // uniform over the block
    const int j = jb + ty;
    const bool need = lane && j <= j1;
    const int slot = step * BY + ty;  // of the row below
    const R* wm = win + (slot % NR) * NA * WC;
    const R* w0 = win + ((slot + 1) % NR) * NA * WC;
    const R* wp = win + ((slot + 2) % NR) * NA * WC;
    auto Wv = [&](int a, int k) -> R {   // moment array a of stencil cell k (0..8)
      const R* rowp = (k < 3) ? wm : (k < 6 ? w0 : wp);
      return rowp[a * WC + tx + (k % 3)];
    };
    const bool xrow = (j >= j0 && j < j1);  // uniform over a row's threads
    R* cmine = car + (ty < BY - 1 ? ty : BY - 1 + (step & 1)) * 6 * NC * BX + tx;
    const R* cbelow = car + (ty > 0 ? ty - 1 : BY - 1 + ((step + 1) & 1)) * 6 * NC * BX + tx;

    R xl[3][NC], xr[3][NC], volf[NC], vh[NC];
    R yb[3][NC], yt[3][NC], volg[NC], wh[NC];
    R rx[NC][3];                     // x-face and f-volume part of the RHS of (i, j)
#pragma unroll
    for (int c = 0; c < NC; ++c) rx[c][0] = rx[c][1] = rx[c][2] = R(0);

    // x faces of row j (output rows only): traces through shared memory, one flux per face;
    // called by every thread of the row (they synchronise)
    auto xfaces = [&]() {
      R fl[3][NC], fr[3][NC];
      if (need) {
#pragma unroll
        for (int g = 0; g < 3; ++g) {
          flux_dir<EQ, R>(P, 0, xl[g], fl[g]);
          flux_dir<EQ, R>(P, 0, xr[g], fr[g]);
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            trL[((c * 3 + g) * 2 + 0) * BX + tx] = xl[g][c];
            trL[((c * 3 + g) * 2 + 1) * BX + tx] = fl[g][c];
          }
        }
      }
      row_sync();
      if (need && tx <= wout && i < nx) {
#pragma unroll
        for (int g = 0; g < 3; ++g)
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const R uR = trL[((c * 3 + g) * 2 + 0) * BX + tx + 1];
            const R fR = trL[((c * 3 + g) * 2 + 1) * BX + tx + 1];
            // twice the LF flux (Eq. 2.4 without its factor 1/2, folded into the weights)
            fhx(c * 3 + g, tx + 1) = fr[g][c] + fR - a1 * (uR - xr[g][c]);
          }
      }
      row_sync();
      if (outc) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const R L0 = fhx(c * 3 + 0, tx), L1 = fhx(c * 3 + 1, tx), L2 = fhx(c * 3 + 2, tx);
          const R R0 = fhx(c * 3 + 0, tx + 1), R1 = fhx(c * 3 + 1, tx + 1),
                  R2 = fhx(c * 3 + 2, tx + 1);
          const R sdiff = R(0.5 * GW0) * ((R0 - L0) + (R2 - L2)) + R(0.5 * GW1) * (R1 - L1);
          const R ssum = R(0.5 * GW0) * ((L0 + R0) + (L2 + R2)) + R(0.5 * GW1) * (L1 + R1);
          const R smom = R(0.5 * GW0) * s15 * ((R2 - L2) - (R0 - L0));
          rx[c][0] = -sdiff * idx;
          rx[c][1] = (volf[c] - R(0.5) * ssum) * idx;
          rx[c][2] = -smom * idx;
        }
      }
    };

    if constexpr (CHAR && EQ == EQ_EULER) {
      // two characteristic passes (x: edge points of the x faces, f-volume, v-hat; y: edge
      // points of the y faces, g-volume, w-hat); the x faces are formed between them so the
      // x-pass results are dead during the y pass.  The eigenvector state is shared.
      Eig2<R> E;
      if (need) {
        R U5[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) U5[c] = Wv(c * NM, 4);
        E.init_state(P, U5);
      }
#pragma unroll
      for (int pass = 0; pass < 2; ++pass) {
        if (pass == 0 && !xrow) continue;
        if (need) {
          E.set_dir(pass);
          R ch[16][4];  // characteristic values: 6 edge points, 9 interior, modification
          // the combined polynomial of field f -> its points and modification
          auto evaluate = [&](int f, const R (&C)[15]) {
            R ea[3], eb[3], in[9];
            if (pass == 0) {
              eval_xpass(C, ea, eb, in);
              ch[15][f] = vhat2d(C);
            } else {
              eval_ypass(C, ea, eb, in);
              ch[15][f] = what2d(C);
            }
#pragma unroll
            for (int g = 0; g < 3; ++g) {
              ch[g][f] = ea[g];
              ch[3 + g][f] = eb[g];
            }
#pragma unroll
            for (int p = 0; p < 9; ++p) ch[6 + p][f] = in[p];
          };
          {
            // the stencil in characteristic variables, all four fields at once: 9 averages
            // and the x / y first moments of cells 2, 4, 6, 8
            R Wu[9][4], Wv_[4][4], Ww[4][4];
#pragma unroll
            for (int k = 0; k < 9; ++k) {
              R Uk[4];
#pragma unroll
              for (int c = 0; c < 4; ++c) Uk[c] = Wv(c * NM, k);
              E.project_all(Uk, Wu[k]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int k = 2 * e + 1;
              R Vk[4], Zk[4];
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                Vk[c] = Wv(c * NM + 1, k);
                Zk[c] = Wv(c * NM + 2, k);
              }
              E.project_all(Vk, Wv_[e]);
              E.project_all(Zk, Ww[e]);
            }
            // one field's stencil in characteristic variables
            auto field = [&](int f, R (&u)[9], R (&v)[4], R (&w)[4]) {
#pragma unroll
              for (int k = 0; k < 9; ++k) u[k] = Wu[k][f];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                v[e] = Wv_[e][f];
                w[e] = Ww[e][f];
              }
            };
#pragma unroll
            for (int f = 0; f < 4; ++f) {
              R u[9], v[4], w[4], C[15];
              field(f, u, v, w);
              coeffs2d<R>(u, v, w, C);
              fast_weights &= weigh_field<R>(o, u, P, C);
              evaluate(f, C);
            }
          }
          R cons[16][4];
#pragma unroll
          for (int p = 0; p < 16; ++p) E.unproject(ch[p], cons[p]);
          R inn[9][4];
#pragma unroll
          for (int p = 0; p < 9; ++p)
#pragma unroll
            for (int c = 0; c < 4; ++c) inn[p][c] = cons[6 + p][c];
          if (pass == 0) {
#pragma unroll
            for (int g = 0; g < 3; ++g)
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                xl[g][c] = cons[g][c];
                xr[g][c] = cons[3 + g][c];
              }
#pragma unroll
            for (int c = 0; c < 4; ++c) vh[c] = cons[15][c];
            volume_sum<EQ, NC, R>(P, 0, inn, volf);
          } else {
#pragma unroll
            for (int g = 0; g < 3; ++g)
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                yb[g][c] = cons[g][c];
                yt[g][c] = cons[3 + g][c];
              }
#pragma unroll
            for (int c = 0; c < 4; ++c) wh[c] = cons[15][c];
            volume_sum<EQ, NC, R>(P, 1, inn, volg);
          }
        }
        if (pass == 0) xfaces();
      }
    } else {
      if (need) {
        // component-wise: one reconstruction per conserved component gives all points
        R inn[9][NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          R u[9], v[4], w[4];
#pragma unroll
          for (int k = 0; k < 9; ++k) u[k] = Wv(c * NM, k);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            v[e] = Wv(c * NM + 1, 2 * e + 1);
            w[e] = Wv(c * NM + 2, 2 * e + 1);
          }
          R C[15];
          coeffs2d<R>(u, v, w, C);
          fast_weights &= weigh_field<R>(o, u, P, C);
          R ea[3], eb[3], in[9];
          eval_xpass(C, ea, eb, in);
#pragma unroll
          for (int g = 0; g < 3; ++g) {
            xl[g][c] = ea[g];
            xr[g][c] = eb[g];
          }
#pragma unroll
          for (int p = 0; p < 9; ++p) inn[p][c] = in[p];
          R qb[3], qt[3], in2[9];
          eval_ypass(C, qb, qt, in2);
#pragma unroll
          for (int g = 0; g < 3; ++g) {
            yb[g][c] = qb[g];
            yt[g][c] = qt[g];
          }
          vh[c] = vhat2d(C);
          wh[c] = what2d(C);
        }
        volume_sum<EQ, NC, R>(P, 0, inn, volf);
        volume_sum<EQ, NC, R>(P, 1, inn, volg);
      }
      if (xrow) xfaces();
    }

    // y face j-1/2 between (i, j-1) and (i, j): Eq. 2.16
    R ybg[3][NC];
    if (need) {
#pragma unroll
      for (int g = 0; g < 3; ++g) flux_dir<EQ, R>(P, 1, yb[g], ybg[g]);
#pragma unroll
      for (int g = 0; g < 3; ++g) {
        R tg[NC];
        flux_dir<EQ, R>(P, 1, yt[g], tg);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          cmine[(g * NC + c) * BX] = yt[g][c];
          cmine[((3 + g) * NC + c) * BX] = tg[c];
        }
      }
    }
    __syncthreads();  // the step's traces are in place and nothing reads the window any more
    R rhs[NC][3];
#pragma unroll
    for (int c = 0; c < NC; ++c) rhs[c][0] = rhs[c][1] = rhs[c][2] = R(0);
    if (need && j > j0 - 1) {
      R gh[3][NC];
#pragma unroll
      for (int g = 0; g < 3; ++g)
#pragma unroll
        for (int c = 0; c < NC; ++c)
          gh[g][c] = cbelow[((3 + g) * NC + c) * BX] + ybg[g][c] -
                     a2 * (yb[g][c] - cbelow[(g * NC + c) * BX]);  // 2 x LF flux
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const R sw = R(0.5 * GW0) * (gh[0][c] + gh[2][c]) + R(0.5 * GW1) * gh[1][c];
        const R sm = R(0.5 * GW0) * s15 * (gh[2][c] - gh[0][c]);
        fm[(2 * c) * T + t] = sw;
        fm[(2 * c + 1) * T + t] = sm;
        // bottom face of (i, j): F1 += sum/dy, F2 += sum xi/dy, F3 -= sum/(2 dy)
        rhs[c][0] = __fmul_rn(sw, idy);
        rhs[c][1] = __fmul_rn(sm, idy);
        rhs[c][2] = __fmul_rn(-R(0.5) * sw, idy);
      }
    }
    // the x-face and volume terms of (i, j)
    if (xrow && outc) {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        rhs[c][0] = __fadd_rn(rhs[c][0], rx[c][0]);
        rhs[c][1] = __fadd_rn(rhs[c][1], rx[c][1]);
        rhs[c][2] = __fadd_rn(rhs[c][2], __fmaf_rn(volg[c], idy, rx[c][2]));
      }
    }
    // the window's next BY rows, into the slots of the rows no longer needed
    if (j + BY + 1 <= j1 + 1) load_row(j + BY + 1);
    __syncthreads();

    // the row whose top face is now known: this thread's row j, or in the tile's last row the
    // one it processed a step ago (row j takes its place)
    const bool last = ty == BY - 1;
    const int jc = last ? j - BY : j;
    const R* face = fm + (last ? tx : t + BX);
    if (last) {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const R x = rhs[c][m];
          rhs[c][m] = pend[c][m];
          pend[c][m] = x;
        }
        const R x = vh[c], y = wh[c];
        vh[c] = pvh[c];
        wh[c] = pwh[c];
        pvh[c] = x;
        pwh[c] = y;
      }
    }
    if (outc && jc >= j0 && jc < j1) {
      // its top face: F1 -= sum/dy, F2 -= sum xi/dy, F3 -= sum/(2 dy); then the update: Eq. 2.13
      const size_t q = (size_t)jc * nx + i;
      double outv[NC * NM];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const R sw = face[(2 * c) * T], sm = face[(2 * c + 1) * T];
        rhs[c][0] = __fsub_rn(rhs[c][0], __fmul_rn(sw, idy));
        rhs[c][1] = __fsub_rn(rhs[c][1], __fmul_rn(sm, idy));
        rhs[c][2] = __fsub_rn(rhs[c][2], __fmul_rn(R(0.5) * sw, idy));
        const double own[3] = {S.Uin[(size_t)(c * NM) * plane + q], to_f64(vh[c]), to_f64(wh[c])};
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const size_t qa = (size_t)(c * NM + m) * plane + q;
          double base;
          if (S.k == 1) {
            base = own[m];
            if (m > 0) S.Vh[(size_t)(c * 2 + m - 1) * plane + q] = own[m];
          } else {
            base = (m == 0) ? S.Un[qa] : S.Vh[(size_t)(c * 2 + m - 1) * plane + q];
          }
          const double adv = fma(dt, to_f64(rhs[c][m]), own[m]);
          double o;
          if (S.k == 1) o = adv;
          else if (S.k == 2) o = fma(0.75, base, 0.25 * adv);
          else o = fma(1.0 / 3.0, base, 2.0 / 3.0 * adv);
          S.Uout[qa] = o;
          outv[c * NM + m] = o;
        }
      }
      double ua[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) ua[c] = outv[c * NM];
      bool bad = false;
#pragma unroll
      for (int q2 = 0; q2 < NC * NM; ++q2) bad |= !finite_bits(outv[q2]);
      if constexpr (EQ == EQ_EULER) {
        double s0, s1;
        bad |= !euler_speeds<2>(P, ua, s0, s1);
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
  const int any_direct = __syncthreads_or(fast_weights ? 0 : 1);
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

// One work item of the class.
template <int EQ, bool CHAR, typename R, int BW>
__device__ __forceinline__ void stage2d_item(const KProblem& P, const KStage& S, int band,
                                             int j0, int j1, int wout, double* smem,
                                             double (*red)[kThreads2D<R, BW> / 32]) {
  if constexpr (sizeof(R) == sizeof(double))
    stage2d_tile64_item<EQ, CHAR, BW, kTileRows<R, BW>>(P, S, band, j0, j1, wout, smem, red);
  else
    stage2d_mixed_item<EQ, CHAR, R, BW, kTileRows<R, BW>>(P, S, band, j0, j1, wout, smem, red);
}

}  // namespace hw
