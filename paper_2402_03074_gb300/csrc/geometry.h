// geometry.h -- launch geometry of the fused 2D stage: how a grid is cut into work items of
// (band of columns) x (chunk of rows).  Host code in plain C++ (no CUDA types), shared by the
// single-solve launch (stage2d.cu), the batched launches (batch.cu, static_batch.cu) and the
// serving loop (server.cu).
//
// A block of bw columns (by one to eight rows) of threads covers a band of at most bw - 2 output
// columns plus one ring column on each side, and sweeps a chunk of rows (one ring row above and
// below), several rows at a time.  The time of a launch is set by its waves of items over the
// resident block slots and by the steps of an item (tile_time64).
#pragma once

namespace hw {

// lanes (threads in whole warps) that `bands` equal bands over nx columns occupy, each band
// with its two ring columns
inline int band_lanes(int nx, int bands) {
  const int w = (nx + bands - 1) / bands;
  return bands * 32 * ((w + 2 + 31) / 32);
}

// Default band count for blocks of bw columns: the widest bands (at most bw - 2 output columns).
// With lane_aware, which no launch asks for since the tiles have several rows (the host tests do),
// bands of at most bw - 34 columns when they leave fewer idle lanes.
inline int default_bands(int nx, int bw, bool lane_aware) {
  int b = (nx + (bw - 2) - 1) / (bw - 2);
  if (lane_aware && bw > 34) {
    const int b3 = (nx + (bw - 34) - 1) / (bw - 34);
    if (b3 <= nx && 100LL * band_lanes(nx, b3) < 99LL * band_lanes(nx, b)) b = b3;
  }
  return b;
}

// Equal bands: the output columns per band for `bands` requested bands, and the band count
// that leaves no band empty.
inline void split_bands(int nx, int bands_req, int* bands, int* wout) {
  *wout = (nx + bands_req - 1) / bands_req;
  *bands = (nx + *wout - 1) / *wout;
}

// Single-solve launch: bands as above (or fixed, but never wider than bw - 2 columns), swept
// by one wave of blocks in one of two layouts:
//  * chunks: row chunks sized so that bands x chunks fills the `slots` resident blocks once
//    (or fixed rows); a block sweeps one chunk of one band;
//  * segments (seg > 0): the bands' rows taken one after another (band-row q = band ny + row)
//    and cut into `blocks` equal segments of seg band-rows, one per block; a segment that
//    crosses the end of a band is swept as two (or more) pieces.  When the band count does not
//    divide the slots, chunks leave slots empty (2048^2 in 94-column bands: 22 x 6 = 132 of
//    152), while segments fill them (152 blocks of 297 band-rows instead of 342 rows).
// Fixed rows > 0 give chunks of that height, fixed rows < -1 segments of -rows band-rows (the rule
// for a grid without a tuned shape, default_tile64, fixes one or the other); the default (0), of a
// stored width, takes segments where they cost at least 2 % less than chunks, a piece costing its
// rows plus about 1.5 rows (its two ring rows of the y pass and the window prologue).
struct Geom2D {
  int bands, wout, chunks, rows;
  int seg;     // > 0: segment layout, band-rows per block
  int blocks;  // blocks of the launch (bands x chunks, or the segments)
};
inline Geom2D geom2d(int nx, int ny, int bw, int slots, int rows_fixed, int bands_fixed,
                     bool lane_aware) {
  Geom2D g;
  const int bwide = (nx + (bw - 2) - 1) / (bw - 2);
  int b = bands_fixed > 0 ? (bands_fixed < nx ? bands_fixed : nx) : default_bands(nx, bw, lane_aware);
  if (bands_fixed > 0 && b < bwide) b = bwide;  // a band is at most bw - 2 columns wide
  split_bands(nx, b, &g.bands, &g.wout);
  g.seg = 0;
  if (rows_fixed > 0) {
    g.rows = rows_fixed < ny ? rows_fixed : ny;
  } else {
    int ch = slots / g.bands;
    if (ch < 1) ch = 1;
    if (ch > ny) ch = ny;
    g.rows = (ny + ch - 1) / ch;
  }
  g.chunks = (ny + g.rows - 1) / g.rows;
  g.blocks = g.bands * g.chunks;
  const long long total = (long long)g.bands * ny;
  long long seg = 0;
  if (rows_fixed < -1) {
    seg = -(long long)rows_fixed;
  } else if (rows_fixed == 0 && slots > 0 && g.bands <= slots) {
    const long long s = (total + slots - 1) / slots;
    const long long pieces = 1 + (s - 1 + ny - 1) / ny;   // most pieces a segment can have
    if ((double)s + 1.5 * (double)pieces < 0.98 * ((double)g.rows + 1.5)) seg = s;
  }
  if (seg > 0) {
    if (seg > total) seg = total;
    g.seg = (int)seg;
    g.blocks = (int)((total + seg - 1) / seg);
  }
  return g;
}

// ---- Tiles: FP64 bx columns x tile_rows64(bx) rows of threads per block (stage2d_tile64.cuh):
// eight warps, two per scheduler, of 255 registers a thread (96 columns: six, the shared memory's
// limit).  Against seven and six warps (32 x 7, 64 x 3): 240^2 Euler, 12 steps, 11.55 -> 10.05 ms,
// 240^2 Burgers, 48 steps, 7.98 -> 7.00 ms, eight-solve batch 7.41 -> 6.78 ms, 768^2 component-wise
// 5.30 -> 5.19 ms; 320^2 (whose chunks of 27 rows fill 7-row steps better) 1.62 -> 1.66 ms.
constexpr int tile_rows64(int bx) { return bx == 32 ? 8 : bx == 64 ? 4 : bx == 96 ? 2 : 1; }
// The same for the FP32-bulk kernels: six warps per block, two blocks per SM (128 columns: four
// warps, three blocks).
constexpr int tile_rows32(int bx) { return bx == 32 ? 6 : bx == 64 ? 3 : bx == 96 ? 2 : 1; }

// Time of `blocks` blocks sharing an SM, each sweeping a piece of `rows` output rows (and the two
// ring rows, 0.46 of a row's work each: the y pass without its volume sums) by rows at a time, in
// units of one row of one warp at the SM's full rate: a step takes the work of its rows
// (`warps` warps each), but at least `step`, because a warp alone runs far below that rate (one FP64
// instruction in 64 clocks against the SM's 16).  kStep64: 4.6 (40^2 Euler: 108 us per stage, a
// warp-row 21 us of an SM at 2048^2); kStep32, the FP32-bulk kernels: 7 (65 us and 9.2 us).
constexpr double kStep64 = 4.6, kStep32 = 7.0;
inline double tile_time64(int warps, int by, int rows, int blocks, double step) {
  const int full = (rows + 2) / by, rest = (rows + 2) % by;
  const double w = (double)warps * blocks;
  // a last step of one row holds the upper ring row alone: half a step
  const double last = rest == 1 ? 0.5 * step : rest ? (w * rest > step ? w * rest : step) : 0.0;
  const double t = full * (w * by > step ? w * by : step) + last - 1.08 * w;
  const double least = step * (full + (rest > 1 ? 1.0 : 0.5 * rest));
  return t > least ? t : least;
}

// The default tile of a grid: over the widths bx[0..n-1] (with slots[] resident blocks per GPU
// each, on `sms` SMs) and the chunk heights (or one segment per resident block), the launch of
// least time.  240^2 FP64: 32 x 8, 8 bands x 19 chunks of 13 rows (0.84 ms per three stages); 2048^2
// FP64: 96 x 2, 22 bands in 152 segments of 297 band-rows (54.5 ms; 54.2 in 64 x 4 and 54.5 in 32 x 8,
// whose eight warps make up for ring columns of 3 and 7 % instead of 2 %); 320^2: 32 x 8 in
// chunks of 25 rows, the last step with three rows (1.66 ms; 1.68 in 64 x 4).
struct Tile64 {
  int bx;
  int rows;  // output rows per chunk; < -1: segments of -rows band-rows
};
inline Tile64 default_tile64(int nx, int ny, int sms, const int* bx, const int* slots, int n,
                             bool mixed = false) {
  Tile64 best{96, 0};
  double best_time = 1e300;
  const double step = mixed ? kStep32 : kStep64;
  for (int q = 0; q < n; ++q) {
    const int by = mixed ? tile_rows32(bx[q]) : tile_rows64(bx[q]);
    int bands, wout;
    split_bands(nx, default_bands(nx, bx[q], false), &bands, &wout);
    const int warps = (wout + 2 + 31) / 32;
    const int per_sm = slots[q] > sms ? slots[q] / sms : 1;
    // every wave and every further piece of a segment (`extra`) costs a window prologue, about 2.5
    // units, the piece also its ring rows (1024^2 FP64: one wave of segments in two pieces 14.70 ms,
    // three waves of 25-row chunks 14.98 ms)
    constexpr double prologue = 2.5;
    auto consider = [&](long long blocks, int rows, int extra, int encoded) {
      const long long waves = blocks / slots[q], rest = blocks % slots[q];
      double time = 0.0;
      if (waves > 0) time += (double)waves * tile_time64(warps, by, rows, per_sm, step);
      if (rest > 0)
        time += tile_time64(warps, by, rows, (int)((rest + sms - 1) / sms), step);
      time += (double)(waves + (rest > 0 ? 1 : 0)) * prologue +
              extra * (prologue + 0.92 * warps * per_sm);
      if (time < 0.995 * best_time) {
        best_time = time;
        best = Tile64{bx[q], encoded};
      }
    };
    for (int r = 1; r <= 16 && r <= ny; ++r) consider((long long)bands * ((ny + r - 1) / r), r, 0, r);
    for (int m = 1; m <= 6; ++m) {
      int c = m * sms / bands;
      c = c < 1 ? 1 : (c > ny ? ny : c);
      const int r = (ny + c - 1) / c;
      consider((long long)bands * ((ny + r - 1) / r), r, 0, r);
    }
    const long long total = (long long)bands * ny;
    const long long seg = (total + slots[q] - 1) / slots[q];
    if (bands <= slots[q] && seg > 1)
      consider((total + seg - 1) / seg, (int)seg, (int)((seg - 1 + ny - 1) / ny), -(int)seg);
  }
  return best;
}

// Whether a shape of the tuning table (launch.h, TileShape) leaves the tile to the rule above: no
// width and nothing fixed, or the autotuner's entry for it, {0, 0, kDefaultWidth2D}.  Any other
// shape with a width is of that width, with the band and row geometry of geom2d where these are
// not fixed (the same bits, another kernel: 240^2 Euler FP64 in 96 columns, {-1, -1, 96}, takes
// 1.4 times the rule's 32).
constexpr int kDefaultWidth2D = 96;
inline bool takes_default_tile(int rows, int bands, int width) {
  if (width == 0) return (rows == 0 || rows == -1) && bands <= 0;
  return width == kDefaultWidth2D && rows == 0 && bands == 0;
}

// Rows per item of a batched 2D class in tiles of bx columns (bands[s] bands of warps[s] warps
// per row, ny[s] rows), whose persistent launch has `slots` resident blocks: the rows of least
// waves x item time (per_sm blocks sharing an SM), the smallest (the most items) among equals.
// An item's time does not fall with its rows, so of the heights with as many waves the smallest is
// the cheapest: only the heights at which the waves drop are looked at, each found by doubling
// steps and halving, up to the one from which the fewest waves there can be cost more than the
// best so far.  Nothing is allocated.  On one x86 core, 16 grids of about 2000 rows: 27 us (every
// height in turn, every solve's time at each: 124 us); 12 of about 200: 1.5 us (8.9 us).
inline int batch_rows64(const int* bands, const int* warps, const int* ny, int n, int bx,
                        int slots, int per_sm, bool mixed = false) {
  if (n <= 0 || slots <= 0) return 32;
  constexpr int kMaxWarps = 8;  // a band has at most bx / 32 warps, six in the widest blocks
  int tallest[kMaxWarps + 1] = {};  // of the grids with bands of that many warps
  int nymax = 1;
  long long fewest = 0;  // items of one chunk per band
  for (int s = 0; s < n; ++s) {
    const int w = warps[s] < kMaxWarps ? warps[s] : kMaxWarps;
    tallest[w] = ny[s] > tallest[w] ? ny[s] : tallest[w];
    nymax = ny[s] > nymax ? ny[s] : nymax;
    fewest += bands[s];
  }
  fewest = (fewest + slots - 1) / slots;
  auto waves = [&](long long r) {
    long long items = 0;
    for (int s = 0; s < n; ++s) items += (long long)bands[s] * ((ny[s] + r - 1) / r);
    return (items + slots - 1) / slots;
  };
  const int by = mixed ? tile_rows32(bx) : tile_rows64(bx);
  const double step = mixed ? kStep32 : kStep64;
  int best = 1;
  double best_cost = 1e300;
  long long r = 1, w = waves(1);
  for (;;) {
    double time = 0.0;
    for (int q = 0; q <= kMaxWarps; ++q) {
      if (tallest[q] == 0) continue;
      const double t = tile_time64(q, by, (int)(r < tallest[q] ? r : tallest[q]), per_sm, step);
      time = t > time ? t : time;
    }
    if ((double)w * time < best_cost) {
      best_cost = (double)w * time;
      best = (int)r;
    }
    if (r >= nymax || (double)fewest * time >= best_cost) return best;
    long long lo = r, hi = r + 1, w_hi = waves(hi);  // waves(lo) == w
    for (long long d = 2; w_hi == w && hi < nymax; d *= 2) {
      lo = hi;
      hi = hi + d < nymax ? hi + d : nymax;
      w_hi = waves(hi);
    }
    if (w_hi == w) return best;  // no height has fewer waves
    while (hi - lo > 1) {
      const long long mid = lo + (hi - lo) / 2, w_mid = waves(mid);
      if (w_mid == w) {
        lo = mid;
      } else {
        hi = mid;
        w_hi = w_mid;
      }
    }
    r = hi;
    w = w_hi;
  }
}

// The rule for blocks of one row of threads, which the batched launches no longer are (batch_rows64
// is theirs; the host tests keep this one): rows per work item for the 2D solves of one batched class
// (bands[s] bands and ny[s] rows each) whose persistent launch has `slots` resident blocks.  The
// launch runs ceil(items / slots) waves, a partial last wave costing a whole item time, and an item
// costs its rows plus about 1.5 rows (its two ring rows of the y pass and the three-row window
// prologue); the rows minimising waves x (rows + 1.5) give the shortest launch, the smallest
// such rows (the most items) winning ties.
inline int batch_rows(const int* bands, const int* ny, int n, int slots) {
  if (n <= 0 || slots <= 0) return 32;
  int nymax = 1;
  for (int s = 0; s < n; ++s) nymax = ny[s] > nymax ? ny[s] : nymax;
  int best = 4;
  double best_cost = 1e300;
  for (int r = 4; r <= (nymax > 4 ? nymax : 4); ++r) {
    long long items = 0;
    for (int s = 0; s < n; ++s) items += (long long)bands[s] * ((ny[s] + r - 1) / r);
    const long long waves = (items + slots - 1) / slots;
    const double cost = (double)waves * (r + 1.5);
    if (cost < best_cost) {
      best_cost = cost;
      best = r;
    }
  }
  return best;
}

}  // namespace hw
