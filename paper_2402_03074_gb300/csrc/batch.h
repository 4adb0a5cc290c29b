// batch.h -- device work lists of the batched persistent stage launches (batch.cu).
#pragma once
#include <cuda_runtime.h>

#include "geometry.h"
#include "launch.h"

namespace hw {

// Block width of the batched stage kernels: the 1D classes 128 threads, the 2D classes tiles of 64
// columns by 4 rows in FP64 and 3 in FP32-bulk (against one row at a time in 128-thread blocks, which
// hold only four warps per SM in FP64, and FP64 tiles of 3 rows: a batch of eight FP64 solves of
// 200 x 184 to 284 x 261 cells, one step, 9.00, 7.58 and now 6.80 ms; a served mix of six grids of
// 128^2 to 352^2 cells, a third of them FP32-bulk, 114, 95.5 and now 85.4 ms).
constexpr int kBatchBW = 128;
constexpr int kBatchBX = 64;
constexpr int kBatchClasses = 16;  // {2D, 1D} x {advection, Burgers, Euler comp.-wise,
                                   // Euler char.} x {FP64, mixed}

// One solve in a batch (device-resident array, rewritten on admission / retirement).
struct BatchSolve {
  KProblem P;
  double* U[3];        // U^n, U^(1), U^(2)
  double* Vh;
  DevScal* sc;
  int mixed;           // 1: FP32 bulk / FP64 weights
  int bands, wout, rows, chunks;  // 1D: bands = blocks of kBatchBW - 2 cells, chunks = 1
  int item_base;       // first work item of the solve
};

// Control block of one class's launches.
struct BatchCtl {
  int n_solves;
  int n_items;
  unsigned int next[3];  // work counters of the three stage launches of a step
};

// Per-solve step scalars of every solve in the batch (all classes).
constexpr int kBatchCap = 1024;
struct BatchDt {
  int n;       // solves whose step starts here (the batched ones, first in the list)
  int n_all;   // all live solves (the gather of their scalars)
  DevScal* sc[kBatchCap];
  double inv_dx[kBatchCap], inv_dy[kBatchCap];
  int dim[kBatchCap];
};

int batch_class(int equation, int characteristic, int mixed, int dim = 2);
// bands of at most kBatchBX - 2 columns and row chunks of `rows` rows
void batch_geometry(int nx, int ny, int rows, int* bands, int* wout, int* chunks);
// SMs of the current device
int batch_sms();
// rows per item for the 2D solves of one class (n grids) on `slots` resident blocks of `sms` SMs;
// bands and warps: the caller's scratch of n entries each (nothing is allocated)
int batch_item_rows(const int* nx, const int* ny, int n, bool mixed, int slots, int sms,
                    int* bands, int* warps);
void batch_geometry1d(int nx, int* blocks);
int batch_slots(int cls);  // resident blocks of the class's persistent launch
cudaError_t launch_batch_dt(BatchDt* d, BatchCtl* ctl, int nctl, int cap, cudaStream_t st);
cudaError_t launch_batch_stage(int cls, const BatchSolve* bs, BatchCtl* ctl, int k,
                               cudaStream_t st);

}  // namespace hw
