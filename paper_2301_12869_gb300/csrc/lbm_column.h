// Small lattices iterated on chip (lbm_column.cuh): what the batched columns (lbm_batch.cu) and
// a single handle's lattice (lbm_api.cu) share.
#pragma once

#include "lbm_internal.h"

#include <cuda_runtime.h>

namespace lbm {

struct BatchCol {
  int ny, form;
  long long node_off;  // nodes of the columns before this one
  double RT, gx, gy, rho_ref;
};

constexpr int kMpeK = 4;  // extrapolation order: kMpeK + 2 snapshots per cycle

struct RunParams {
  double tol;
  long long max_steps;
  int check_every;
  int stall_checks;  // > 0: a column also stops after this many checks without a 1 % gain
  int mpe_checks;    // > 0: a state snapshot every mpe_checks residual checks, extrapolation per cycle
  void* snap;        // kMpeK + 2 slots of 9 * total_nodes reals (NULL: no extrapolation)
  long long slot;    // elements per slot (9 * total_nodes)
};

// stalls count only below this residual: about 30 ulp of an FP32 / FP64 density of 0.3
template <typename T>
constexpr double kStallBelow = sizeof(T) == 4 ? 1e-6 : 1e-13;

struct ColumnArgs {
  const BatchCol* cols;  // NULL: the one lattice `one`
  BatchCol one;
  const int* order;      // columns of this launch, tallest first (NULL: one lattice)
  int ncols, nx;
  void* f;               // populations, concatenated [col][9][ny][nx]: read at the start, written at the end
  void* scratch;         // as large as f: the densities a residual compares with
  double a, b, G, sig_e;
  const RunParams* run;  // NULL: run_one
  RunParams run_one;
  int* counter;          // work-stealing counter, zero at launch (NULL: one lattice)
  long long* steps;      // per column, may be NULL with one lattice, as the next three
  double* resid;
  int* col_status;
  long long* col_ns;
  int* status;           // one lattice: the handle's status word
  int zh;
  int row_log2;          // log2 of the lanes a row takes
  int cluster;           // CTAs that share a column's rows
  int rows_cap;          // rows a CTA's shared memory holds
};

struct ColumnPlan {
  bool ok = false;       // the lattice fits
  int row_log2 = 0, cluster = 1, threads = 0, per_thread = 0, rows_cap = 0;
  size_t smem = 0;
};

// the launch of columns nx wide and up to ny rows tall (at least min_ny); `cluster_goal`: as many
// CTAs a column as are useful and allowed (a power of two); min_items: items (threads) a CTA keeps
// when a column is split, 0: what pays when other columns wait. precision: LBM_FP32 / FP64 / DOUBLE_FLOAT
ColumnPlan plan_columns(int precision, int nx, int ny, int min_ny, int cluster_goal, int min_items = 0);
// resident clusters of a plan on the current device (0: it cannot run)
int column_clusters(int precision, const ColumnPlan& p, bool acc);
cudaError_t launch_columns(int precision, const ColumnPlan& p, bool acc, int clusters, const ColumnArgs& args,
                           cudaStream_t stream);

// kernels of one precision (lbm_column_f32.cu, _f64.cu, _dd.cu): NULL where there is none
const void* column_kernel_f32(int per_thread, bool acc, bool alone);
const void* column_kernel_f64(int per_thread, bool acc);
const void* column_kernel_dd(int per_thread, bool acc);

}  // namespace lbm
