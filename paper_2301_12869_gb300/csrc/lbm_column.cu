// Planning and launching the on-chip kernels of lbm_column.cuh.
#include "lbm_column.h"

#include "lbm.h"

#include <cuda_runtime.h>

#include <algorithm>

namespace lbm {
namespace {

// per precision: nodes of an item, most items a thread, most threads a CTA, bytes of shared memory
// an item slot takes, and the items a CTA needs before splitting a column further pays
struct Shape {
  int Q, most_items, most_threads, slot_bytes, min_items;
};
Shape shape_of(int precision) {
  // FP32: a step of up to 256 items (1024 nodes) is bound by its dependency chain and its two
  // barriers, which cost a cluster more. FP64: 128 nodes are one warp on each of the SM's four FP64 pipes - fewer do
  // not shorten a step. Double-float: 128 nodes are half a microsecond of arithmetic.
  if (precision == LBM_FP32) return {4, 4, 256, 8 * 16, 256};
  return {1, 4, 256, 6 * 8, 128};
}
constexpr size_t kMostShared = 208 * 1024;  // beside up to 18 KB of static arrays

const void* kernel_of(int precision, const ColumnPlan& p, bool acc) {
  const int per_thread = p.per_thread;
  if (precision == LBM_FP32) return column_kernel_f32(per_thread, acc, p.row_log2 == 0);
  if (precision == LBM_FP64) return column_kernel_f64(per_thread, acc);
  return column_kernel_dd(per_thread, acc);
}

void fill_config(const ColumnPlan& p, int clusters, cudaStream_t stream, cudaLaunchConfig_t* cfg,
                 cudaLaunchAttribute* attr) {
  cfg->gridDim = dim3(clusters * p.cluster);
  cfg->blockDim = dim3(p.threads);
  cfg->dynamicSmemBytes = p.smem;
  cfg->stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.cluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = p.cluster > 1 ? 1 : 0;
}

}  // namespace

ColumnPlan plan_columns(int precision, int nx, int ny, int min_ny, int cluster_goal, int min_items) {
  ColumnPlan p;
  Shape s = shape_of(precision);
  if (min_items > 0) s.min_items = min_items;
  const int m = nx / s.Q;  // items of a row
  if (nx % s.Q || m < 1 || m > 32) return p;
  while ((1 << p.row_log2) < m) ++p.row_log2;
  const int P = 1 << p.row_log2;
  auto rows = [&](int cs) { return (ny + cs - 1) / cs; };
  auto fits = [&](int cs) {
    return rows(cs) * P <= s.most_items * s.most_threads &&
           size_t(rows(cs) + 2) * P * s.slot_bytes <= kMostShared;
  };
  int cs = 1;
  while (cs < 8 && !fits(cs)) cs *= 2;
  if (!fits(cs)) return p;
  while (2 * cs <= std::min(cluster_goal, 8) && rows(2 * cs) * P >= s.min_items) cs *= 2;
  if (cs > min_ny) return p;
  p.cluster = cs;
  p.rows_cap = rows(cs);
  const int items = p.rows_cap * P;
  p.per_thread = 1;
  while ((items + p.per_thread - 1) / p.per_thread > s.most_threads) p.per_thread *= 2;
  // a multiple of four warps: a share of the work for each of the SM's four schedulers
  p.threads = ((items + p.per_thread - 1) / p.per_thread + 31) / 32 * 32;
  if (p.threads > 128) p.threads = (p.threads + 127) / 128 * 128;
  p.smem = size_t(p.rows_cap + 2) * P * s.slot_bytes;
  p.ok = kernel_of(precision, p, false) != nullptr;
  return p;
}

int column_clusters(int precision, const ColumnPlan& p, bool acc) {
  const void* fn = kernel_of(precision, p, acc);
  if (!fn || cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kMostShared)) != cudaSuccess)
    return 0;
  if (p.cluster > 1) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    fill_config(p, 1, nullptr, &cfg, attr);
    int n = 0;
    return cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess ? n : 0;
  }
  int dev = 0, nsm = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, p.threads, p.smem) != cudaSuccess)
    return 0;
  return nsm * per_sm;
}

cudaError_t launch_columns(int precision, const ColumnPlan& p, bool acc, int clusters, const ColumnArgs& args,
                           cudaStream_t stream) {
  const void* fn = kernel_of(precision, p, acc);
  if (!fn) return cudaErrorInvalidValue;
  ColumnArgs a = args;
  a.row_log2 = p.row_log2;
  a.cluster = p.cluster;
  a.rows_cap = p.rows_cap;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  fill_config(p, clusters, stream, &cfg, attr);
  void* kargs[] = {&a};
  return cudaLaunchKernelExC(&cfg, fn, kargs);
}

}  // namespace lbm
