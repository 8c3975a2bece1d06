// The FP32 kernels of lbm_column.cuh.
#include "lbm_column.cuh"

namespace lbm {
namespace {
template <bool ALONE>
const void* kernel(int per_thread, bool acc) {
  switch (per_thread) {
    case 1: return acc ? (const void*)&column_kernel<float, 1, true, ALONE> : (const void*)&column_kernel<float, 1, false, ALONE>;
    case 2: return acc ? (const void*)&column_kernel<float, 2, true, ALONE> : (const void*)&column_kernel<float, 2, false, ALONE>;
    case 4: return acc ? (const void*)&column_kernel<float, 4, true, ALONE> : (const void*)&column_kernel<float, 4, false, ALONE>;
    default: return nullptr;
  }
}
}  // namespace

const void* column_kernel_f32(int per_thread, bool acc, bool alone) {
  return alone ? kernel<true>(per_thread, acc) : kernel<false>(per_thread, acc);
}

}  // namespace lbm
