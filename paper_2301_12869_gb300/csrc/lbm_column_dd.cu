// The double-float kernels of lbm_column.cuh.
#include "lbm_column.cuh"

namespace lbm {
const void* column_kernel_dd(int per_thread, bool acc) {
  switch (per_thread) {
    case 1: return acc ? (const void*)&column_kernel<dd, 1, true, false> : (const void*)&column_kernel<dd, 1, false, false>;
    case 2: return acc ? (const void*)&column_kernel<dd, 2, true, false> : (const void*)&column_kernel<dd, 2, false, false>;
    case 4: return acc ? (const void*)&column_kernel<dd, 4, true, false> : (const void*)&column_kernel<dd, 4, false, false>;
    default: return nullptr;
  }
}

}  // namespace lbm
