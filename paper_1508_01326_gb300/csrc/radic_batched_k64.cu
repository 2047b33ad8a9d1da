// Binary64 kernels of the batched path, up to 8 rows.
#include "radic_batched.cuh"

namespace radic {
const void* batch_kernel_f64(int m, int path) {
  return m <= 8 ? batch_kernel<double, false, 1, 8>(m, path) : batch_kernel_f64_hi(m, path);
}
}  // namespace radic
