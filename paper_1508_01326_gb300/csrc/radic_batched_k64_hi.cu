// Binary64 kernels of the batched path, 9 and 10 rows.
#include "radic_batched.cuh"

namespace radic {
const void* batch_kernel_f64_hi(int m, int path) { return batch_kernel<double, false, 9, 10>(m, path); }
}  // namespace radic
