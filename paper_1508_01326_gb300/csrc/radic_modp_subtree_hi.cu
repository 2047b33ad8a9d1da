// Exact subtree kernels of 9 to 12 rows (radic_modp_subtree.cuh).
#include "radic_modp_subtree.cuh"

namespace radic {

const void* modp_subtree_kernel_hi(int m, int G) {
  switch (m) {
    case 9: return kernel_m<9>(G);
    case 10: return kernel_m<10>(G);
    case 11: return kernel_m<11>(G);
    case 12: return kernel_m<12>(G);
    default: return nullptr;
  }
}

}  // namespace radic
