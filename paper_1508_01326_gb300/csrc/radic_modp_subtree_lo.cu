// Exact subtree kernels of 3 to 8 rows (radic_modp_subtree.cuh).
#include "radic_modp_subtree.cuh"

namespace radic {

const void* modp_subtree_kernel(int m, int G) {
  switch (m) {
    case 3: return kernel_m<3>(G);
    case 4: return kernel_m<4>(G);
    case 5: return kernel_m<5>(G);
    case 6: return kernel_m<6>(G);
    case 7: return kernel_m<7>(G);
    case 8: return kernel_m<8>(G);
    default: return modp_subtree_kernel_hi(m, G);
  }
}

size_t modp_subtree_smem(int m, int n) { return SubtreeSmem(nullptr, n, m).bytes; }

}  // namespace radic
