// Binary64 prefix kernels of depth 3 whose lane groups factor a prefix per lane
// (prefix_group): small launches, where every prefix is shared by many lanes.
#include "radic_prefix.cuh"

namespace radic {

const void* fp64_shared_kernel(int m) {
  switch (m) {
    case 7: return reinterpret_cast<const void*>(&k_fp_prefix<double, 7, 3, false, false, true>);
    case 8: return reinterpret_cast<const void*>(&k_fp_prefix<double, 8, 3, false, false, true>);
    case 9: return reinterpret_cast<const void*>(&k_fp_prefix<double, 9, 3, false, false, true>);
    case 10: return reinterpret_cast<const void*>(&k_fp_prefix<double, 10, 3, false, false, true>);
    default: return nullptr;
  }
}

}  // namespace radic
