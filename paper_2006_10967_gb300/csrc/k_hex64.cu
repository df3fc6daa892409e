// Hexahedron kernel instantiations in FP64 (p = 1..5).
#include "k_tensor_inst.cuh"

namespace frp {
bool kernels_hex64(int order, int64_t E, KernelSet* ks) {
  switch (order) {
    case 1: fill_tensor<3, 2, double>(E, ks); return true;
    case 2: fill_tensor<3, 3, double>(E, ks); return true;
    case 3: fill_tensor<3, 4, double>(E, ks); return true;
    case 4: fill_tensor<3, 5, double>(E, ks); return true;
    case 5: fill_tensor<3, 6, double>(E, ks); return true;
    default: return false;
  }
}
}  // namespace frp
