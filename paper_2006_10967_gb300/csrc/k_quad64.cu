// Quadrilateral kernel instantiations in FP64 (p = 1..6).
#include "k_tensor_inst.cuh"

namespace frp {
bool kernels_quad64(int order, int64_t E, KernelSet* ks) {
  switch (order) {
    case 1: fill_tensor<2, 2, double>(E, ks); return true;
    case 2: fill_tensor<2, 3, double>(E, ks); return true;
    case 3: fill_tensor<2, 4, double>(E, ks); return true;
    case 4: fill_tensor<2, 5, double>(E, ks); return true;
    case 5: fill_tensor<2, 6, double>(E, ks); return true;
    case 6: fill_tensor<2, 7, double>(E, ks); return true;
    default: return false;
  }
}
}  // namespace frp
