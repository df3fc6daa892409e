// Line-kernel instantiations for hexahedra (mixed precision, p = 1..4: at p = 5
// an element has 36 lines, more than a warp's lanes).
#include "k_line_inst.cuh"

namespace frp {
bool line_kernels_hex(int order, bool gen, bool tab, bool nphi, KernelSet* ks) {
  switch (order) {
    case 1: return fill_line<3, 2>(gen, tab, nphi, ks);
    case 2: return fill_line<3, 3>(gen, tab, nphi, ks);
    case 3: return fill_line<3, 4>(gen, tab, nphi, ks);
    case 4: return fill_line<3, 5>(gen, tab, nphi, ks);
    default: return false;
  }
}
bool line_pseudo_hex(int order, bool gen, KernelSet* ks) {
  switch (order) {
    case 1: return gen ? fill_line_pseudo<3, 2, true>(ks) : fill_line_pseudo<3, 2, false>(ks);
    case 2: return gen ? fill_line_pseudo<3, 3, true>(ks) : fill_line_pseudo<3, 3, false>(ks);
    case 3: return gen ? fill_line_pseudo<3, 4, true>(ks) : fill_line_pseudo<3, 4, false>(ks);
    case 4: return gen ? fill_line_pseudo<3, 5, true>(ks) : fill_line_pseudo<3, 5, false>(ks);
    default: return false;
  }
}
}  // namespace frp
