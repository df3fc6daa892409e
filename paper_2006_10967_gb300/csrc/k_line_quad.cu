// Line-kernel instantiations for quadrilaterals (mixed precision, p = 1..6).
#include "k_line_inst.cuh"

namespace frp {
bool line_kernels_quad(int order, bool gen, bool tab, bool nphi, KernelSet* ks) {
  switch (order) {
    case 1: return fill_line<2, 2>(gen, tab, nphi, ks);
    case 2: return fill_line<2, 3>(gen, tab, nphi, ks);
    case 3: return fill_line<2, 4>(gen, tab, nphi, ks);
    case 4: return fill_line<2, 5>(gen, tab, nphi, ks);
    case 5: return fill_line<2, 6>(gen, tab, nphi, ks);
    case 6: return fill_line<2, 7>(gen, tab, nphi, ks);
    default: return false;
  }
}
bool line_pseudo_quad(int order, bool gen, KernelSet* ks) {
  switch (order) {
    case 1: return gen ? fill_line_pseudo<2, 2, true>(ks) : fill_line_pseudo<2, 2, false>(ks);
    case 2: return gen ? fill_line_pseudo<2, 3, true>(ks) : fill_line_pseudo<2, 3, false>(ks);
    case 3: return gen ? fill_line_pseudo<2, 4, true>(ks) : fill_line_pseudo<2, 4, false>(ks);
    case 4: return gen ? fill_line_pseudo<2, 5, true>(ks) : fill_line_pseudo<2, 5, false>(ks);
    case 5: return gen ? fill_line_pseudo<2, 6, true>(ks) : fill_line_pseudo<2, 6, false>(ks);
    case 6: return gen ? fill_line_pseudo<2, 7, true>(ks) : fill_line_pseudo<2, 7, false>(ks);
    default: return false;
  }
}
}  // namespace frp
