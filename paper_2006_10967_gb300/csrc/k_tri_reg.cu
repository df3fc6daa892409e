// Instantiations of the thread-per-element triangle kernels (mixed precision, p = 1..4).
#include "kdispatch.hpp"
#include "ktri_reg.cuh"

namespace frp {

template <int P>
unsigned tri_grid(int64_t E) {
  return (unsigned)((E + TriReg<P>::TB - 1) / TriReg<P>::TB);
}
template <int P, int MODE>
void launch_kb_trir(const KArgs& A, cudaStream_t s) {
  kb_trir<P, MODE><<<tri_grid<P>(A.E), TriReg<P>::TB, TriReg<P>::KB_SMEM, s>>>(A);
}
template <int P, int MODE, int SF>
void launch_ka_stage(const KArgs& A, cudaStream_t s) {
  constexpr int per = TriReg<P>::TB / 32 * TriReg<P>::ka_elems(MODE);
  ka_trir<P, MODE, SF><<<(unsigned)((A.E + per - 1) / per), TriReg<P>::TB, TriReg<P>::ka_smem(MODE), s>>>(A);
}
template <int P, int MODE>
void launch_ka_trir(const KArgs& A, cudaStream_t s) {
  switch (A.stage) {
    case 0: launch_ka_stage<P, MODE, 0>(A, s); return;
    case 1: launch_ka_stage<P, MODE, 1>(A, s); return;
    case 2: launch_ka_stage<P, MODE, 2>(A, s); return;
    case 3: launch_ka_stage<P, MODE, 3>(A, s); return;
    default: launch_ka_stage<P, MODE, 4>(A, s); return;
  }
}
template <int P>
bool fill_trir(bool physical, KernelSet* ks) {
  static_assert(TriReg<P>::KB_SMEM <= 48 * 1024 && TriReg<P>::ka_smem(1) <= 48 * 1024, "no shared-memory opt-in needed");
  if (physical) {
    ks->kb[0] = launch_kb_trir<P, 0>;
    ks->ka[0] = launch_ka_trir<P, 0>;
  }
  ks->kb[1] = launch_kb_trir<P, 1>;
  ks->ka[1] = launch_ka_trir<P, 1>;
  return true;
}

bool reg_kernels_tri(int order, bool physical, KernelSet* ks) {
  switch (order) {
    case 1: return fill_trir<1>(physical, ks);
    case 2: return fill_trir<2>(physical, ks);
    case 3: return fill_trir<3>(physical, ks);
    case 4: return fill_trir<4>(physical, ks);
    default: return false;
  }
}

}  // namespace frp
