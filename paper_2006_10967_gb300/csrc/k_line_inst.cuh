// Instantiation helpers of the line kernels (included by k_line_quad.cu, k_line_hex.cu).
#pragma once
#include "kdispatch.hpp"
#include "kline.cuh"
#include "kline_pseudo.cuh"

namespace frp {

template <int DIM, int N>
unsigned line_grid(int64_t E, int warps) {
  const int per = warps * LL<DIM, N>::EPW;
  return (unsigned)((E + per - 1) / per);
}

template <int DIM, int N, bool GEN, bool TAB>
void launch_kb_line(const KArgs& A, cudaStream_t s) {
  constexpr int smem = KBLine<DIM, N, GEN, TAB>::F * 4 * kLineWarps;
  static_assert(smem <= 48 * 1024, "no shared-memory opt-in needed");
  const unsigned grid = line_grid<DIM, N>(A.E, kLineWarps);
  launch_pdl(kb_line<DIM, N, GEN, TAB, false, kLineWarps>, grid, kLineWarps * 32, smem, A, s);
}
// The unpreconditioned method (normal from phi) takes one kernel for all meshes.
template <int DIM, int N>
void launch_kb_line_phi(const KArgs& A, cudaStream_t s) {
  launch_pdl(kb_line<DIM, N, true, false, true, kLineWarps>, line_grid<DIM, N>(A.E, kLineWarps), kLineWarps * 32,
             KBLine<DIM, N, true, false>::F * 4 * kLineWarps, A, s);
}

template <int DIM, int N, bool GEN, int SF>
void launch_ka_stage(const KArgs& A, cudaStream_t s) {
  launch_pdl(ka_line<DIM, N, GEN, kLineWarps, SF>, line_grid<DIM, N>(A.E, kLineWarps), kLineWarps * 32,
             KALine<DIM, N, SF, GEN>::F * 4 * kLineWarps, A, s);
}

template <int DIM, int N, bool GEN>
void launch_ka_line(const KArgs& A, cudaStream_t s) {
  switch (A.stage) {
    case 0: launch_ka_stage<DIM, N, false, 0>(A, s); return;  // no metric
    case 1: launch_ka_stage<DIM, N, GEN, 1>(A, s); return;
    case 2: launch_ka_stage<DIM, N, GEN, 2>(A, s); return;
    case 3: launch_ka_stage<DIM, N, GEN, 3>(A, s); return;
    default: launch_ka_stage<DIM, N, GEN, 4>(A, s); return;
  }
}

template <int DIM, int N>
void launch_vel_tab(const KArgs& A, cudaStream_t s) {
  k_vel_tab<DIM, N><<<152 * 8, kThreads, 0, s>>>(A);
}

template <int DIM, int N, bool GEN, int SF>
bool prepare_ka_line() {
  return cudaFuncSetAttribute(ka_line<DIM, N, GEN, kLineWarps, SF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              KALine<DIM, N, SF, GEN>::F * 4 * kLineWarps) == cudaSuccess;
}

template <int DIM, int N, bool GEN>
bool fill_line_set(bool tab, KernelSet* ks) {
  if constexpr (GEN) ks->kb[0] = launch_kb_line<DIM, N, true, false>;
  else ks->kb[0] = tab ? launch_kb_line<DIM, N, false, true> : launch_kb_line<DIM, N, false, false>;
  ks->ka[0] = launch_ka_line<DIM, N, GEN>;
  ks->vtab = launch_vel_tab<DIM, N>;
  return prepare_ka_line<DIM, N, false, 0>() && prepare_ka_line<DIM, N, GEN, 1>() && prepare_ka_line<DIM, N, GEN, 2>() &&
         prepare_ka_line<DIM, N, GEN, 3>() && prepare_ka_line<DIM, N, GEN, 4>();
}

template <int DIM, int N>
bool fill_line(bool gen, bool tab, bool nphi, KernelSet* ks) {
  const bool ok = gen ? fill_line_set<DIM, N, true>(tab, ks) : fill_line_set<DIM, N, false>(tab, ks);
  if (nphi) ks->kb[0] = launch_kb_line_phi<DIM, N>;
  return ok;
}

template <int DIM, int N, bool GEN>
void launch_kb_pseudo(const KArgs& A, cudaStream_t s) {
  kbp_line<DIM, N, GEN, kPseudoWarps>
      <<<line_grid<DIM, N>(A.E, kPseudoWarps), kPseudoWarps * 32, KBPLine<DIM, N, GEN>::F * 4 * kPseudoWarps, s>>>(A);
}

template <int DIM, int N, bool GEN, int SF>
void launch_kap_stage(const KArgs& A, cudaStream_t s) {
  constexpr int smem = KAPLine<DIM, N, GEN>::F * 4 * kPseudoWarps;
  unsigned grid = line_grid<DIM, N>(A.E, kPseudoWarps);
  if (SF == 4 && grid > kPseudoBlocks) grid = kPseudoBlocks;
  kap_line<DIM, N, GEN, kPseudoWarps, SF><<<grid, kPseudoWarps * 32, smem, s>>>(A);
}

template <int DIM, int N, bool GEN>
void launch_ka_pseudo(const KArgs& A, cudaStream_t s) {
  switch (A.stage) {
    case 0: launch_kap_stage<DIM, N, false, 0>(A, s); return;
    case 1: launch_kap_stage<DIM, N, GEN, 1>(A, s); return;
    case 2: launch_kap_stage<DIM, N, GEN, 2>(A, s); return;
    case 3: launch_kap_stage<DIM, N, GEN, 3>(A, s); return;
    default: launch_kap_stage<DIM, N, GEN, 4>(A, s); return;
  }
}

template <int DIM, int N, bool GEN>
bool fill_line_pseudo(KernelSet* ks) {
  static_assert(KBPLine<DIM, N, GEN>::F * 4 * kPseudoWarps <= 48 * 1024 && KAPLine<DIM, N, GEN>::F * 4 * kPseudoWarps <= 48 * 1024,
                "no shared-memory opt-in needed");
  ks->kb[1] = launch_kb_pseudo<DIM, N, GEN>;
  ks->ka[1] = launch_ka_pseudo<DIM, N, GEN>;
  return true;
}

}  // namespace frp
