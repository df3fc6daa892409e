// Instantiation helpers of the line kernels (included by k_line_quad.cu, k_line_hex.cu).
#pragma once
#include "kdispatch.hpp"
#include "kline.cuh"

namespace frp {

// Warps a block: the time factor (FP64) and the element balances (FP64) are
// computed once a block, so a block holds several warps.
constexpr int kLineWarps = 4;

template <int DIM, int N>
unsigned line_grid(int64_t E) {
  constexpr int per = kLineWarps * LL<DIM, N>::EPW;
  return (unsigned)((E + per - 1) / per);
}

template <int DIM, int N, bool GEN>
void launch_kb_line(const KArgs& A, cudaStream_t s) {
  kb_line<DIM, N, GEN, kLineWarps><<<line_grid<DIM, N>(A.E), kLineWarps * 32, KBLine<DIM, N>::F * 4 * kLineWarps, s>>>(A);
}

template <int DIM, int N, bool GEN, int SF>
void launch_ka_stage(const KArgs& A, cudaStream_t s) {
  ka_line<DIM, N, GEN, kLineWarps, SF>
      <<<line_grid<DIM, N>(A.E), kLineWarps * 32, KALine<DIM, N, SF>::F * 4 * kLineWarps, s>>>(A);
}

template <int DIM, int N, bool GEN>
void launch_ka_line(const KArgs& A, cudaStream_t s) {
  switch (A.stage) {
    case 0: launch_ka_stage<DIM, N, GEN, 0>(A, s); return;
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
                              KALine<DIM, N, SF>::F * 4 * kLineWarps) == cudaSuccess;
}

template <int DIM, int N, bool GEN>
bool fill_line(KernelSet* ks) {
  ks->kb[0] = launch_kb_line<DIM, N, GEN>;
  ks->ka[0] = launch_ka_line<DIM, N, GEN>;
  ks->vtab = launch_vel_tab<DIM, N>;
  return cudaFuncSetAttribute(kb_line<DIM, N, GEN, kLineWarps>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              KBLine<DIM, N>::F * 4 * kLineWarps) == cudaSuccess &&
         prepare_ka_line<DIM, N, GEN, 0>() && prepare_ka_line<DIM, N, GEN, 1>() && prepare_ka_line<DIM, N, GEN, 2>() &&
         prepare_ka_line<DIM, N, GEN, 3>() && prepare_ka_line<DIM, N, GEN, 4>();
}

}  // namespace frp
