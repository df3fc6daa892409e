// Instantiation helpers for the tensor kernels (included by k_quad.cu, k_hex.cu).
#pragma once
#include <algorithm>
#include <cmath>

#include "kdispatch.hpp"
#include "ktensor.cuh"

namespace frp {

// The mixed preconditioning of quads and of hexes p <= 4 always runs in the line
// kernels (use_line_pseudo); only its update kernel's rate output is kept here.
template <int DIM, int N, typename T, int MODE>
struct HasKB {
  static constexpr bool v = !(MODE == 1 && sizeof(T) == 4 && (DIM == 2 || N <= 5));
};

template <int DIM, int N, typename T, int MODE, int TD = 1>
void launch_kb_tensor(const KArgs& A, cudaStream_t s) {
  using LY = KBLayout<DIM, N, T, MODE, TD>;
  launch_kernel(kb_tensor<DIM, N, T, MODE, TD>, LY::SMEM, LY::ET, A, s, LY::THREADS);
}

template <int DIM, int N, typename T, int MODE, int TD = 1>
void launch_ka_tensor(const KArgs& A, cudaStream_t s) {
  using LY = KALayout<DIM, N, T, MODE, TD>;
  if constexpr (StageKA<DIM, T, MODE>::v) {
    switch (A.stage) {
      case 1: launch_kernel(ka_tensor<DIM, N, T, MODE, TD, 1>, LY::SMEM, LY::ET, A, s, LY::THREADS); return;
      case 2: launch_kernel(ka_tensor<DIM, N, T, MODE, TD, 2>, LY::SMEM, LY::ET, A, s, LY::THREADS); return;
      case 3: launch_kernel(ka_tensor<DIM, N, T, MODE, TD, 3>, LY::SMEM, LY::ET, A, s, LY::THREADS); return;
      case 4: launch_kernel(ka_tensor<DIM, N, T, MODE, TD, 4>, LY::SMEM, LY::ET, A, s, LY::THREADS); return;
      default: break;
    }
  }
  launch_kernel(ka_tensor<DIM, N, T, MODE, TD>, LY::SMEM, LY::ET, A, s, LY::THREADS);
}

template <int DIM, int N, typename T, int MODE, int TD, int SF>
bool prepare_ka() {
  return cudaFuncSetAttribute(ka_tensor<DIM, N, T, MODE, TD, SF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)KALayout<DIM, N, T, MODE, TD>::SMEM) == cudaSuccess;
}

template <int DIM, int N, typename T>
void launch_mconst(const KArgs& A, cudaStream_t s) {
  const int64_t g = (A.E + kThreads - 1) / kThreads;
  k_metric_const<DIM, T><<<(unsigned)(g < 152 * 8 ? g : 152 * 8), kThreads, 0, s>>>(A, TS<DIM, N>::NG, TS<DIM, N>::NU);
}

template <int DIM, int N, typename T>
void launch_vcache(const KArgs& A, cudaStream_t s) {
  k_vel_cache<DIM, N, T><<<152 * 8, kThreads, 0, s>>>(A);
}

// Shared-memory opt-in of one (kb, ka) pair; done when the kernel table is
// filled, so that no launch (and no graph capture) has to do it.
template <int DIM, int N, typename T, int MODE, int TD = 1>
bool prepare_tensor() {
  bool ok = prepare_ka<DIM, N, T, MODE, TD, -2>();
  if constexpr (HasKB<DIM, N, T, MODE>::v)
    ok = ok && cudaFuncSetAttribute(kb_tensor<DIM, N, T, MODE, TD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)KBLayout<DIM, N, T, MODE, TD>::SMEM) == cudaSuccess;
  if constexpr (StageKA<DIM, T, MODE>::v)
    ok = ok && prepare_ka<DIM, N, T, MODE, TD, 1>() && prepare_ka<DIM, N, T, MODE, TD, 2>() &&
         prepare_ka<DIM, N, T, MODE, TD, 3>() && prepare_ka<DIM, N, T, MODE, TD, 4>();
  return ok;
}

template <int DIM, int N>
void launch_vel_tab64(const KArgs& A, cudaStream_t s) {
  k_vel_tab64<DIM, N><<<152 * 8, kThreads, 0, s>>>(A);
}

// FP64 fields: the residual kernel's time in clocks with tile layout LY, as the
// larger of the FP64 pipe's work on the busiest SM (16 clocks a warp
// instruction whatever its active lanes) and one block's chain of dependent
// instructions (about 90 clocks each with few warps on an SM).  A warp executes
// about DIM 4 N (N + 4) FP64 instructions in the line passes, 90 a round of
// points (in the line pass for odd N) and 110 a round of common-flux points.
// 256 quads p = 3: 39.8 us with the default tile (11 blocks), 38.8 with one
// warp's eight elements, 28.7 with four, 22.4 with one or two; 4,096 quads
// p = 4: 67 us with the default tile (two blocks of three warps on an SM), 55
// with one warp's.
template <int DIM, int N, typename LY>
double kb_clocks(int64_t E) {
  using S = TS<DIM, N>;
  constexpr int W = LY::THREADS / 32;
  constexpr double line = DIM * 4.0 * N * (N + 4) + (N % 2 ? 90.0 * N : 0.0);
  constexpr double pts = N % 2 ? 0.0 : 90.0, flux = 110.0;
  const auto up = [](double a, double b) { return std::ceil(a / b); };
  const double work = W * line + up(LY::ET * S::NU, 32) * pts + up(LY::ET * S::NF / 2.0, 32) * flux;
  const double chain = line + up(LY::ET * S::NU, LY::THREADS) * pts + up(LY::ET * S::NF / 2.0, LY::THREADS) * flux;
  return std::max(16.0 * up(up((double)E, LY::ET), 152) * work, 90.0 * chain);
}
// The update kernel has no rounds: the warps on the busiest SM decide.
template <typename LY>
int64_t ka_warps(int64_t E) {
  return ((E + LY::ET - 1) / LY::ET + 151) / 152 * (LY::THREADS / 32);
}

// TB, TA: the tile divisors of the physical-step residual and update
// kernels (the kernel variant; the preconditioning kernels keep the default
// tiles)
template <int DIM, int N, typename T, int TB = 1, int TA = 1>
void fill_tensor(int64_t E, KernelSet* ks) {
  ks->prepared = prepare_tensor<DIM, N, T, 0, TB>() && prepare_tensor<DIM, N, T, 0, TA>() &&
                 prepare_tensor<DIM, N, T, 1>();
  ks->vcache = launch_vcache<DIM, N, T>;
  ks->mconst = launch_mconst<DIM, N, T>;
  ks->kb[0] = launch_kb_tensor<DIM, N, T, 0, TB>;
  if constexpr (HasKB<DIM, N, T, 1>::v) ks->kb[1] = launch_kb_tensor<DIM, N, T, 1>;
  ks->ka[0] = launch_ka_tensor<DIM, N, T, 0, TA>;
  ks->ka_rate = ks->ka[0];
  ks->ka[1] = launch_ka_tensor<DIM, N, T, 1>;
  ks->ka_rate_pseudo = ks->ka[1];
  if constexpr (sizeof(T) == 8) {
    ks->vtab64 = launch_vel_tab64<DIM, N>;
    ks->prepared = ks->prepared && prepare_tensor<DIM, N, T, 0, 0>() && prepare_tensor<DIM, N, T, 0, -1>();
    const double t1 = kb_clocks<DIM, N, KBLayout<DIM, N, T, 0, TB>>(E), t0 = kb_clocks<DIM, N, KBLayout<DIM, N, T, 0, 0>>(E),
                 tq = kb_clocks<DIM, N, KBLayout<DIM, N, T, 0, -1>>(E);
    if (tq < t0 && tq < t1) ks->kb[0] = launch_kb_tensor<DIM, N, T, 0, -1>;
    else if (t0 < t1) ks->kb[0] = launch_kb_tensor<DIM, N, T, 0, 0>;
    // the preconditioning's reduction keeps a partial a block: small tiles only
    // where they stay within the slots every field has
    if (E <= kSmallTileElems) {
      ks->prepared = ks->prepared && prepare_tensor<DIM, N, T, 1, 0>();
      if (kb_clocks<DIM, N, KBLayout<DIM, N, T, 1, 0>>(E) < kb_clocks<DIM, N, KBLayout<DIM, N, T, 1>>(E))
        ks->kb[1] = launch_kb_tensor<DIM, N, T, 1, 0>;
      if (ka_warps<KALayout<DIM, N, T, 1, 0>>(E) < ka_warps<KALayout<DIM, N, T, 1>>(E)) {
        ks->ka[1] = launch_ka_tensor<DIM, N, T, 1, 0>;
        ks->ka_rate_pseudo = ks->ka[1];
      }
    }
    if (ka_warps<KALayout<DIM, N, T, 0, 0>>(E) < ka_warps<KALayout<DIM, N, T, 0, TA>>(E)) {
      ks->ka[0] = launch_ka_tensor<DIM, N, T, 0, 0>;
      ks->ka_rate = ks->ka[0];
    }
  }
  const int et_min = KBLayout<DIM, N, T, 0, TB>::ET < KALayout<DIM, N, T, 0, TA>::ET ? KBLayout<DIM, N, T, 0, TB>::ET
                                                                                      : KALayout<DIM, N, T, 0, TA>::ET;
  const int et_min1 = KBLayout<DIM, N, T, 1>::ET < KALayout<DIM, N, T, 1>::ET ? KBLayout<DIM, N, T, 1>::ET
                                                                               : KALayout<DIM, N, T, 1>::ET;
  const int et = et_min < et_min1 ? et_min : et_min1;
  ks->max_blocks = (int)((E + et - 1) / et);
}

}  // namespace frp
