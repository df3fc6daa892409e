// Kernel tables per element type, order and precision (see k_*.cu).
#pragma once
#include <cuda_runtime.h>

#include "kcommon.cuh"

namespace frp {

typedef void (*LaunchFn)(const KArgs&, cudaStream_t);

struct KernelSet {
  LaunchFn kb[2] = {nullptr, nullptr};  // [mode]: 0 physical, 1 preconditioning
  LaunchFn ka[2] = {nullptr, nullptr};
  LaunchFn ka_rate = nullptr;           // the block-wide ka[0], ka[1]: their stage -1 writes the
  LaunchFn ka_rate_pseudo = nullptr;    // rate into KArgs.out
  LaunchFn vtab = nullptr;              // fills the velocity factor table (line kernels)
  LaunchFn vtab64 = nullptr;            // fills the separable velocity tables (FP64 tensor fields)
  int max_blocks = 0;                   // upper bound on blocks of any launch (per element count)
  LaunchFn vcache = nullptr;            // fills the spatial velocity cache (nullptr: not supported)
  LaunchFn mconst = nullptr;            // fills the per-element metric records (tensor elements)
  bool prepared = false;                // shared-memory limits set for every kernel of the set
};

// Return false if the (order, precision) pair is not built.
bool kernels_quad(int order, int precision, int64_t E, int variant, KernelSet* ks);
bool kernels_hex(int order, int precision, int64_t E, int variant, KernelSet* ks);
bool kernels_tri(int order, int precision, int64_t E, int variant, KernelSet* ks);

// Largest mesh whose FP64 preconditioning may take small tiles; every field has
// a reduction slot an element up to that size.
constexpr int64_t kSmallTileElems = 16384;

// Replace the physical-step kernels of a mixed tensor field by the line kernels
// (kline.cuh); false where they are not built (the set is then unchanged) or
// could not be prepared.  gen, tab: see KBLine; nphi: normal from phi.
bool line_kernels_quad(int order, bool gen, bool tab, bool nphi, KernelSet* ks);
bool line_kernels_hex(int order, bool gen, bool tab, bool nphi, KernelSet* ks);
// The same for the preconditioning kernels of a mixed tensor field; gen false:
// every element is affine with a diagonal Jacobian.
bool line_pseudo_quad(int order, bool gen, KernelSet* ks);
bool line_pseudo_hex(int order, bool gen, KernelSet* ks);

// Triangles of p <= 4 in mixed precision: the thread-per-element kernels for the
// preconditioning and, when asked (the field has its velocity cache), the
// physical step.
bool reg_kernels_tri(int order, bool physical, KernelSet* ks);

// Warps a block of the line kernels.  Their warps are independent, so small
// blocks spread best (64^3 hexes p = 3, residual + update: 185 + 183 us with
// four, 183 + 178 with two).  The preconditioning's stage 4 leaves one partial
// a block for the last block to add up, on a grid of a fixed number of blocks:
// four warps each, half the partials of two.
constexpr int kLineWarps = 2, kPseudoWarps = 4;
// Blocks of the preconditioning's stage 4 update: six of 128 threads on each SM.
constexpr unsigned kPseudoBlocks = 152 * 6;

// Launch with programmatic stream serialisation: the kernel's blocks may start
// while the kernel before it on the stream drains (the kernel itself waits, see
// pdl_wait in kline.cuh).  After a kernel that does not let its dependents
// start early, it is an ordinary launch.  us a stage with and without: 128^2
// quads p = 4 11.93 and 12.04, 200^2 p = 5 29.2 and 29.5, jittered 211 x 187 p = 3
// 17.5 and 18.2, jittered hexes 27 x 22 x 19 p = 2 21.0 and 21.8, 32^3 p = 3 71.8
// and 72.8, regular 32^3 p = 4 the same (123.6 and 123.5); past kEarlyBlocks there
// is little to hide and the early blocks cost more (64^3 hexes p = 3: 354 and 351).
constexpr unsigned kEarlyBlocks = 152 * 160;
template <typename K>
inline void launch_pdl(K kern, unsigned grid, int threads, size_t smem, const KArgs& A, cudaStream_t s) {
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = grid <= kEarlyBlocks ? 1 : 0;
  cudaLaunchKernelEx(&c, kern, A);
}

template <typename K>
inline void launch_kernel(K kern, size_t smem, int et, const KArgs& A, cudaStream_t s, int threads = kThreads) {
  const int64_t grid = (A.E + et - 1) / et;
  kern<<<(unsigned)grid, threads, smem, s>>>(A);
}

}  // namespace frp
