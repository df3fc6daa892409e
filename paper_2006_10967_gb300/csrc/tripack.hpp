// Layout of the packed triangle operators (ktri_reg.cuh), shared with the host
// code that fills them.
#pragma once
#ifndef __CUDACC__
#define __host__
#define __device__
#endif

namespace frp {

// Offsets, in floats, of the packed operators of order p (host and device):
// rows of output pairs, padded to an even number of pairs where there are
// several, one row per input.
struct TriPack {
  int n, nu, nf, npe, npu, o_l, o_d, o_lift, o_v, size;
  __host__ __device__ constexpr TriPack(int p)
      : n(p + 1), nu((p + 1) * (p + 2) / 2), nf(3 * (p + 1)), npe(even((p + 2) / 2)),
        npu(even(((p + 1) * (p + 2) / 2 + 1) / 2)), o_l(0), o_d(0), o_lift(0), o_v(0), size(0) {
    o_d = (o_l + 3 * nu * npe * 2 + 3) / 4 * 4;  // L: [edge][input][pairs of the edge's points]
    o_lift = o_d + 2 * nu * npu * 2;             // D: [direction][input][pairs]
    o_v = o_lift + nf * npu * 2;                 // LIFT: [flux point][pairs]
    size = o_v + nu * npu * 2;                   // Vinv: [input][mode pairs]
  }
  static __host__ __device__ constexpr int even(int x) { return x <= 1 ? 1 : (x + 1) / 2 * 2; }
};

}  // namespace frp
