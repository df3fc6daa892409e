// Warp-per-element kernels of the mixed path's physical RK stage on
// quadrilaterals and hexahedra: the same Steps 1-6, arrays and face
// conventions as kb_tensor / ka_tensor (ktensor.cuh), organised so that an
// element lives in the registers of one warp.
//
// One lane owns one solution-point line along axis 0 (LN = N^(DIM-1) lines an
// element, EPW = 32 / LN elements a warp) and keeps both fields, their
// gradient and the flux of its points in registers.  For axis a > 0 the same
// lane l also plays line l of that axis: it reads the line's points from a
// warp-private shared array (written as rows by the axis-0 owners), applies
// the 1D operators and writes the result back in place.  A lane therefore
// holds both ends of one line of every axis: traces, partner traces, common
// fluxes and corrections of the face points never leave registers, and no
// barrier wider than a warp separates the passes.
//
// Arithmetic is paired (fma.rn.f32x2): along a line two neighbouring outputs,
// at the faces the two ends of a line, and in the pointwise flux two points
// of an axis-0 line share one instruction; the 1D operators come from the
// kernel parameters laid out in those pairs (LineOps).
//
// What bounds it: the residual kernel (kb_line) issues instructions (the
// block-wide kb_tensor executed 796 a point and stage, at 67 % of the issue
// slots; here 272 on hexes p = 3, at 61 to 66 %), the update kernel (ka_line)
// moves memory.  Per stage on 64^3 hexes p = 3 (16.8 M points): residual 483 ->
// 172 us, update 228 -> 182 us (61 bytes of DRAM traffic a point: 5.6 TB/s).
#pragma once
#include "ktensor.cuh"

namespace frp {

// ---- paired FP32 (two lanes of one 64-bit register pair) --------------------
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{.reg .b64 ra, rb, rc, rd;\n"
      "mov.b64 ra, {%2, %3}; mov.b64 rb, {%4, %5}; mov.b64 rc, {%6, %7};\n"
      "fma.rn.ftz.f32x2 rd, ra, rb, rc;\n"
      "mov.b64 {%0, %1}, rd;}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 d;
  asm("{.reg .b64 ra, rb, rd;\n"
      "mov.b64 ra, {%2, %3}; mov.b64 rb, {%4, %5};\n"
      "mul.rn.ftz.f32x2 rd, ra, rb;\n"
      "mov.b64 {%0, %1}, rd;}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("{.reg .b64 ra, rb, rd;\n"
      "mov.b64 ra, {%2, %3}; mov.b64 rb, {%4, %5};\n"
      "add.rn.ftz.f32x2 rd, ra, rb;\n"
      "mov.b64 {%0, %1}, rd;}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }
// c - a b, a - b
__device__ __forceinline__ float2 nfma2(float2 a, float2 b, float2 c) {
  return make_float2(__fmaf_rn(-a.x, b.x, c.x), __fmaf_rn(-a.y, b.y, c.y));
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, make_float2(-1.f, -1.f), a); }

// ---- layout -----------------------------------------------------------------
// Elements per warp, padded row (RS), plane (PS) and array (AS) strides of the
// warp-private arrays, in floats.  A row (axis-0 line) moves in 8-byte words,
// or one 16-byte word for N = 4; a line of another axis in 4-byte words.  The
// strides come from counting the shared-memory wavefronts of one row and one
// line access over the 32 banks: (row, axis-1 line, axis-2 line) in wavefronts
// for quads N = 3..7 (4,6) (4,4) (6,10) (6,12) (8,14), where dense rows of
// 2 NP floats with arrays padded for the lines alone gave (8,6) (8,4) (21,10)
// (18,6) (36,7); for hexes N = 3, 4, 5 (4,6,6) (8,4,4) (6,15,5).
template <int DIM, int N>
struct LL {
  using S = TS<DIM, N>;
  static constexpr int NU = S::NU, NF = S::NF, NFP = S::NFP, LN = S::NFP;
  static constexpr int EPW = 32 / LN;
  static constexpr int NP = (N + 1) / 2;
  static constexpr int RS = DIM == 3 ? (N == 3 ? 6 : 2 * NP) : (N == 3 ? 6 : N == 4 ? 8 : N == 5 || N == 7 ? 10 : 2 * NP);
  static constexpr int PS = DIM == 3 ? (N == 2 ? 4 : N == 3 ? 18 : N == 4 ? 20 : 30) : N * RS;
  static constexpr int AS = DIM == 3 ? (N == 2 ? 8 : N == 3 ? 54 : N == 4 ? 80 : 150) : (N == 4 ? 36 : N * RS);
  static constexpr bool V4 = N == 4;  // a row is one 16-byte word
  static_assert(RS % 2 == 0 && PS % 2 == 0 && AS % 2 == 0, "rows on 8-byte boundaries");
  static_assert(!V4 || (RS % 4 == 0 && PS % 4 == 0 && AS % 4 == 0), "rows on 16-byte boundaries");
  static constexpr bool FULL = 32 % LN == 0;  // every lane owns a line
  // rows read and written as vectors straight from global memory (a whole
  // number of 8- or 16-byte words, neighbouring lanes contiguous); other N
  // pass through a warp-private buffer copied with unit stride
  static constexpr bool DIRECT = N == 2 || N == 4;
  static constexpr int OTH = DIM == 3 ? N : 1;  // rows of a face buffer
  static_assert(LN <= 32, "one line per lane");
};

// offset of line l of axis a in the padded array, and its stride
template <int DIM, int N>
__device__ __forceinline__ int pline(int a, int l) {
  using L = LL<DIM, N>;
  if (DIM == 2) return a == 0 ? l * L::RS : l;
  if (a == 0) return (l / N) * L::PS + (l % N) * L::RS;
  if (a == 1) return (l / N) * L::PS + l % N;
  return (l / N) * L::RS + l % N;
}
template <int DIM, int N>
__host__ __device__ constexpr int pstride(int a) {
  return a == 0 ? 1 : (a == 1 ? LL<DIM, N>::RS : LL<DIM, N>::PS);
}

// one padded row (2 NP floats, 8-byte aligned; 16 for V4)
template <int NP, bool V4>
__device__ __forceinline__ void row_put(float* p, const float2* v) {
  if constexpr (V4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  } else {
#pragma unroll
    for (int i = 0; i < NP; ++i) reinterpret_cast<float2*>(p)[i] = v[i];
  }
}
template <int NP, bool V4>
__device__ __forceinline__ void row_get(const float* p, float2* v) {
  if constexpr (V4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = make_float2(q.x, q.y);
    v[1] = make_float2(q.z, q.w);
  } else {
#pragma unroll
    for (int i = 0; i < NP; ++i) v[i] = reinterpret_cast<const float2*>(p)[i];
  }
}
// a line's N values with stride ST
template <int N, int ST>
__device__ __forceinline__ void line_get(const float* p, float* v) {
#pragma unroll
  for (int m = 0; m < N; ++m) v[m] = p[m * ST];
}
template <int N, int ST>
__device__ __forceinline__ void line_put(float* p, const float2* v) {
#pragma unroll
  for (int m = 0; m < N; ++m) p[m * ST] = (m & 1) ? v[m / 2].y : v[m / 2].x;
}
template <int N>
__device__ __forceinline__ void unpair(const float2* v, float* s) {
#pragma unroll
  for (int m = 0; m < N; ++m) s[m] = (m & 1) ? v[m / 2].y : v[m / 2].x;
}

// both end values of a line: (sum_j l_j(-1) v_j, sum_j l_j(+1) v_j)
template <int N>
__device__ __forceinline__ float2 line_ends(const LineOps& O, const float* v) {
  float2 t = mul2(O.lend[0], dup2(v[0]));
#pragma unroll
  for (int m = 1; m < N; ++m) t = fma2(O.lend[m], dup2(v[m]), t);
  return t;
}
// derivative along a line plus the lifts of c at the two ends (signs in g0, g1)
template <int N>
__device__ __forceinline__ void line_deriv(const LineOps& O, const float* v, const float2* g0, const float2* g1,
                                           float2 c, float2* out) {
  constexpr int NP = (N + 1) / 2;
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    float2 r = fma2(g1[p], dup2(c.y), mul2(g0[p], dup2(c.x)));
#pragma unroll
    for (int m = 0; m < N; ++m) r = fma2(O.D[m][p], dup2(v[m]), r);
    out[p] = r;
  }
}

// asynchronous copy of n8 8-byte words between a warp-private buffer and
// global memory, unit stride over the lanes
__device__ __forceinline__ void cp_async_8(void* sdst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
// A tile's share of an array of PER bytes an element, ne of at most EPW
// elements: whole tiles in a compile-time count of the widest words that every
// tile's start allows (arrays start on 256-byte boundaries).
// `dst` is on a 16-byte boundary (every buffer offset is a multiple of 4 floats).
template <int EPW, int PER>
__device__ __forceinline__ void tile_fetch(float* dst, const void* src, int ne, int lane) {
  constexpr int FULL = EPW * PER, W = FULL % 16 == 0 ? 16 : FULL % 8 == 0 ? 8 : 4;
  char* d = reinterpret_cast<char*>(dst);
  const char* s = static_cast<const char*>(src);
  if (ne == EPW) {
#pragma unroll
    for (int r = 0; r < (FULL / W + 31) / 32; ++r) {
      const int i = r * 32 + lane;
      if (i < FULL / W) {
        if constexpr (W == 16) cp_async_16(d + 16 * i, s + 16 * i);
        else if constexpr (W == 8) cp_async_8(d + 8 * i, s + 8 * i);
        else cp_async_4(d + 4 * i, s + 4 * i);
      }
    }
  } else {
    for (int i = lane; i < ne * PER / 4; i += 32) cp_async_4(d + 4 * i, s + 4 * i);
  }
}
// Programmatic dependent launch: a kernel's blocks start while the kernel before
// it drains.  Only pdl_wait makes another kernel's writes visible, so before it
// they read nothing that a kernel of the march writes: connectivity, metric,
// weights, parameters and velocity data, all written at set-up.  The solution,
// accumulator and flux balances of the update kernels come from the update two
// kernels before, which is complete by then, but they are read after pdl_wait
// like the rest.  Every kernel waits before it returns.
// kEarly: regular hexes of N >= 4 (the large 3D runs) load their state before the
// connectivity: with thousands of blocks a wave there is little to hide (64^3
// p = 3 358 and 350 us a stage; their update kernels' metric and weights still
// come first, 32^3 p = 4 123.4 and 125.2 us with them after the state).
template <int DIM, int N, bool GEN>
constexpr bool kEarly = !(DIM == 3 && N >= 4 && !GEN);
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void cp_async_wait_but() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(LEFT) : "memory");
}
__device__ __forceinline__ void warp_flush(void* dst, const float* src, int nfloats, int lane) {
  float2* d = static_cast<float2*>(dst);
  for (int i = lane; i < nfloats / 2; i += 32) d[i] = reinterpret_cast<const float2*>(src)[i];
}

// a row of N floats (pairs, the pad of odd N zero) from global memory
template <int N>
__device__ __forceinline__ void grow_get(const float* p, float2* v) {
  if constexpr (N == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = make_float2(q.x, q.y);
    v[1] = make_float2(q.z, q.w);
  } else if constexpr (N == 2) {
    v[0] = *reinterpret_cast<const float2*>(p);
  } else {
#pragma unroll
    for (int i = 0; i < (N + 1) / 2; ++i) v[i] = make_float2(p[2 * i], 2 * i + 1 < N ? p[2 * i + 1] : 0.f);
  }
}
template <int N>
__device__ __forceinline__ void grow_put(float* p, const float2* v) {
  if constexpr (N == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  } else if constexpr (N == 2) {
    *reinterpret_cast<float2*>(p) = v[0];
  } else {
#pragma unroll
    for (int m = 0; m < N; ++m) p[m] = (m & 1) ? v[m / 2].y : v[m / 2].x;
  }
}

// ---- metric of the general path ---------------------------------------------
// Column b of the Jacobian, J[c][b] = d x_c / d xi_b, at paired points.
template <int DIM>
__device__ __forceinline__ void jac_col(const float* g, int b, const float2* xi, float2* J) {
#pragma unroll
  for (int c = 0; c < DIM; ++c) {
    if (DIM == 2) {
      const float* k = g + c * 4;
      J[c] = fma2(dup2(k[3]), xi[1 - b], dup2(k[1 + b]));
    } else {
      const float* k = g + c * 8;
      // other axes p < q; cross coefficients k4 (01), k5 (02), k6 (12), k7 (012)
      const int p = b == 0 ? 1 : 0, q = b == 2 ? 1 : 2;
      const float kp = k[b == 2 ? 5 : 4];  // with axis p: (01), (01), (02)
      const float kq = k[b == 0 ? 5 : 6];  // with axis q: (02), (12), (12)
      const float2 t = fma2(dup2(k[7]), xi[q], dup2(kp));
      J[c] = fma2(t, xi[p], fma2(dup2(kq), xi[q], dup2(k[1 + b])));
    }
  }
}
__device__ __forceinline__ void cross2(const float2* a, const float2* b, float2* r) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int j = (i + 1) % 3, k = (i + 2) % 3;
    r[i] = nfma2(a[k], b[j], mul2(a[j], b[k]));
  }
}
// Row a of S = det J J^{-1} at paired points (the transformed normal of axis a).
template <int DIM>
__device__ __forceinline__ void metric_row(const float* g, int a, const float2* xi, float2* Sr) {
  if (DIM == 2) {
    float2 J[2];
    jac_col<2>(g, 1 - a, xi, J);
    // S0 = (J11, -J01), S1 = (-J10, J00)
    Sr[a] = J[1 - a];
    Sr[1 - a] = make_float2(-J[a].x, -J[a].y);
  } else {
    float2 P[3], Q[3];
    jac_col<DIM>(g, (a + 1) % 3, xi, P);
    jac_col<DIM>(g, (a + 2) % 3, xi, Q);
    cross2(P, Q, Sr);
  }
}
// All rows and det J.
template <int DIM>
__device__ __forceinline__ float2 metric_all(const float* g, const float2* xi, float2 Sm[3][3]) {
  if (DIM == 2) {
    float2 A[2], B[2];
    jac_col<2>(g, 0, xi, A);
    jac_col<2>(g, 1, xi, B);
    Sm[0][0] = B[1];
    Sm[0][1] = make_float2(-B[0].x, -B[0].y);
    Sm[1][0] = make_float2(-A[1].x, -A[1].y);
    Sm[1][1] = A[0];
    return nfma2(B[0], A[1], mul2(A[0], B[1]));
  }
  float2 A[3], B[3], C[3];
  jac_col<DIM>(g, 0, xi, A);
  jac_col<DIM>(g, 1, xi, B);
  jac_col<DIM>(g, 2, xi, C);
  cross2(B, C, Sm[0]);
  cross2(C, A, Sm[1]);
  cross2(A, B, Sm[2]);
  float2 d = mul2(A[0], Sm[0][0]);
  d = fma2(A[1], Sm[0][1], d);
  return fma2(A[2], Sm[0][2], d);
}
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(1.f / a.x, 1.f / a.y); }

// Multiplier max(|v|, gamma) and the sharpening factor gamma u (1 - u) / max(|q|, delta)
// for a pair: v2 = |v|^2, g2 = |q|^2.
__device__ __forceinline__ float2 flux_mult(float2 v2, float gamma) {
  return make_float2(fmaxf(sqrtf(v2.x), gamma), fmaxf(sqrtf(v2.y), gamma));
}
__device__ __forceinline__ float2 sharp2(float2 u, float2 g2, float gamma, float rdelta) {
  const float2 r = make_float2(fminf(rsqrtf(g2.x), rdelta), fminf(rsqrtf(g2.y), rdelta));
  const float2 w = mul2(u, sub2(dup2(1.f), u));
  return mul2(mul2(dup2(gamma), w), r);
}

// Velocity factors of the elements whose map is affine with a diagonal
// Jacobian (record flag 2) under a separable velocity field: per axis b and
// coordinate j (the N solution coordinates, then the ends -1 and +1) a pair
// (A, B) such that v_c = vs[c] g prod_b (b == c ? A : B)_b(j_b).  Evaluated once
// in double; the residual kernel read sines per element and stage before
// (40 instructions a lane).
template <int DIM, int N>
__global__ void k_vel_tab(const KArgs A) {
  constexpr int NT = N + 2, NC = DIM == 2 ? 4 : 8;
  const int64_t n = A.E * DIM * NT;
  float2* out = const_cast<float2*>(A.vtab);
  const int kind = A.cd.vel.kind;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < n; g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = g / (DIM * NT);
    const int r = (int)(g % (DIM * NT)), b = r / NT, j = r % NT;
    const double* k = A.geo + (e * DIM + b) * NC;
    const double xi = j < N ? A.cd.ops.x[j] : (j == N ? -1.0 : 1.0);
    const double x = k[0] + k[1 + b] * xi;
    double a = 1.0, f = 1.0;
    if (kind == 2 && DIM == 2) {  // LeVeque's field is a 3D one: zero in 2D, as in velocity()
      a = f = 0.0;
    } else if (kind == 1 || kind == 2) {  // Rider-Kothe (in 3D constant along axis 2), LeVeque
      if (kind == 2 || b < 2) {
        double s, c;
        sincospi(x, &s, &c);
        a = s * s;
        f = 2.0 * s * c;
      }
    } else if (kind == 4) {  // rotation: v_0 = a_1 - x_1, v_1 = x_0 - a_0
      if (b == 0) f = x - A.cd.vel.a[0];
      if (b == 1) f = A.cd.vel.a[1] - x;
    }
    out[g] = make_float2((float)a, (float)f);
  }
}

// ---- residual kernel ----------------------------------------------------------
// GEN false: every element of the mesh is axis-aligned and affine (record flag
// 2), so only that path is compiled; true: each element takes that path or the
// general one (metric from the map's coefficients) by its own flag, so that an
// element's result does not depend on what else is in the mesh.  Axis-aligned
// elements take the velocity from the factor table where the field has one
// (TAB; with GEN known at run time), the others from the point cache.
template <int DIM, int N, bool GEN, bool TAB>
struct KBLine {
  using L = LL<DIM, N>;
  static constexpr int WARP_F = (2 * (1 + DIM) * L::AS) * L::EPW;  // floats a warp
  static constexpr int IN_F = L::DIRECT ? 0 : ((L::EPW * 2 * L::NU + 3) / 4) * 4;
  // read in the middle of the tile, copied in at its start: the velocity table
  // and, on the general path, the point velocities and the map coefficients
  static constexpr bool PTS = GEN || !TAB;  // point velocities may be read
  static constexpr int TAB_F = GEN || TAB ? (L::EPW * DIM * (N + 2) * 2 + 3) / 4 * 4 : 0;
  static constexpr int VF_F = PTS ? (L::EPW * DIM * L::NF + 3) / 4 * 4 : 0;
  static constexpr int VU_F = PTS ? (L::EPW * DIM * L::NU + 3) / 4 * 4 : 0;
  static constexpr int GEO_F = GEN ? L::EPW * L::S::NG : 0;
  static constexpr int O_IN = (WARP_F + 3) / 4 * 4, O_TAB = O_IN + IN_F, O_VF = O_TAB + TAB_F, O_VU = O_VF + VF_F,
                       O_GEO = O_VU + VU_F;
  static constexpr int F = O_GEO + GEO_F;
  static_assert(O_IN % 4 == 0 && O_TAB % 4 == 0 && O_VF % 4 == 0 && O_VU % 4 == 0 && O_GEO % 4 == 0 && F % 4 == 0,
                "16-byte boundaries");
};

// NPHI: the interface normal comes from phi (the unpreconditioned method).
template <int DIM, int N, bool GEN, bool TAB, bool NPHI, int WPB>
__global__ void __launch_bounds__(WPB * 32, (GEN || (DIM == 3 && N == 5) ? 16 : 20) / WPB) kb_line(const KArgs A) {
  using L = LL<DIM, N>;
  using K = KBLine<DIM, N, GEN, TAB>;
  constexpr int NU = L::NU, NF = L::NF, NFP = L::NFP, LN = L::LN, EPW = L::EPW, NP = L::NP, AS = L::AS;
  constexpr int NT = N + 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* wsm = reinterpret_cast<float*>(smem_raw) + warp * K::F;
  const int es = L::FULL ? lane / LN : min(lane / LN, EPW - 1), l = lane - (lane / LN) * LN;
  const bool lane_ok = L::FULL || lane < EPW * LN;
  const int64_t e0 = ((int64_t)blockIdx.x * WPB + warp) * EPW;
  const int64_t eraw = e0 + es;
  const bool act = lane_ok && eraw < A.E;
  const int64_t e = eraw < A.E ? eraw : A.E - 1;
  float* fcE = reinterpret_cast<float*>(A.fc) + e * 2 * NF;
  const float* trA = reinterpret_cast<const float*>(A.tr);
  const LineOps& O = A.lo;
  const PrmT<float>& P = A.cf.prm;

  const int ne = (int)max((int64_t)0, min((int64_t)EPW, A.E - e0));
  float2 u[2][NP];
  float2 o[DIM][2];
  auto load_state = [&]() {
    pdl_wait();
    pdl_launch();
    if constexpr (L::DIRECT) {
#pragma unroll
      for (int f = 0; f < 2; ++f)
        grow_get<N>(reinterpret_cast<const float*>(A.ustg) + (e * 2 + f) * NU + l * N, u[f]);
    } else {
      tile_fetch<EPW, 2 * NU * 4>(wsm + K::O_IN, reinterpret_cast<const float*>(A.ustg) + e0 * 2 * NU, ne, lane);
      cp_async_commit();
    }
  };
  if constexpr (!kEarly<DIM, N, GEN>) load_state();
  // ---- loads that no kernel of the march writes: connectivity, mid-tile data, metric
  int fl[DIM][2];
  [[maybe_unused]] int2 fw[DIM][2];     // hexes: face words
  [[maybe_unused]] int32_t w2[DIM][2];  // quads: connectivity words
#pragma unroll
  for (int a = 0; a < DIM; ++a)
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if constexpr (DIM == 3) fw[a][s] = __ldg(A.ffw + e * 6 + 2 * a + s);
      else w2[a][s] = __ldg(A.fnbr + e * NF + (2 * a + s) * NFP + l);
    }
  if (GEN ? A.vtab != nullptr : TAB) tile_fetch<EPW, DIM * NT * 8>(wsm + K::O_TAB, A.vtab + e0 * DIM * NT, ne, lane);
  if constexpr (K::PTS) {
    tile_fetch<EPW, DIM * NF * 4>(wsm + K::O_VF, reinterpret_cast<const float*>(A.vsf) + e0 * DIM * NF, ne, lane);
    tile_fetch<EPW, DIM * NU * 4>(wsm + K::O_VU, reinterpret_cast<const float*>(A.vsu) + e0 * DIM * NU, ne, lane);
  }
  if constexpr (GEN) tile_fetch<EPW, L::S::NG * 4>(wsm + K::O_GEO, A.geof + e0 * L::S::NG, ne, lane);
  const float* mc = reinterpret_cast<const float*>(A.mcg) + e * kMetricRec;
  const bool diag = !GEN || __ldg(mc + 11) == 2.f;
  const bool tab = GEN ? diag && A.vtab != nullptr : TAB;
  float sd[DIM];  // S_aa of the diagonal metric
#pragma unroll
  for (int a = 0; a < DIM; ++a) sd[a] = __ldg(mc + a * 4);
  const float rdet = __ldg(mc + 10);
  if constexpr (kEarly<DIM, N, GEN>) load_state();
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    float t[2][2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int k = (2 * a + s) * NFP + l;
      if constexpr (DIM == 3) {
        const int32_t po = face_link<N, NF>(A, fw[a][s], e, 2 * a + s, l % N, l / N, fl[a][s]);
        const bool nb = (fl[a][s] & (kFwL | kFwWall)) == kFwL;
        t[0][s] = nb ? trA[po] : 0.f;
        t[1][s] = nb ? trA[po + NF] : 0.f;
      } else {
        t[0][s] = trA[e * 2 * NF + k];
        t[1][s] = trA[e * 2 * NF + NF + k];
        fl[a][s] = (w2[a][s] & 1) | ((w2[a][s] >> 1) == (int32_t)(e * NF + k) ? kFwWall : 0);
      }
    }
    o[a][0] = make_float2(t[0][0], t[0][1]);
    o[a][1] = make_float2(t[1][0], t[1][1]);
  }

  // time factor and eps (of the element in a batch), evaluated by every warp for
  // itself: three FP64 instructions a warp cost less than a block barrier
  // behind one thread's evaluation
  float gfac, eps;
  if (A.ep) {
    gfac = time_factor_t<float>(A, A.ep[e].t + rk_c(A.stage) * A.ep[e].dt);
    eps = (float)A.ep[e].eps;
  } else {
    gfac = time_factor_t<float>(A, A.use_dev_time ? A.dstate[DS_TIME] + rk_c(A.stage) * A.dt : A.t);
    eps = P.eps;
  }
  if constexpr (!L::DIRECT) {
    cp_async_wait_all();
    __syncwarp();
    const float* in = wsm + K::O_IN;
#pragma unroll
    for (int f = 0; f < 2; ++f) grow_get<N>(in + (es * 2 + f) * NU + l * N, u[f]);
  }

  float* U = wsm + es * AS;               // [f]: + f * AS * EPW
  float* Q = wsm + (2 * EPW + es) * AS;   // [f][a]: + (f * DIM + a) * AS * EPW
  constexpr int FA = AS * EPW;            // stride between arrays

  // ---- Steps 1-3 -------------------------------------------------------------
  float2 tr[DIM][2];     // own traces at the line's ends
  float2 q[2][DIM][NP];  // gradient at the lane's points (reference, then physical)
  float2 qe[DIM][2];     // axis-a gradient of both fields at the ends of the axis-a line (diagonal metric)
  float sc[DIM];         // diagonal metric: S_aa / det J
  if (diag) {
#pragma unroll
    for (int a = 0; a < DIM; ++a) sc[a] = __fmul_rn(sd[a], rdet);
  } else {
#pragma unroll
    for (int a = 0; a < DIM; ++a) sc[a] = 1.f;
  }
  if (lane_ok) {
#pragma unroll
    for (int f = 0; f < 2; ++f) row_put<NP, L::V4>(U + f * FA + pline<DIM, N>(0, l), u[f]);
  }
  __syncwarp();
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      float v[N];
      if (a == 0) unpair<N>(u[f], v);
      else if (a == 1) line_get<N, pstride<DIM, N>(1)>(U + f * FA + pline<DIM, N>(1, l), v);
      else line_get<N, pstride<DIM, N>(2)>(U + f * FA + pline<DIM, N>(2, l), v);
      const float2 t = line_ends<N>(O, v);
      tr[a][f] = t;
      // C = u_R on both sides: the jump is the partner's minus the own trace at L ends
      float2 ot = o[a][f];
      ot.x = (fl[a][0] & (kFwL | kFwWall)) == kFwL ? ot.x : t.x;
      ot.y = (fl[a][1] & (kFwL | kFwWall)) == kFwL ? ot.y : t.y;
      o[a][f] = ot;
      float2 d[NP];
      line_deriv<N>(O, v, O.gL, O.gR, sub2(ot, t), d);
#pragma unroll
      for (int p = 0; p < NP; ++p) d[p] = mul2(d[p], dup2(sc[a]));
      {
        float s[N];
        unpair<N>(d, s);
        qe[a][f] = line_ends<N>(O, s);
      }
      if (a == 0) {
#pragma unroll
        for (int p = 0; p < NP; ++p) q[f][0][p] = d[p];
      } else if (lane_ok) {
        float* dst = Q + (f * DIM + a) * FA + pline<DIM, N>(a, l);
        if (a == 1) line_put<N, pstride<DIM, N>(1)>(dst, d);
        else line_put<N, pstride<DIM, N>(2)>(dst, d);
      }
    }
  }
  // the other fields' faces need the axis-0 component of the field that gives the normal
  constexpr int kn = NPHI ? 0 : 1;
  if (lane_ok && diag) row_put<NP, L::V4>(Q + (kn * DIM) * FA + pline<DIM, N>(0, l), q[kn][0]);
  if constexpr (L::DIRECT) cp_async_wait_all();  // the mid-tile data
  __syncwarp();
#pragma unroll
  for (int f = 0; f < 2; ++f)
#pragma unroll
    for (int a = 1; a < DIM; ++a) row_get<NP, L::V4>(Q + (f * DIM + a) * FA + pline<DIM, N>(0, l), q[f][a]);

  int lc[3];  // the lane's point coordinates on axes 1, 2
  lc[1] = DIM == 3 ? l % N : l;
  lc[2] = DIM == 3 ? l / N : 0;
  const float* geo = wsm + K::O_GEO + es * L::S::NG;
  if (GEN && !diag) {
    // physical gradient q_b = sum_a S[a][b] q~_a / det J, kept in registers and in the rows
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      float2 xi[3], Sm[3][3];
      xi[0] = O.xp[p];
#pragma unroll
      for (int b = 1; b < DIM; ++b) xi[b] = dup2(A.cf.ops.x[lc[b]]);
      const float2 rdj = rcp2(metric_all<DIM>(geo, xi, Sm));
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        float2 r[3];
#pragma unroll
        for (int b = 0; b < DIM; ++b) {
          r[b] = mul2(Sm[0][b], q[f][0][p]);
#pragma unroll
          for (int a = 1; a < DIM; ++a) r[b] = fma2(Sm[a][b], q[f][a][p], r[b]);
          r[b] = mul2(r[b], rdj);
        }
#pragma unroll
        for (int b = 0; b < DIM; ++b) q[f][b][p] = r[b];
      }
    }
    if (lane_ok) {
#pragma unroll
      for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int b = 0; b < DIM; ++b) row_put<NP, L::V4>(Q + (f * DIM + b) * FA + pline<DIM, N>(0, l), q[f][b]);
    }
  }
  if (GEN) __syncwarp();

  // ---- Step 5: the common flux at both ends of the lane's line of every axis ---
  const float2* vt = reinterpret_cast<const float2*>(wsm + K::O_TAB) + es * DIM * NT;  // (A, B) per axis and coordinate
  const float gv = P.vel_g ? gfac : 1.f;
  float2 cor[DIM][2];
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    float2 Fp, Fs;
    const float2 pL = tr[a][0], sL = tr[a][1], pR = o[a][0], sR = o[a][1];
    const float2 dp = sub2(pL, pR), ds = sub2(sL, sR);
    const float2 ap = mul2(dup2(0.5f), add2(pL, pR)), as = mul2(dup2(0.5f), add2(sL, sR));
    if (diag) {
      // the transformed normal is -+S_aa e_a: q along axis a of both fields,
      // and the whole gradient of the field that gives the normal
      const float2 qn = qe[a][kn];
      float2 g2 = mul2(qn, qn);
#pragma unroll
      for (int b = 0; b < DIM; ++b) {
        if (b == a) continue;
        float v[N];
        if (a == 0) unpair<N>(q[kn][b], v);
        else if (a == 1) line_get<N, pstride<DIM, N>(1)>(Q + (kn * DIM + b) * FA + pline<DIM, N>(1, l), v);
        else line_get<N, pstride<DIM, N>(2)>(Q + (kn * DIM + b) * FA + pline<DIM, N>(2, l), v);
        const float2 t = line_ends<N>(O, v);
        g2 = fma2(t, t, g2);
      }
      float2 va, v2;
      if (tab) {
        // velocity factors: v_c = s_c g prod_b (b == c ? A : B)_b
        float kc[DIM];
        const int j1 = l % N, j2 = l / N;  // the line's coordinates on the two other axes, lowest first
#pragma unroll
        for (int c = 0; c < DIM; ++c) kc[c] = P.vs[c] * gv;
        {
          int i = 0;
#pragma unroll
          for (int b = 0; b < DIM; ++b) {
            if (b == a) continue;
            const float2 ab = vt[b * NT + (i == 0 ? (DIM == 2 ? l : j1) : j2)];
            ++i;
#pragma unroll
            for (int c = 0; c < DIM; ++c) kc[c] = __fmul_rn(kc[c], c == b ? ab.x : ab.y);
          }
        }
        const float2 e0v = vt[a * NT + N], e1v = vt[a * NT + N + 1];
        const float2 Ae = make_float2(e0v.x, e1v.x), Be = make_float2(e0v.y, e1v.y);
        float ko = 0.f;  // sum of the other components' squares
#pragma unroll
        for (int c = 0; c < DIM; ++c)
          if (c != a) ko = __fmaf_rn(kc[c], kc[c], ko);
        va = mul2(Ae, dup2(kc[a]));
        v2 = fma2(va, va, mul2(mul2(Be, Be), dup2(ko)));
      } else {
        const float* vf = wsm + K::O_VF + es * DIM * NF + 2 * a * NFP + l;
        v2 = dup2(0.f);
#pragma unroll
        for (int c = 0; c < DIM; ++c) {
          const float2 v = mul2(dup2(gfac), make_float2(vf[c * NF], vf[c * NF + NFP]));
          if (c == a) va = v;
          v2 = fma2(v, v, v2);
        }
      }
      const float2 M = flux_mult(v2, P.gamma);
      const float2 sh = sharp2(pL, g2, P.gamma, P.rdelta);
      const float2 nvis = fma2(sh, qn, mul2(dup2(-eps), qe[a][0]));  // minus the viscous flux over M
      const float saa = sd[a], pm = fabsf(saa);
      const float2 sg = make_float2(-saa, saa);
      Fp = fma2(dup2(__fmul_rn(pm, P.tau)), dp, mul2(sg, fma2(ap, va, mul2(M, nvis))));
      Fs = fma2(dup2(__fmul_rn(pm, P.tau_psi)), ds, mul2(sg, mul2(as, va)));
    } else if (GEN) {
      float2 qf[2][DIM];
#pragma unroll
      for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int b = 0; b < DIM; ++b) {
          float v[N];
          if (a == 0) unpair<N>(q[f][b], v);
          else if (a == 1) line_get<N, pstride<DIM, N>(1)>(Q + (f * DIM + b) * FA + pline<DIM, N>(1, l), v);
          else line_get<N, pstride<DIM, N>(2)>(Q + (f * DIM + b) * FA + pline<DIM, N>(2, l), v);
          qf[f][b] = line_ends<N>(O, v);
        }
      float2 xi[3], Sr[3];
      {
        int i = 0;
#pragma unroll
        for (int b = 0; b < DIM; ++b) {
          if (b == a) {
            xi[b] = make_float2(-1.f, 1.f);
          } else {
            xi[b] = dup2(A.cf.ops.x[i == 0 ? (DIM == 2 ? l : l % N) : l / N]);
            ++i;
          }
        }
      }
      metric_row<DIM>(geo, a, xi, Sr);
      const float2 sgn = make_float2(-1.f, 1.f);
      const float* vf = wsm + K::O_VF + es * DIM * NF + 2 * a * NFP + l;
      float2 vn = dup2(0.f), v2 = dup2(0.f), g2 = dup2(0.f), pm2 = dup2(0.f), qp = dup2(0.f), qs = dup2(0.f);
#pragma unroll
      for (int c = 0; c < DIM; ++c) {
        const float2 v = mul2(dup2(gfac), make_float2(vf[c * NF], vf[c * NF + NFP]));
        const float2 pn = mul2(sgn, Sr[c]);
        const float2 qn = qf[kn][c];
        vn = fma2(v, pn, vn);
        v2 = fma2(v, v, v2);
        pm2 = fma2(pn, pn, pm2);
        g2 = fma2(qn, qn, g2);
        qp = fma2(qf[0][c], pn, qp);
        qs = fma2(qn, pn, qs);
      }
      const float2 pm = make_float2(sqrtf(pm2.x), sqrtf(pm2.y));
      const float2 M = flux_mult(v2, P.gamma);
      const float2 sh = sharp2(pL, g2, P.gamma, P.rdelta);
      const float2 nvis = fma2(sh, qs, mul2(dup2(-eps), qp));
      Fp = fma2(mul2(pm, dup2(P.tau)), dp, fma2(ap, vn, mul2(M, nvis)));
      Fs = fma2(mul2(pm, dup2(P.tau_psi)), ds, mul2(as, vn));
    }
    // R ends carry no flux here (ka lifts minus the partner's); no-flux walls none at all
    const bool l0 = fl[a][0] & kFwL, l1 = fl[a][1] & kFwL;
    const bool z0 = !l0 || (P.noflux && (fl[a][0] & kFwWall)), z1 = !l1 || (P.noflux && (fl[a][1] & kFwWall));
    Fp = make_float2(z0 ? 0.f : Fp.x, z1 ? 0.f : Fp.y);
    Fs = make_float2(z0 ? 0.f : Fs.x, z1 ? 0.f : Fs.y);
    cor[a][0] = Fp;
    cor[a][1] = Fs;
    if (act) {
      const int k0 = 2 * a * NFP + l;
      if (l0) {
        fcE[k0] = Fp.x;
        fcE[k0 + NF] = Fs.x;
      }
      if (l1) {
        fcE[k0 + NFP] = Fp.y;
        fcE[k0 + NFP + NF] = Fs.y;
      }
      if constexpr (FaceScatter<DIM>::v) {
        // quads: the common flux also goes to the R-side partner's slot
#pragma unroll
        for (int sd = 0; sd < 2; ++sd)
          if ((fl[a][sd] & (kFwL | kFwWall)) == kFwL) {
            const int32_t pg = partner<NF>(A, w2[a][sd], (int32_t)(e * NF + k0 + sd * NFP));
            float* d = reinterpret_cast<float*>(A.fc) + (int64_t)(pg / NF) * 2 * NF + pg % NF;
            d[0] = sd ? Fp.y : Fp.x;
            d[NF] = sd ? Fs.y : Fs.x;
          }
      }
    }
  }
  __syncwarp();  // the faces have read the gradient rows

  // ---- Step 4: the transformed flux at the lane's points; axis 0 stays in registers
  float2 fx[2][NP];
  {
    float2 k[DIM];  // diagonal metric: velocity factors of the line
    float ko = 0.f;
    if (tab) {
      float kc[DIM];
#pragma unroll
      for (int c = 0; c < DIM; ++c) kc[c] = P.vs[c] * gv;
#pragma unroll
      for (int b = 1; b < DIM; ++b) {
        const float2 ab = vt[b * NT + lc[b]];
#pragma unroll
        for (int c = 0; c < DIM; ++c) kc[c] = __fmul_rn(kc[c], c == b ? ab.x : ab.y);
      }
#pragma unroll
      for (int c = 0; c < DIM; ++c) k[c] = dup2(kc[c]);
#pragma unroll
      for (int c = 1; c < DIM; ++c) ko = __fmaf_rn(kc[c], kc[c], ko);
    }
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      float2 v[DIM], v2, Sm[3][3];
      if (tab) {
        const float2 t0 = vt[2 * p], t1 = 2 * p + 1 < N ? vt[2 * p + 1] : make_float2(0.f, 0.f);
        const float2 Ax = make_float2(t0.x, t1.x), Bx = make_float2(t0.y, t1.y);
        v[0] = mul2(Ax, k[0]);
#pragma unroll
        for (int c = 1; c < DIM; ++c) v[c] = mul2(Bx, k[c]);
        v2 = fma2(v[0], v[0], mul2(mul2(Bx, Bx), dup2(ko)));
      } else {
        const float* vc = wsm + K::O_VU + es * DIM * NU + l * N + 2 * p;
        v2 = dup2(0.f);
#pragma unroll
        for (int c = 0; c < DIM; ++c) {
          v[c] = mul2(dup2(gfac), make_float2(vc[c * NU], 2 * p + 1 < N ? vc[c * NU + 1] : 0.f));
          v2 = fma2(v[c], v[c], v2);
        }
      }
      if (GEN && !diag) {
        float2 xi[3];
        xi[0] = O.xp[p];
#pragma unroll
        for (int b = 1; b < DIM; ++b) xi[b] = dup2(A.cf.ops.x[lc[b]]);
        metric_all<DIM>(geo, xi, Sm);
      }
      float2 qs[DIM], g2 = dup2(0.f);
#pragma unroll
      for (int c = 0; c < DIM; ++c) {
        qs[c] = q[kn][c][p];
        g2 = fma2(qs[c], qs[c], g2);
      }
      const float2 M = flux_mult(v2, P.gamma);
      const float2 sh = sharp2(u[0][p], g2, P.gamma, P.rdelta);
      float2 f0[DIM], f1[DIM];
#pragma unroll
      for (int c = 0; c < DIM; ++c) {
        const float2 t = fma2(sh, qs[c], mul2(dup2(-eps), q[0][c][p]));
        // the larger term in the last multiply-add: one rounding of its size (added first, phi's rate was
        // 4 % further from FP64 on regular hexes)
        f0[c] = fma2(u[0][p], v[c], mul2(M, t));
        f1[c] = mul2(u[1][p], v[c]);
      }
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        float2 t0, t1;
        if (diag) {
          const float2 s = dup2(sd[a]);
          t0 = mul2(s, f0[a]);
          t1 = mul2(s, f1[a]);
        } else {
          t0 = mul2(Sm[a][0], f0[0]);
          t1 = mul2(Sm[a][0], f1[0]);
#pragma unroll
          for (int c = 1; c < DIM; ++c) {
            t0 = fma2(Sm[a][c], f0[c], t0);
            t1 = fma2(Sm[a][c], f1[c], t1);
          }
        }
        if (a == 0) {
          fx[0][p] = t0;
          fx[1][p] = t1;
        } else {  // the gradient's registers carry the flux from here on
          q[0][a][p] = t0;
          q[1][a][p] = t1;
        }
      }
    }
  }
  if (lane_ok) {
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
      for (int a = 1; a < DIM; ++a) row_put<NP, L::V4>(Q + (f * DIM + a) * FA + pline<DIM, N>(0, l), q[f][a]);
  }
  __syncwarp();

  // ---- Step 6 -------------------------------------------------------------------
  float2 dv[2][NP];
#pragma unroll
  for (int a = 0; a < DIM; ++a)
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      float v[N];
      float* src = Q + (f * DIM + a) * FA + pline<DIM, N>(a, l);
      if (a == 0) unpair<N>(fx[f], v);
      else if (a == 1) line_get<N, pstride<DIM, N>(1)>(src, v);
      else line_get<N, pstride<DIM, N>(2)>(src, v);
      const float2 fp = line_ends<N>(O, v);
      // F~ - f~perp with f~perp = -+ f~_a at the two ends
      const float2 c = fma2(fp, make_float2(1.f, -1.f), cor[a][f]);
      float2 d[NP];
      line_deriv<N>(O, v, O.ngL, O.gR, c, d);
      if (a == 0) {
#pragma unroll
        for (int p = 0; p < NP; ++p) dv[f][p] = d[p];
      } else if (lane_ok) {
        if (a == 1) line_put<N, pstride<DIM, N>(1)>(src, d);
        else line_put<N, pstride<DIM, N>(2)>(src, d);
      }
    }
  __syncwarp();
  float* rp = reinterpret_cast<float*>(A.rp);
#pragma unroll
  for (int f = 0; f < 2; ++f) {
#pragma unroll
    for (int a = 1; a < DIM; ++a) {
      float2 t[NP];
      row_get<NP, L::V4>(Q + (f * DIM + a) * FA + pline<DIM, N>(0, l), t);
#pragma unroll
      for (int p = 0; p < NP; ++p) dv[f][p] = add2(dv[f][p], t[p]);
    }
    if constexpr (L::DIRECT) {
      if (act) grow_put<N>(rp + (e * 2 + f) * NU + l * N, dv[f]);
    } else if (lane_ok) {
      grow_put<N>(wsm + K::O_IN + (es * 2 + f) * NU + l * N, dv[f]);
    }
  }
  if constexpr (!L::DIRECT) {
    __syncwarp();
    if (ne > 0) warp_flush(rp + e0 * 2 * NU, wsm + K::O_IN, ne * 2 * NU, lane);
  }
}

// ---- update kernel -------------------------------------------------------------
// R-side lift, RK4 update and next-stage traces (ka_tensor's work), one line a
// lane.  SF: the RK stage 1..4, or 0 to recompute the traces of ustg alone.
// GEN false: every element is affine (1 / det J from the record).
template <int DIM, int N, int SF, bool GEN>
struct KALine {
  using L = LL<DIM, N>;
  // rows of both fields; face corrections of the axes > 0: [axis][end][field][other][row]
  static constexpr int ROWS_F = 2 * L::AS * L::EPW;
  static constexpr int COR_F = (DIM - 1) * 2 * 2 * L::OTH * L::RS * L::EPW;
  // input and output buffer of the strided forms: rp (later the stage value), u, acc, w det J
  static constexpr int C = L::EPW * L::NU;
  static constexpr int O_U = (2 * C + 3) / 4 * 4, O_A = (O_U + 4 * C + 3) / 4 * 4;  // 16-byte boundaries
  static constexpr int IN_F = L::DIRECT ? 0 : SF == 0 ? O_U : (O_A + 2 * C + 3) / 4 * 4;
  static constexpr int O_IN = (ROWS_F + 3) / 4 * 4 + (SF >= 1 ? (COR_F + 3) / 4 * 4 : 0);
  // stage 4: w det J pairs; general path: the map coefficients
  static constexpr int O_W = O_IN + IN_F, O_GEO = O_W + (SF == 4 ? (2 * C + 3) / 4 * 4 : 0);
  static constexpr int F = O_GEO + (SF >= 1 && GEN ? L::EPW * L::S::NG : 0);
  static_assert(O_IN % 4 == 0 && O_U % 4 == 0 && O_A % 4 == 0 && O_W % 4 == 0 && O_GEO % 4 == 0 && F % 4 == 0,
                "16-byte boundaries");
};

// (hi, lo) += f: error-free sum of the high parts, the errors beside
__device__ __forceinline__ void sum_add(float2& hi, float2& lo, float2 f) {
  const float2 s = add2(hi, f);
  const float2 bb = sub2(s, hi);
  lo = add2(lo, add2(sub2(hi, sub2(s, bb)), sub2(f, bb)));
  hi = s;
}
// (hi, lo) += w f with w = wh + wl: error-free product and sum of the high parts
__device__ __forceinline__ void dot_add(float2& hi, float2& lo, float2 wh, float2 wl, float2 f) {
  const float2 p = mul2(wh, f);
  lo = add2(lo, fma2(wl, f, fma2(wh, f, make_float2(-p.x, -p.y))));
  sum_add(hi, lo, p);
}
// product of two float-float values
__device__ __forceinline__ float2 ff_mul2(float2 a, float2 b) {
  const float p = a.x * b.x;
  const float e = __fmaf_rn(a.x, b.x, -p) + __fmaf_rn(a.x, b.y, a.y * b.x);
  const float hi = p + e;
  return make_float2(hi, e - (hi - p));
}
// Sums of the LN lanes' float-float values a, b (of the two fields) of an
// element, in a fixed tree; lane 0 gets a's sum, lane `lb` b's.  With a power
// of two of lanes the first step leaves a in the lower and b in the upper
// half, so that both trees share the later steps.
template <int LN>
struct LineTree {
  static constexpr bool SPLIT = (LN & (LN - 1)) == 0;
  static constexpr int LB = SPLIT ? LN / 2 : 0;
};
__device__ __forceinline__ float2 shfl_down2(float2 v, int o) {
  return make_float2(__shfl_down_sync(0xffffffffu, v.x, o), __shfl_down_sync(0xffffffffu, v.y, o));
}
template <int LN>
__device__ __forceinline__ void line_tree(float2& a, float2& b, int l) {
  if constexpr (LineTree<LN>::SPLIT) {
    const bool up = l >= LN / 2;
    const float2 give = up ? a : b, keep = up ? b : a;
    float2 got;
    got.x = __shfl_xor_sync(0xffffffffu, give.x, LN / 2);
    got.y = __shfl_xor_sync(0xffffffffu, give.y, LN / 2);
    // the lower lane's value first in both halves' sums
    float2 v = up ? ff_add(got, keep) : ff_add(keep, got);
#pragma unroll
    for (int o = LN / 4; o > 0; o >>= 1) v = ff_add(v, shfl_down2(v, o));
    a = b = v;
  } else {
    constexpr int TOP = LN > 16 ? 16 : LN > 8 ? 8 : LN > 4 ? 4 : LN > 2 ? 2 : 1;
#pragma unroll
    for (int o = TOP; o > 0; o >>= 1) {
      const float2 s = shfl_down2(a, o), t = shfl_down2(b, o);
      if (l + o < LN) {
        a = ff_add(a, s);
        b = ff_add(b, t);
      }
    }
  }
}

template <int DIM, int N, bool GEN, int WPB, int SF>
__global__ void __launch_bounds__(WPB * 32, (DIM == 3 ? 24 : 20) / WPB) ka_line(const KArgs A) {
  using L = LL<DIM, N>;
  using K = KALine<DIM, N, SF, GEN>;
  constexpr int NU = L::NU, NF = L::NF, NFP = L::NFP, LN = L::LN, EPW = L::EPW, NP = L::NP, AS = L::AS;
  constexpr int NEL = WPB * EPW;  // at most 16 elements a warp: one thread an element and field
  static_assert(2 * NEL <= WPB * 32, "the block's threads finish the elements' balances");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ float2 balS[SF >= 1 ? 2 * NEL : 1];  // element flux balances
  __shared__ float2 incS[SF == 4 ? 2 * NEL : 1];  // stage 4: element sums of w det J * increment
  __shared__ float2 dltS[SF == 4 ? 2 * NEL : 1];  // stage 4: the elements' uniform shifts
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* wsm = reinterpret_cast<float*>(smem_raw) + warp * K::F;
  float* R0 = wsm;                                   // rows [f][es]
  float* C0 = wsm + (K::ROWS_F + 3) / 4 * 4;         // face corrections
  float* in = C0 + (SF >= 1 ? (K::COR_F + 3) / 4 * 4 : 0);
  const int es = L::FULL ? lane / LN : min(lane / LN, EPW - 1), l = lane - (lane / LN) * LN;
  const bool lane_ok = L::FULL || lane < EPW * LN;
  const int64_t e0 = ((int64_t)blockIdx.x * WPB + warp) * EPW;
  const int64_t eraw = e0 + es;
  const bool act = lane_ok && eraw < A.E;
  const int64_t e = eraw < A.E ? eraw : A.E - 1;
  const int ne = (int)max((int64_t)0, min((int64_t)EPW, A.E - e0));
  const float* fcA = reinterpret_cast<const float*>(A.fc);
  float* ustg = reinterpret_cast<float*>(A.ustg);
  float* acc = reinterpret_cast<float*>(A.acc);
  float2* U = reinterpret_cast<float2*>(A.u);
  const LineOps& O = A.lo;
  const bool cons = SF >= 1 && A.tacc != nullptr;

  // ---- loads ------------------------------------------------------------------
  float2 y[2][NP];       // partial divergence, then the stage value
  float2 u[2][N];        // solution pairs (hi, lo)
  float ac[2][N];        // RK accumulator
  float aff = 1.f, rdet = 0.f;  // record: affine flag, 1 / det J
  [[maybe_unused]] RKConstF rk;
  double ta = 0.0;  // this thread's element balance so far (finished by the first threads of the block)
  const int64_t gt = (int64_t)blockIdx.x * NEL * 2 + threadIdx.x;
  float2 rW = make_float2(0.f, 0.f);  // stage 4: 1 / W
  // what the march writes: the rate, the solution, the accumulator and the flux
  // balances, all after pdl_wait
  auto load_state = [&]() {
    pdl_wait();
    pdl_launch();
    const float* src = SF == 0 ? ustg : reinterpret_cast<const float*>(A.rp);
    if constexpr (L::DIRECT) {
#pragma unroll
      for (int f = 0; f < 2; ++f) grow_get<N>(src + (e * 2 + f) * NU + l * N, y[f]);
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        const int64_t r = (e * 2 + f) * NU + l * N;
        if constexpr (SF >= 1) {
#pragma unroll
          for (int j = 0; j < N; j += 2) {
            const float4 t = *reinterpret_cast<const float4*>(U + r + j);
            u[f][j] = make_float2(t.x, t.y);
            u[f][j + 1] = make_float2(t.z, t.w);
          }
        }
        if constexpr (SF >= 2) {
          float2 t[NP];
          grow_get<N>(acc + r, t);
          unpair<N>(t, ac[f]);
        }
      }
    } else if (ne > 0) {
      tile_fetch<EPW, 2 * NU * 4>(in, src + e0 * 2 * NU, ne, lane);
      if constexpr (SF >= 1) tile_fetch<EPW, 2 * NU * 8>(in + K::O_U, U + e0 * 2 * NU, ne, lane);
      if constexpr (SF >= 2) tile_fetch<EPW, 2 * NU * 4>(in + K::O_A, acc + e0 * 2 * NU, ne, lane);
    }
    if constexpr (SF >= 2)
      if (cons && threadIdx.x < 2 * NEL && gt < 2 * A.E) ta = A.tacc[gt];
  };
  if constexpr (SF >= 1) {
    const float* mc = reinterpret_cast<const float*>(A.mcg) + e * kMetricRec;
    rdet = __ldg(mc + 10);
    if (GEN) aff = DIM == 3 ? __ldg(mc + 11) : 0.f;
    if (SF == 4 && cons && ne > 0) tile_fetch<EPW, NU * 8>(wsm + K::O_W, A.wdetf + e0 * NU, ne, lane);
    if (GEN && ne > 0) tile_fetch<EPW, L::S::NG * 4>(wsm + K::O_GEO, A.geof + e0 * L::S::NG, ne, lane);
    rk = A.ep ? A.ep[e].rk : A.rk;
    if (SF == 4 && cons && threadIdx.x < 2 * NEL && gt < 2 * A.E)
      rW = *reinterpret_cast<const float2*>(reinterpret_cast<const float*>(A.mcg) + (gt / 2) * kMetricRec + 12);
  }
  if constexpr (!kEarly<DIM, N, GEN>) load_state();
  int fl[DIM][2];
  [[maybe_unused]] int2 fw[DIM][2];
  [[maybe_unused]] int32_t w2[DIM][2];
#pragma unroll
  for (int a = 0; a < DIM; ++a)
#pragma unroll
    for (int sd = 0; sd < 2; ++sd) {
      if constexpr (DIM == 3) fw[a][sd] = __ldg(A.ffw + e * 6 + 2 * a + sd);
      else w2[a][sd] = __ldg(A.fnbr + e * NF + (2 * a + sd) * NFP + l);
    }
  if constexpr (kEarly<DIM, N, GEN>) load_state();
  float2 F[DIM][2];  // transformed common flux at the two ends: the own at L ends, the partner's at R ends
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    float t[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
    for (int sd = 0; sd < 2; ++sd) {
      const int k = (2 * a + sd) * NFP + l;
      int32_t at = (int32_t)(e * 2 * NF + k);
      if constexpr (DIM == 3) {
        const int32_t po = face_link<N, NF>(A, fw[a][sd], e, 2 * a + sd, l % N, l / N, fl[a][sd]);
        if (!(fl[a][sd] & kFwL)) at = po;
      } else {
        fl[a][sd] = (w2[a][sd] & 1) | ((w2[a][sd] >> 1) == (int32_t)(e * NF + k) ? kFwWall : 0);
      }
      if constexpr (SF >= 1) {
        t[0][sd] = fcA[at];
        t[1][sd] = fcA[at + NF];
      }
    }
    F[a][0] = make_float2(t[0][0], t[0][1]);
    F[a][1] = make_float2(t[1][0], t[1][1]);
  }
  if constexpr (!L::DIRECT) {
    cp_async_wait_all();
    __syncwarp();
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      const int r = (es * 2 + f) * NU + l * N;
      grow_get<N>(in + r, y[f]);
      if constexpr (SF >= 1)
#pragma unroll
        for (int j = 0; j < N; ++j) u[f][j] = reinterpret_cast<const float2*>(in + K::O_U)[r + j];
      if constexpr (SF >= 2)
#pragma unroll
        for (int j = 0; j < N; ++j) ac[f][j] = in[K::O_A + r + j];
    }
  }

  if constexpr (SF >= 1) {
    // ---- lift of the R-side fluxes (minus the partner's F~); element flux balance
    float2 bh[2], bl[2];
#pragma unroll
    for (int f = 0; f < 2; ++f) bh[f] = bl[f] = dup2(0.f);
    float2 c0[2];
#pragma unroll
    for (int a = 0; a < DIM; ++a)
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        const bool L0 = fl[a][0] & kFwL, L1 = fl[a][1] & kFwL;
        const float2 c = make_float2(L0 ? 0.f : -F[a][f].x, L1 ? 0.f : -F[a][f].y);
        if (cons) {
          const float2 out = make_float2(L0 ? F[a][f].x : c.x, L1 ? F[a][f].y : c.y);
          if (a == 0) bh[f] = out;
          else sum_add(bh[f], bl[f], out);
        }
        if (a == 0) {
          c0[f] = c;
        } else if (lane_ok) {
          // face buffer: position (x, other) of the line
          const int other = DIM == 3 ? l / N : 0, x = DIM == 3 ? l % N : l;
          float* d = C0 + (((((a - 1) * 2) * 2 + f) * EPW + es) * L::OTH + other) * L::RS + x;
          d[0] = c.x;
          d[2 * EPW * L::OTH * L::RS] = c.y;
        }
      }
    if (cons) {
      // both ends, times the face weight (the same for all axes), then the element's lines
      const float2 wf = A.cf.ops.wff[l];
      float2 v[2];
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        v[f] = ff_mul2(wf, ff_add(make_float2(bh[f].x, bl[f].x), make_float2(bh[f].y, bl[f].y)));
        if (!lane_ok) v[f] = make_float2(0.f, 0.f);
      }
      line_tree<LN>(v[0], v[1], l);
      if (lane_ok && l == 0) balS[(warp * EPW + es) * 2] = v[0];
      if (lane_ok && l == LineTree<LN>::LB) balS[(warp * EPW + es) * 2 + 1] = v[1];
    }
    cp_async_wait_all();
    __syncwarp();
    const int lc1 = DIM == 3 ? l % N : l, lc2 = l / N;
    float gl[3], gr[3];
    gl[1] = -A.cf.ops.gLd[lc1];
    gr[1] = A.cf.ops.gRd[lc1];
    if (DIM == 3) {
      gl[2] = -A.cf.ops.gLd[lc2];
      gr[2] = A.cf.ops.gRd[lc2];
    }
    float2 rdj[NP];
    if (GEN) {
      if (DIM == 3 && aff != 0.f) {
#pragma unroll
        for (int p = 0; p < NP; ++p) rdj[p] = dup2(rdet);
      } else {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          float2 xi[3], Sm[3][3];
          xi[0] = O.xp[p];
          xi[1] = dup2(A.cf.ops.x[lc1]);
          xi[2] = dup2(A.cf.ops.x[DIM == 3 ? lc2 : 0]);
          rdj[p] = rcp2(metric_all<DIM>(wsm + K::O_GEO + es * L::S::NG, xi, Sm));
        }
      }
    } else {
#pragma unroll
      for (int p = 0; p < NP; ++p) rdj[p] = dup2(rdet);
    }
    float bad = 0.f;   // becomes NaN when a new value is not finite
    float inc[2][N];   // stage 4: the increments
#pragma unroll
    for (int f = 0; f < 2; ++f) {
#pragma unroll
      for (int p = 0; p < NP; ++p) y[f][p] = fma2(O.ngL[p], dup2(c0[f].x), fma2(O.gR[p], dup2(c0[f].y), y[f][p]));
#pragma unroll
      for (int a = 1; a < DIM; ++a) {
        // the face row of this line: other coordinate z (axis 1) or y (axis 2)
        const int other = DIM == 3 ? (a == 1 ? lc2 : lc1) : 0;
        const float* s = C0 + (((((a - 1) * 2) * 2 + f) * EPW + es) * L::OTH + other) * L::RS;
        float2 r0[NP], r1[NP];
        row_get<NP, L::V4>(s, r0);
        row_get<NP, L::V4>(s + 2 * EPW * L::OTH * L::RS, r1);
#pragma unroll
        for (int p = 0; p < NP; ++p) y[f][p] = fma2(dup2(gl[a]), r0[p], fma2(dup2(gr[a]), r1[p], y[f][p]));
      }
      // du/dt = -div~ f~ / det J and the RK4 register update
      float R[N];
#pragma unroll
      for (int p = 0; p < NP; ++p) y[f][p] = mul2(make_float2(-y[f][p].x, -y[f][p].y), rdj[p]);
      unpair<N>(y[f], R);
      float yn[2 * NP];
#pragma unroll
      for (int j = 0; j < 2 * NP; ++j) yn[j] = 0.f;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const float2 uu = u[f][j];
        if constexpr (SF == 1) {
          ac[f][j] = R[j];
          yn[j] = uu.x + __fmaf_rn(rk.half_dt, R[j], uu.y);
        } else if constexpr (SF == 2 || SF == 3) {
          ac[f][j] = __fmaf_rn(2.f, R[j], ac[f][j]);
          yn[j] = uu.x + __fmaf_rn(SF == 2 ? rk.half_dt : rk.dt, R[j], uu.y);
        } else {
          const float d = rk.dt6 * (ac[f][j] + R[j]);
          const float s2 = uu.x + d;
          const float e2 = two_sum_lo(uu.x, d, s2) + uu.y;
          const float hi = s2 + e2;
          inc[f][j] = d;
          u[f][j] = make_float2(hi, e2 - (hi - s2));
          yn[j] = hi;
        }
        bad = __fmaf_rn(yn[j], 0.f, bad);
      }
#pragma unroll
      for (int p = 0; p < NP; ++p) y[f][p] = make_float2(yn[2 * p], yn[2 * p + 1]);
    }
    if constexpr (SF == 4) {
      if (cons) {
        // element sums of w det J * increment (float-float), the target mass
        // change of the step, and the uniform shift that makes them equal
        float2 wd[2 * NP], v[2];
#pragma unroll
        for (int j = 0; j < 2 * NP; ++j) wd[j] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < N; ++j) wd[j] = reinterpret_cast<const float2*>(wsm + K::O_W)[es * NU + l * N + j];
#pragma unroll
        for (int f = 0; f < 2; ++f) {
          float2 sh = dup2(0.f), sl = dup2(0.f);
#pragma unroll
          for (int p = 0; p < NP; ++p)
            dot_add(sh, sl, make_float2(wd[2 * p].x, wd[2 * p + 1].x), make_float2(wd[2 * p].y, wd[2 * p + 1].y),
                    make_float2(inc[f][2 * p], 2 * p + 1 < N ? inc[f][2 * p + 1] : 0.f));
          v[f] = ff_add(make_float2(sh.x, sl.x), make_float2(sh.y, sl.y));
          if (!lane_ok) v[f] = make_float2(0.f, 0.f);
        }
        line_tree<LN>(v[0], v[1], l);
        if (lane_ok && l == 0) incS[(warp * EPW + es) * 2] = v[0];
        if (lane_ok && l == LineTree<LN>::LB) incS[(warp * EPW + es) * 2 + 1] = v[1];
        __syncthreads();
        if (const int t = threadIdx.x; t < 2 * NEL) {
          const int64_t g = (int64_t)blockIdx.x * NEL * 2 + t;
          if (g < 2 * A.E) {
            const double Te = -((double)balS[t].x + (double)balS[t].y);
            const double tgt = (A.ep ? A.ep[g / 2].rk.ddt6 : A.rk.ddt6) * (ta + Te);
            const double S = (double)incS[t].x + (double)incS[t].y;
            const double d = (tgt - S) * ((double)rW.x + (double)rW.y);
            const float dh = (float)d;
            dltS[t] = make_float2(dh, (float)(d - (double)dh));
          }
        }
        __syncthreads();
#pragma unroll
        for (int f = 0; f < 2; ++f) {
          const float2 dl = dltS[(warp * EPW + es) * 2 + f];
#pragma unroll
          for (int j = 0; j < N; ++j) {
            const float2 uu = u[f][j];
            const float s2 = uu.x + dl.x;
            const float e2 = two_sum_lo(uu.x, dl.x, s2) + (uu.y + dl.y);
            const float hi = s2 + e2;
            u[f][j] = make_float2(hi, e2 - (hi - s2));
            if (j & 1) y[f][j / 2].y = hi;
            else y[f][j / 2].x = hi;
            bad = __fmaf_rn(hi, 0.f, bad);
          }
        }
      }
    }
    if (act && bad != 0.f) atomicExch(&A.status[ST_STATUS], -4);
    // ---- stage value, accumulator (stages 1-3), solution (stage 4)
    if constexpr (L::DIRECT) {
      if (act) {
#pragma unroll
        for (int f = 0; f < 2; ++f) {
          const int64_t r = (e * 2 + f) * NU + l * N;
          grow_put<N>(ustg + r, y[f]);
          if constexpr (SF < 4) {
            float2 t[NP];
#pragma unroll
            for (int p = 0; p < NP; ++p) t[p] = make_float2(ac[f][2 * p], ac[f][2 * p + 1]);
            grow_put<N>(acc + r, t);
          } else {
#pragma unroll
            for (int j = 0; j < N; j += 2)
              *reinterpret_cast<float4*>(U + r + j) = make_float4(u[f][j].x, u[f][j].y, u[f][j + 1].x, u[f][j + 1].y);
          }
        }
      }
    } else {
      // every lane has read its rows of the buffer (they are its own), so they take the results
      if (lane_ok) {
#pragma unroll
        for (int f = 0; f < 2; ++f) {
          const int r = (es * 2 + f) * NU + l * N;
          grow_put<N>(in + r, y[f]);
#pragma unroll
          for (int j = 0; j < N; ++j) {
            if constexpr (SF < 4) in[K::O_A + r + j] = ac[f][j];
            else reinterpret_cast<float2*>(in + K::O_U)[r + j] = u[f][j];
          }
        }
      }
      __syncwarp();
      if (ne > 0) {
        warp_flush(ustg + e0 * 2 * NU, in, ne * 2 * NU, lane);
        if constexpr (SF < 4) warp_flush(acc + e0 * 2 * NU, in + K::O_A, ne * 2 * NU, lane);
        else warp_flush(U + e0 * 2 * NU, in + K::O_U, ne * 4 * NU, lane);
      }
    }
  }

  // ---- flux-point traces of the new stage value (Step 1 of the next stage) ------
  if (lane_ok) {
#pragma unroll
    for (int f = 0; f < 2; ++f) row_put<NP, L::V4>(R0 + (f * EPW + es) * AS + pline<DIM, N>(0, l), y[f]);
  }
  __syncwarp();
  float* tr = reinterpret_cast<float*>(A.tr);
#pragma unroll
  for (int a = 0; a < DIM; ++a)
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      float v[N];
      const float* src = R0 + (f * EPW + es) * AS + pline<DIM, N>(a, l);
      if (a == 0) unpair<N>(y[f], v);
      else if (a == 1) line_get<N, pstride<DIM, N>(1)>(src, v);
      else line_get<N, pstride<DIM, N>(2)>(src, v);
      const float2 t = line_ends<N>(O, v);
      if (!act) continue;
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        const int k = (2 * a + sd) * NFP + l;
        const float val = sd ? t.y : t.x;
        const int w = fl[a][sd];
        if (!(!(w & kFwL) || (w & kFwWall))) continue;  // read by a partner (R ends) or kept (walls)
        if constexpr (FaceScatter<DIM>::v) {
          const int32_t pg = partner<NF>(A, w2[a][sd], (int32_t)(e * NF + k));
          tr[(int64_t)(pg / NF) * 2 * NF + f * NF + pg % NF] = val;
        } else {
          tr[(e * 2 + f) * NF + k] = val;
        }
      }
    }

  if constexpr (SF >= 1 && SF < 4) {
    if (cons) {
      // element mass rates, accumulated with the RK4 weights in FP64 by the block's first threads
      __syncthreads();
      if (const int t = threadIdx.x; t < 2 * NEL) {
        const int64_t g = (int64_t)blockIdx.x * NEL * 2 + t;
        if (g < 2 * A.E) {
          const double Te = -((double)balS[t].x + (double)balS[t].y);
          A.tacc[g] = SF == 1 ? Te : ta + 2.0 * Te;
        }
      }
    }
  }
  if constexpr (SF == 4) {
    if (A.use_dev_time) {
      if (blockIdx.x == 0 && threadIdx.x == 0) A.dstate[DS_TIME] = A.dstate[DS_TIME] + A.dt;
      if (A.ep && act && l == 0) A.ep[e].t += A.ep[e].dt;
    }
  }
}

}  // namespace frp
