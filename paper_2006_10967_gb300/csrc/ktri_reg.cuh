// Thread-per-element kernels of the mixed path on triangles, p <= 4: the Steps
// and arrays of kb_tri / ka_tri (ktri.cuh) with an element's points, gradient
// and fluxes in one thread's registers.
//
// The dense reference operators are a few hundred coefficients; a block keeps
// them in shared memory, transposed and in pairs of outputs (TriPack), so that
// one broadcast 16-byte load feeds four to eight paired multiply-adds
// (fma.rn.f32x2: two outputs of a field).  Rows of elements pass between global
// memory and the threads through warp-private buffers copied with unit stride.
//
// The block-wide kernels computed each output as a dot product of two
// shared-memory vectors (two loads a multiply-add, with a barrier a Step) and
// were latency bound: 30.3 + 20.8 us a stage on 29,768 triangles of order 3, now
// 7.8 + 8.1.  1 / det J, edge lengths and normals come from a record rounded once
// from FP64 (KArgs.trig): formed in float in the kernels, their errors are alike
// at all points and stages of an element and add up (four steps 6 % further from
// FP64 than the block-wide kernels, 4 % nearer with the record).
#pragma once
#include "kline_pseudo.cuh"
#include "ktri.cuh"
#include "tripack.hpp"

namespace frp {

// Between operator rows: keeps the compiler from carrying operator values from
// one use to a later one in registers (they are several times the register
// file); within a row's uses the loads are shared.
__device__ __forceinline__ void tri_fence() { asm volatile("" ::: "memory"); }

// acc[q] += M[j][q] x_j for one input j
template <int NP>
__device__ __forceinline__ void tri_acc(const float2* row, float x, float2* acc) {
  if constexpr (NP % 2 == 0) {
#pragma unroll
    for (int q = 0; q < NP; q += 2) {
      const float4 r = *reinterpret_cast<const float4*>(row + q);
      acc[q] = fma2(make_float2(r.x, r.y), dup2(x), acc[q]);
      acc[q + 1] = fma2(make_float2(r.z, r.w), dup2(x), acc[q + 1]);
    }
  } else {
#pragma unroll
    for (int q = 0; q < NP; ++q) acc[q] = fma2(row[q], dup2(x), acc[q]);
  }
}
template <int NP>
__device__ __forceinline__ float pair_at(const float2 (&v)[NP], int i) {
  return (i & 1) ? v[i / 2].y : v[i / 2].x;
}

template <int P>
struct TriReg {
  using S = TriS<P>;
  static constexpr int N = P + 1, NU = S::NU, NF = S::NF, NPE = TriPack(P).npe, NPU = TriPack(P).npu;
  static constexpr int O_L = TriPack(P).o_l, O_D = TriPack(P).o_d, O_LIFT = TriPack(P).o_lift, O_V = TriPack(P).o_v,
                       SIZE = TriPack(P).size;
  static constexpr int TB = 32;  // threads a block
  // floats an element of the residual kernel's buffers: state (then the
  // divergence), velocities at the points, at the flux points (then the fluxes)
  static constexpr int KB_F = 2 * NU + 2 * NU + 2 * NF;
  static constexpr size_t KB_SMEM = ((size_t)SIZE + TB * KB_F) * 4;
  // update kernel: rp (then the stage value), solution pairs, accumulator, face
  // weights (then traces), w det J pairs
  static constexpr int KA_F = 2 * NU + 4 * NU + 2 * NU + 2 * NF + 2 * NU;
  static_assert(SIZE % 4 == 0 && O_D % 4 == 0 && O_LIFT % 4 == 0 && O_V % 4 == 0, "16-byte boundaries");
  __host__ __device__ static constexpr int ka_elems(int mode) { return mode == 0 ? 16 : 32; }  // elements a warp of the update kernel
  static constexpr size_t ka_smem(int mode) { return ((size_t)SIZE + TB / 32 * ka_elems(mode) * KA_F) * 4; }
};

// edge ed of element e: flags, partner's first flux point (of the edge's first point; the partner's points run
// backwards, which a field that takes these kernels has of every edge, see tri_edges_backwards) as an offset into an
// E x 2 x NF array (field 0).  The checked build looks at all words of the edge; an edge that is not whole becomes a wall.
template <int P>
__device__ __forceinline__ int tri_edge(const KArgs& A, int64_t e, int ed, int64_t& off) {
  constexpr int NF = TriS<P>::NF, N = P + 1;
  const int32_t own = (int32_t)(e * NF + ed * N);
  const int32_t w = __ldg(A.fnbr + own);
  const int32_t p = w >> 1;
#ifdef FR_BOUNDS_CHECK
  if (const int k = tri_edge_broken<N>(A.fnbr, A.E * NF, own); k >= 0) {
    atomicExch(&A.status[ST_STATUS], kStatusBounds);
    atomicExch(&A.status[ST_BAD_INDEX], A.fnbr[own + k]);
    off = (int64_t)e * 2 * NF + ed * N;
    return kFwL | kFwWall;
  }
#endif
  off = (int64_t)(p / NF) * 2 * NF + p % NF;
  return (w & 1) | (p == own ? kFwWall : 0);
}

__device__ __forceinline__ void tri_ops(const KArgs& A, float* ops, int n) {
  const float4* s = reinterpret_cast<const float4*>(A.tripack);
  for (int i = threadIdx.x; i < (n + 3) / 4; i += blockDim.x) reinterpret_cast<float4*>(ops)[i] = __ldg(s + i);
}

// warp's elements x PER bytes, contiguous on both sides
template <int PER>
__device__ __forceinline__ void tri_flush(void* dst, const float* src, int ne, int lane) {
  float2* d = static_cast<float2*>(dst);
  for (int i = lane; i < ne * PER / 8; i += 32) d[i] = reinterpret_cast<const float2*>(src)[i];
}

// ---- residual kernel: MODE 0 physical, 1 preconditioning (psi alone) ------------
template <int P, int MODE>
__global__ void __launch_bounds__(TriReg<P>::TB) kb_trir(const __grid_constant__ KArgs A) {
  using R = TriReg<P>;
  constexpr int N = R::N, NU = R::NU, NF = R::NF, NPE = R::NPE, NPU = R::NPU, NFLD = MODE == 0 ? 2 : 1, F0 = 2 - NFLD;
  if (MODE == 1 && *(volatile int32_t*)&A.status[ST_PSEUDO_DONE]) return;
  extern __shared__ __align__(16) float smem_f[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* ops = smem_f;
  float* ub = ops + R::SIZE + warp * 32 * R::KB_F;
  float* vub = ub + 32 * 2 * NU;
  float* vfb = vub + 32 * 2 * NU;
  const int64_t e0 = ((int64_t)blockIdx.x * R::TB) + warp * 32;
  const int ne = (int)max((int64_t)0, min((int64_t)32, A.E - e0));
  const int64_t e = min(e0 + lane, A.E - 1);
  const float2* Lt = reinterpret_cast<const float2*>(ops + R::O_L);
  const float2* Dt = reinterpret_cast<const float2*>(ops + R::O_D);
  const float2* Lf = reinterpret_cast<const float2*>(ops + R::O_LIFT);
  const float* trA = reinterpret_cast<const float*>(A.tr);
  const PrmT<float>& Pm = A.cf.prm;

  // ---- loads
  tile_fetch<32, 2 * NU * 4>(ub, reinterpret_cast<const float*>(A.ustg) + e0 * 2 * NU, ne, lane);
  if (MODE == 0) {
    tile_fetch<32, 2 * NU * 4>(vub, reinterpret_cast<const float*>(A.vsu) + e0 * 2 * NU, ne, lane);
    tile_fetch<32, 2 * NF * 4>(vfb, reinterpret_cast<const float*>(A.vsf) + e0 * 2 * NF, ne, lane);
  }
  tri_ops(A, ops, R::SIZE);
  int fl[3];
  float o[NFLD][3][N];
#pragma unroll
  for (int ed = 0; ed < 3; ++ed) {
    int64_t off;
    fl[ed] = tri_edge<P>(A, e, ed, off);
    const bool nb = fl[ed] == kFwL;
#pragma unroll
    for (int f = 0; f < NFLD; ++f)
#pragma unroll
      for (int k = 0; k < N; ++k) o[f][ed][k] = nb ? __ldg(trA + off + (F0 + f) * NF - k) : 0.f;
  }
  float g[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) g[i] = __ldg(A.geof + e * 6 + i);
  // affine map: S = det J J^{-1}
  const float S00 = g[5], S01 = -g[2], S10 = -g[4], S11 = g[1];
  const float4 rec = __ldg(A.trig + 3 * e), nrm = __ldg(A.trig + 3 * e + 1), nr2 = __ldg(A.trig + 3 * e + 2);
  const float rdj = rec.x, dj = nr2.z;
  constexpr float r2 = 0.70710678f;
  float gfac = 0.f;
  if (MODE == 0) gfac = time_factor_t<float>(A, A.use_dev_time ? A.dstate[DS_TIME] + rk_c(A.stage) * A.dt : A.t);
  cp_async_wait_all();
  __syncthreads();
  const float* ur = ub + lane * 2 * NU;
  float u[NFLD][NU];
#pragma unroll
  for (int f = 0; f < NFLD; ++f)
#pragma unroll
    for (int j = 0; j < NU; ++j) u[f][j] = ur[(F0 + f) * NU + j];

  // ---- Steps 1-3: traces, jumps, gradient (qr, qs: reference derivatives, then physical)
  float2 q[NFLD][2][NPU];
#pragma unroll
  for (int f = 0; f < NFLD; ++f)
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int i = 0; i < NPU; ++i) q[f][c][i] = dup2(0.f);
#pragma unroll
  for (int j = 0; j < NU; ++j)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      tri_fence();
#pragma unroll
      for (int f = 0; f < NFLD; ++f) tri_acc<NPU>(Dt + (c * NU + j) * NPU, u[f][j], q[f][c]);
    }
  float2 uf[NFLD][3][NPE];
#pragma unroll
  for (int ed = 0; ed < 3; ++ed) {
#pragma unroll
    for (int f = 0; f < NFLD; ++f)
#pragma unroll
      for (int i = 0; i < NPE; ++i) uf[f][ed][i] = dup2(0.f);
#pragma unroll
    for (int j = 0; j < NU; ++j) {
      tri_fence();
#pragma unroll
      for (int f = 0; f < NFLD; ++f) tri_acc<NPE>(Lt + (ed * NU + j) * NPE, u[f][j], uf[f][ed]);
    }
    const bool nb = fl[ed] == kFwL;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      tri_fence();
#pragma unroll
      for (int f = 0; f < NFLD; ++f) {
        const float own = pair_at(uf[f][ed], k);
        const float ot = nb ? o[f][ed][k] : own;
        o[f][ed][k] = ot;
        const float jm = ot - own;
        const float2* row = Lf + (ed * N + k) * NPU;
        if (ed == 0) tri_acc<NPU>(row, -jm, q[f][1]);
        else if (ed == 2) tri_acc<NPU>(row, -jm, q[f][0]);
        else {
          tri_acc<NPU>(row, r2 * jm, q[f][0]);
          tri_acc<NPU>(row, r2 * jm, q[f][1]);
        }
      }
    }
  }
#pragma unroll
  for (int f = 0; f < NFLD; ++f)
#pragma unroll
    for (int i = 0; i < NPU; ++i) {
      const float2 a = q[f][0][i], b = q[f][1][i];
      q[f][0][i] = mul2(fma2(dup2(S10), b, mul2(dup2(S00), a)), dup2(rdj));
      q[f][1][i] = mul2(fma2(dup2(S11), b, mul2(dup2(S01), a)), dup2(rdj));
    }
  // ---- resolution indicator
  float nu = 0.f;
  if (MODE == 1) {
    const float2* Vt = reinterpret_cast<const float2*>(ops + R::O_V);
    float2 c[NPU];
#pragma unroll
    for (int i = 0; i < NPU; ++i) c[i] = dup2(0.f);
#pragma unroll
    for (int j = 0; j < NU; ++j) {
      tri_fence();
      tri_acc<NPU>(Vt + j * NPU, u[0][j], c);
    }
    unsigned big = 0;
#pragma unroll
    for (int i = 0; i < NU; ++i) big = max(big, abs_bits(pair_at(c, i)));
    const float unit = energy_scale(big);
    float2 lo = make_float2(0.f, 0.f), hi = lo;
    int m = 0;
#pragma unroll
    for (int i = 0; i <= P; ++i)
#pragma unroll
      for (int j = 0; j <= P - i; ++j, ++m) {
        const float v = pair_at(c, m) * unit;
        const float s = __fmul_rn(v, v);
        float2& t = i + j == P ? hi : lo;
        t = ff_add(t, make_float2(s, __fmaf_rn(v, v, -s)));
      }
    nu = sensor_nu(A.prm, lo, hi, make_float2(A.prm.nu_h, A.prm.nu_l));
  }

  // ---- Step 5 by edge
  const float* vf = vfb + lane * 2 * NF;
  float cor[NFLD][3][N];
#pragma unroll
  for (int ed = 0; ed < 3; ++ed) {
    float2 qf[NFLD][2][NPE];
#pragma unroll
    for (int f = 0; f < NFLD; ++f)
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int i = 0; i < NPE; ++i) qf[f][c][i] = dup2(0.f);
#pragma unroll
    for (int j = 0; j < NU; ++j) {
      tri_fence();
#pragma unroll
      for (int f = 0; f < NFLD; ++f)
#pragma unroll
        for (int c = 0; c < 2; ++c) tri_acc<NPE>(Lt + (ed * NU + j) * NPE, pair_at(q[f][c], j), qf[f][c]);
    }
    const float pm = ed == 0 ? rec.y : ed == 1 ? rec.z : rec.w;
    const float n0 = ed == 0 ? nrm.x : ed == 1 ? nrm.z : nr2.x, n1 = ed == 0 ? nrm.y : ed == 1 ? nrm.w : nr2.y;
    const bool isl = fl[ed] & kFwL, shut = Pm.noflux && (fl[ed] & kFwWall);
    float Fv[NFLD][2 * NPE];
#pragma unroll
    for (int i = 0; i < NPE; ++i) {
      if (2 * i >= N) continue;
      const int k0 = ed * N + 2 * i, k1 = 2 * i + 1 < N ? k0 + 1 : k0;
      const float2 oL0 = uf[0][ed][i], oR0 = make_float2(o[0][ed][2 * i], 2 * i + 1 < N ? o[0][ed][2 * i + 1 < N ? 2 * i + 1 : 0] : 0.f);
      if constexpr (MODE == 0) {
        const float2 v0 = mul2(dup2(gfac), make_float2(vf[k0], vf[k1]));
        const float2 v1 = mul2(dup2(gfac), make_float2(vf[NF + k0], vf[NF + k1]));
        const float2 qn0 = Pm.nphi ? qf[0][0][i] : qf[NFLD - 1][0][i], qn1 = Pm.nphi ? qf[0][1][i] : qf[NFLD - 1][1][i];
        const float2 vn = fma2(v1, dup2(n1), mul2(v0, dup2(n0)));
        const float2 M = flux_mult(fma2(v1, v1, mul2(v0, v0)), Pm.gamma);
        const float2 sh = sharp2(oL0, fma2(qn1, qn1, mul2(qn0, qn0)), Pm.gamma, Pm.rdelta);
        const float2 w0 = fma2(sh, qn0, mul2(dup2(-Pm.eps), qf[0][0][i])), w1 = fma2(sh, qn1, mul2(dup2(-Pm.eps), qf[0][1][i]));
        const float2 nvis = mul2(M, fma2(w1, dup2(n1), mul2(w0, dup2(n0))));
        const float2 hv = mul2(dup2(0.5f), vn);
        const float2 sL = uf[NFLD - 1][ed][i];
        const float2 sR = make_float2(o[NFLD - 1][ed][2 * i], 2 * i + 1 < N ? o[NFLD - 1][ed][2 * i + 1 < N ? 2 * i + 1 : 0] : 0.f);
        const float2 Fp = fma2(dup2(Pm.tau), sub2(oL0, oR0), fma2(add2(oL0, oR0), hv, nvis));
        const float2 Fs = fma2(dup2(Pm.tau_psi), sub2(sL, sR), mul2(add2(sL, sR), hv));
        Fv[0][2 * i] = Fp.x;
        Fv[0][2 * i + 1] = Fp.y;
        Fv[NFLD - 1][2 * i] = Fs.x;
        Fv[NFLD - 1][2 * i + 1] = Fs.y;
      } else {
        const float2 gn = fma2(qf[0][1][i], dup2(n1), mul2(qf[0][0][i], dup2(n0)));
        const float2 F = fma2(dup2(Pm.tau_pseudo), sub2(oL0, oR0), mul2(dup2(-nu), gn));
        Fv[0][2 * i] = F.x;
        Fv[0][2 * i + 1] = F.y;
      }
    }
    // the edge's velocities are read: their place takes the physical flux out of L
    const bool zero = !isl || (MODE == 0 && shut);
#pragma unroll
    for (int f = 0; f < NFLD; ++f)
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const float F = zero ? 0.f : Fv[f][k];
        cor[f][ed][k] = pm * F;
        vfb[lane * 2 * NF + (F0 + f) * NF + ed * N + k] = F;
      }
  }

  // ---- Step 4: transformed flux in place of the gradient
  const float* vu = vub + lane * 2 * NU;
  float src[MODE == 1 ? NU : 1];
#pragma unroll
  for (int i = 0; i < NPU; ++i) {
    if (2 * i >= NU) continue;
    const int i0 = 2 * i, i1 = 2 * i + 1 < NU ? 2 * i + 1 : 2 * i;
    if constexpr (MODE == 0) {
      const float2 v0 = mul2(dup2(gfac), make_float2(vu[i0], vu[i1]));
      const float2 v1 = mul2(dup2(gfac), make_float2(vu[NU + i0], vu[NU + i1]));
      const float2 qs0 = Pm.nphi ? q[0][0][i] : q[NFLD - 1][0][i], qs1 = Pm.nphi ? q[0][1][i] : q[NFLD - 1][1][i];
      const float2 M = flux_mult(fma2(v1, v1, mul2(v0, v0)), Pm.gamma);
      const float2 ph = make_float2(u[0][i0], u[0][i1]), ps = make_float2(u[NFLD - 1][i0], u[NFLD - 1][i1]);
      const float2 sh = sharp2(ph, fma2(qs1, qs1, mul2(qs0, qs0)), Pm.gamma, Pm.rdelta);
      const float2 f00 = fma2(ph, v0, mul2(M, fma2(sh, qs0, mul2(dup2(-Pm.eps), q[0][0][i]))));
      const float2 f01 = fma2(ph, v1, mul2(M, fma2(sh, qs1, mul2(dup2(-Pm.eps), q[0][1][i]))));
      const float2 f10 = mul2(ps, v0), f11 = mul2(ps, v1);
      q[0][0][i] = fma2(dup2(S01), f01, mul2(dup2(S00), f00));
      q[0][1][i] = fma2(dup2(S11), f01, mul2(dup2(S10), f00));
      q[NFLD - 1][0][i] = fma2(dup2(S01), f11, mul2(dup2(S00), f10));
      q[NFLD - 1][1][i] = fma2(dup2(S11), f11, mul2(dup2(S10), f10));
    } else {
      const float2 a = q[0][0][i], b = q[0][1][i];
      const float2 g2 = fma2(b, b, mul2(a, a));
      q[0][0][i] = mul2(dup2(-nu), fma2(dup2(S01), b, mul2(dup2(S00), a)));
      q[0][1][i] = mul2(dup2(-nu), fma2(dup2(S11), b, mul2(dup2(S10), a)));
      const float m0 = sqrtf(g2.x), m1 = sqrtf(g2.y);
      const float p0 = (float)__ldg(A.psi0 + e * NU + i0), p1 = (float)__ldg(A.psi0 + e * NU + i1);
      src[i0] = tanhf(p0 / fmaxf(m0, Pm.delta)) * (1.f - m0) * dj;
      if (i1 != i0) src[i1] = tanhf(p1 / fmaxf(m1, Pm.delta)) * (1.f - m1) * dj;
    }
  }

  // ---- Step 6: flux jumps and divergence
  float2 dv[NFLD][NPU];
#pragma unroll
  for (int f = 0; f < NFLD; ++f)
#pragma unroll
    for (int i = 0; i < NPU; ++i) dv[f][i] = dup2(0.f);
#pragma unroll
  for (int j = 0; j < NU; ++j)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      tri_fence();
#pragma unroll
      for (int f = 0; f < NFLD; ++f) tri_acc<NPU>(Dt + (c * NU + j) * NPU, pair_at(q[f][c], j), dv[f]);
    }
#pragma unroll
  for (int ed = 0; ed < 3; ++ed) {
    float2 fp[NFLD][NPE];  // n~ . f~ at the edge's points, up to its constant factor
#pragma unroll
    for (int f = 0; f < NFLD; ++f)
#pragma unroll
      for (int i = 0; i < NPE; ++i) fp[f][i] = dup2(0.f);
#pragma unroll
    for (int j = 0; j < NU; ++j) {
      tri_fence();
#pragma unroll
      for (int f = 0; f < NFLD; ++f) {
        const float x = ed == 0 ? pair_at(q[f][1], j) : ed == 2 ? pair_at(q[f][0], j) : pair_at(q[f][0], j) + pair_at(q[f][1], j);
        tri_acc<NPE>(Lt + (ed * NU + j) * NPE, x, fp[f]);
      }
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
      tri_fence();
#pragma unroll
      for (int f = 0; f < NFLD; ++f) {
        const float x = pair_at(fp[f], k);
        const float c = ed == 1 ? __fmaf_rn(-r2, x, cor[f][ed][k]) : cor[f][ed][k] + x;
        tri_acc<NPU>(Lf + (ed * N + k) * NPU, c, dv[f]);
      }
    }
  }
  float* out = ub + lane * 2 * NU;
#pragma unroll
  for (int f = 0; f < NFLD; ++f)
#pragma unroll
    for (int j = 0; j < NU; ++j) {
      float d = pair_at(dv[f], j);
      if constexpr (MODE == 1) d -= src[j];
      out[(F0 + f) * NU + j] = d;
    }
  __syncwarp();
  float* rp = reinterpret_cast<float*>(A.rp) + e0 * 2 * NU;
  float* fc = reinterpret_cast<float*>(A.fc) + e0 * 2 * NF;
  if constexpr (MODE == 0) {
    tri_flush<2 * NU * 4>(rp, ub, ne, lane);
    tri_flush<2 * NF * 4>(fc, vfb, ne, lane);
  } else {  // psi's half of the rows
    for (int i = lane; i < ne * NU; i += 32) rp[(i / NU) * 2 * NU + NU + i % NU] = ub[(i / NU) * 2 * NU + NU + i % NU];
    for (int i = lane; i < ne * NF; i += 32) fc[(i / NF) * 2 * NF + NF + i % NF] = vfb[(i / NF) * 2 * NF + NF + i % NF];
  }
}

// ---- update kernel: SF 1..4, or 0 for the traces of ustg alone -----------------
// The fields are independent here, so a thread takes one field of one element
// in the physical step (16 elements a warp, twice the warps of a thread an
// element: 10.0 -> 8.3 us a stage on 29,768 triangles of order 3), psi of one
// element in the preconditioning (32 a warp, rows of both fields in the buffers).
template <int P, int MODE, int SF>
__global__ void __launch_bounds__(TriReg<P>::TB) ka_trir(const __grid_constant__ KArgs A) {
  using R = TriReg<P>;
  constexpr int N = R::N, NU = R::NU, NF = R::NF, NPE = R::NPE, NPU = R::NPU;
  constexpr int EW = R::ka_elems(MODE);  // elements a warp
  if (MODE == 1 && *(volatile int32_t*)&A.status[ST_PSEUDO_DONE]) return;
  extern __shared__ __align__(16) float smem_f[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int el = MODE == 0 ? lane >> 1 : lane, f = MODE == 0 ? lane & 1 : 1;  // the thread's element and field
  float* ops = smem_f;
  float* yb = ops + R::SIZE + warp * EW * R::KA_F;
  float* sb = yb + EW * 2 * NU;   // solution pairs
  float* ab = sb + EW * 4 * NU;   // accumulator
  float* tb = ab + EW * 2 * NU;   // face weights, later the traces
  float* wb = tb + EW * 2 * NF;   // w det J pairs (stage 4)
  const int64_t e0 = ((int64_t)blockIdx.x * (R::TB / 32) + warp) * EW;
  const int ne = (int)max((int64_t)0, min((int64_t)EW, A.E - e0));
  const bool act = el < ne;
  const int64_t e = min(e0 + el, A.E - 1);
  const float2* Lt = reinterpret_cast<const float2*>(ops + R::O_L);
  const float2* Lf = reinterpret_cast<const float2*>(ops + R::O_LIFT);
  const float* fcA = reinterpret_cast<const float*>(A.fc);
  float* ustg = reinterpret_cast<float*>(A.ustg);
  const bool cons = MODE == 0 && SF >= 1 && A.tacc && A.wphys;

  // ---- loads (whole rows of both fields)
  tile_fetch<EW, 2 * NU * 4>(yb, (SF == 0 ? ustg : reinterpret_cast<const float*>(A.rp)) + e0 * 2 * NU, ne, lane);
  if (SF >= 1) tile_fetch<EW, 2 * NU * 8>(sb, reinterpret_cast<const float2*>(A.u) + e0 * 2 * NU, ne, lane);
  // acc: at stage 1 only the other field's half of a preconditioning row is kept
  if (SF >= 2 || (SF == 1 && MODE == 1)) tile_fetch<EW, 2 * NU * 4>(ab, reinterpret_cast<const float*>(A.acc) + e0 * 2 * NU, ne, lane);
  if (cons) {
    tile_fetch<EW, NF * 8>(tb, A.wphys + e0 * NF, ne, lane);
    if (SF == 4) tile_fetch<EW, NU * 8>(wb, A.wdetf + e0 * NU, ne, lane);
  }
  float phi_keep[MODE == 1 ? NU : 1];  // preconditioning: phi's stage value
  if (MODE == 1 && SF >= 1)
#pragma unroll
    for (int j = 0; j < NU; ++j) phi_keep[j] = ustg[e * 2 * NU + j];
  tri_ops(A, ops, R::SIZE);
  float F[3][N];
  int fl[3];
  float pm[3] = {0.f, 0.f, 0.f}, rdj = 0.f;
  if constexpr (SF >= 1) {
    const float4 rec = __ldg(A.trig + 3 * e);
    rdj = rec.x;
    pm[0] = rec.y;
    pm[1] = rec.z;
    pm[2] = rec.w;
#pragma unroll
    for (int ed = 0; ed < 3; ++ed) {
      int64_t off;
      fl[ed] = tri_edge<P>(A, e, ed, off);
      const bool isl = fl[ed] & kFwL;
      // the own flux at L points, the partner's at R points (points backwards)
      const float* b = fcA + (isl ? e * 2 * NF + ed * N : off) + f * NF;
      const int st = isl ? 1 : -1;
#pragma unroll
      for (int k = 0; k < N; ++k) F[ed][k] = (MODE == 0 || !isl) ? b[k * st] : 0.f;
    }
  }
  double ta = 0.0, W = 1.0;
  if (SF >= 2 && cons) ta = A.tacc[e * 2 + f];
  if (SF == 4 && cons) W = __ldg(A.triw + e);
  cp_async_wait_all();
  __syncthreads();
  float* yr = yb + (el * 2 + f) * NU;
  float2 y[NPU];
#pragma unroll
  for (int i = 0; i < NPU; ++i)
    y[i] = make_float2(2 * i < NU ? yr[2 * i < NU ? 2 * i : 0] : 0.f, 2 * i + 1 < NU ? yr[2 * i + 1 < NU ? 2 * i + 1 : 0] : 0.f);
  [[maybe_unused]] double sq = 0.0;  // MODE 1 stage 4: squared changes
  if constexpr (SF >= 1) {
    // ---- lift of minus the partner's flux at R points; flux balance
    float2 bal = make_float2(0.f, 0.f);
#pragma unroll
    for (int ed = 0; ed < 3; ++ed) {
      const bool isl = fl[ed] & kFwL;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        if (cons) {
          const float2 w = reinterpret_cast<const float2*>(tb)[el * NF + ed * N + k];
          bal = ff_add(bal, ff_mul(w, isl ? F[ed][k] : -F[ed][k]));
        }
        tri_fence();
        tri_acc<NPU>(Lf + (ed * N + k) * NPU, isl ? 0.f : -pm[ed] * F[ed][k], y);
      }
    }
    if (cons && SF < 4 && act) {
      const double Te = -((double)bal.x + (double)bal.y);
      A.tacc[e * 2 + f] = SF == 1 ? Te : ta + 2.0 * Te;
    }
    float2* sr = reinterpret_cast<float2*>(sb) + (el * 2 + f) * NU;
    float* ar = ab + (el * 2 + f) * NU;
    float bad = 0.f;
    float2 Ssum = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < NU; ++j) {
      const float Rj = -pair_at(y, j) * rdj;
      const float2 uu = sr[j];
      float yn;
      if constexpr (SF == 1) {
        ar[j] = Rj;
        yn = uu.x + __fmaf_rn(A.rk.half_dt, Rj, uu.y);
      } else if constexpr (SF == 2 || SF == 3) {
        ar[j] = __fmaf_rn(2.f, Rj, ar[j]);
        yn = uu.x + __fmaf_rn(SF == 2 ? A.rk.half_dt : A.rk.dt, Rj, uu.y);
      } else {
        const float inc = A.rk.dt6 * (ar[j] + Rj);
        const float s2 = uu.x + inc;
        const float e2 = two_sum_lo(uu.x, inc, s2) + uu.y;
        yn = s2 + e2;
        const float lo = e2 - (yn - s2);
        sr[j] = make_float2(yn, lo);
        if constexpr (MODE == 0) {
          if (cons) {
            const float2 wd = reinterpret_cast<const float2*>(wb)[el * NU + j];
            Ssum = ff_add(Ssum, ff_mul(wd, inc));
          }
        } else {
          const float h = yn - uu.x;
          const double d = widen(h) + widen(two_sum_lo(yn, -uu.x, h) + (lo - uu.y));
          sq = fma(d, d, sq);
        }
      }
      bad = __fmaf_rn(yn, 0.f, bad);
      if (j & 1) y[j / 2].y = yn;
      else y[j / 2].x = yn;
    }
    if constexpr (SF == 4 && MODE == 0) {
      if (cons) {
        const double Te = -((double)bal.x + (double)bal.y);
        const double tgt = A.rk.ddt6 * (ta + Te);
        const double d = (tgt - ((double)Ssum.x + (double)Ssum.y)) / W;
        const float dh = (float)d, dl = (float)(d - (double)dh);
#pragma unroll
        for (int j = 0; j < NU; ++j) {
          const float2 uu = sr[j];
          const float s2 = uu.x + dh;
          const float e2 = two_sum_lo(uu.x, dh, s2) + (uu.y + dl);
          const float hi = s2 + e2;
          sr[j] = make_float2(hi, e2 - (hi - s2));
          bad = __fmaf_rn(hi, 0.f, bad);
          if (j & 1) y[j / 2].y = hi;
          else y[j / 2].x = hi;
        }
      }
    }
    if (act && bad != 0.f) atomicExch(&A.status[ST_STATUS], -4);
#pragma unroll
    for (int j = 0; j < NU; ++j) yr[j] = pair_at(y, j);
    if (MODE == 1)
#pragma unroll
      for (int j = 0; j < NU; ++j) yr[j - NU] = phi_keep[j];
  }
  // ---- traces of the new stage value, in the weights' place (rows of the warp's threads)
  __syncwarp();
  float* trr = tb + lane * NF;
#pragma unroll
  for (int ed = 0; ed < 3; ++ed) {
    float2 t[NPE];
#pragma unroll
    for (int i = 0; i < NPE; ++i) t[i] = dup2(0.f);
#pragma unroll
    for (int j = 0; j < NU; ++j) {
      tri_fence();
      tri_acc<NPE>(Lt + (ed * NU + j) * NPE, pair_at(y, j), t);
    }
#pragma unroll
    for (int k = 0; k < N; ++k) trr[ed * N + k] = pair_at(t, k);
  }
  __syncwarp();
  float* tr = reinterpret_cast<float*>(A.tr);
  if constexpr (MODE == 0) tri_flush<2 * NF * 4>(tr + e0 * 2 * NF, tb, ne, lane);
  else rows_flush<NF>(tr + (e0 * 2 + 1) * NF, tb, 2 * NF, ne, lane);
  if constexpr (SF >= 1) {
    tri_flush<2 * NU * 4>(ustg + e0 * 2 * NU, yb, ne, lane);
    if (SF < 4) tri_flush<2 * NU * 4>(reinterpret_cast<float*>(A.acc) + e0 * 2 * NU, ab, ne, lane);
    else tri_flush<2 * NU * 8>(reinterpret_cast<float2*>(A.u) + e0 * 2 * NU, sb, ne, lane);
  }
  if (MODE == 0 && SF == 4 && A.use_dev_time && blockIdx.x == 0 && threadIdx.x == 0)
    A.dstate[DS_TIME] = A.dstate[DS_TIME] + A.dt;
  if constexpr (MODE == 1 && SF == 4) {
    __shared__ double part[TriReg<P>::TB / 32];
    __shared__ double red_sh[32];
    double v = act ? sq * (A.rk.rdt * A.rk.rdt) : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) part[warp] = v;
    __syncthreads();
    double s = 0.0;
    for (int w = 0; w < TriReg<P>::TB / 32; ++w) s += part[w];
    pseudo_rms_finish(A, s, red_sh, A.E * NU);
  }
}

}  // namespace frp
