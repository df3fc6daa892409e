// FR kernels for straight-sided triangles (affine map, constant J per
// element) with dense reference operators: the same Steps 1-6 and kernel
// split as ktensor.cuh, with the line applies replaced by small dense
// matrix products over a tile of elements staged in shared memory.  In the
// float (mixed) path every operator apply is a tensor-core contraction
// (mma_tf32.cuh, three-term TF32 with FP32 accumulation) over the tile's
// element-field columns:
//   Step 1      u^f            = L u                       (NF x NU)
//   Step 3      q~_c           = D_c u + LIFT (n~_c (C - u^f))   ([D_c | LIFT n~_c], 2 NU x (NU + NF))
//   Step 5      q^f            = L q                       (per gradient component)
//   Step 4/6    f~perp          = n~ . (L f~)
//   Step 6      div~ f~        = Dr f~_0 + Ds f~_1 + LIFT (F~ - f~perp)   ([Dr | Ds | LIFT], NU x (2 NU + NF))
//   ka          R-side lift LIFT c and the next stage's traces L y
// The FP64 path keeps scalar dot products (FP64 tensor throughput is far
// below the FP64 FMA pipe's on this GPU).  Mixed fields of variant 0 and order
// up to 4 run on ktri_reg.cuh (their physical step where the velocity is cached).
#pragma once
#include <type_traits>

#include "kcommon.cuh"
#include "mma_tf32.cuh"

namespace frp {

template <int P>
struct TriS {
  static constexpr int N = P + 1;
  static constexpr int NU = N * (N + 1) / 2;
  static constexpr int NF = 3 * N;
  static constexpr int NG = 6;
};

template <int P, typename T>
struct TriOpsS {
  static constexpr int NU = TriS<P>::NU, NF = TriS<P>::NF;
  T L[NF][NU], Dr[NU][NU], Ds[NU][NU], LIFT[NU][NF], Vinv[NU][NU];
  T xf[NF][2], nref[NF][2];
  unsigned char high[NU];
};

template <int P, typename T>
__device__ __forceinline__ void load_tri_ops(const TriOpsT<T>& o, TriOpsS<P, T>& s) {
  constexpr int NU = TriS<P>::NU, NF = TriS<P>::NF;
  for (int t = threadIdx.x; t < NF * NU; t += blockDim.x) {
    s.L[t / NU][t % NU] = o.L[t];
    s.LIFT[t / NF][t % NF] = o.LIFT[t];
  }
  for (int t = threadIdx.x; t < NU * NU; t += blockDim.x) {
    s.Dr[t / NU][t % NU] = o.Dr[t];
    s.Ds[t / NU][t % NU] = o.Ds[t];
    s.Vinv[t / NU][t % NU] = o.Vinv[t];
  }
  for (int t = threadIdx.x; t < NF * 2; t += blockDim.x) {
    s.xf[t / 2][t % 2] = o.xf[t];
    s.nref[t / 2][t % 2] = o.nref[t];
  }
  for (int t = threadIdx.x; t < NU; t += blockDim.x) s.high[t] = o.high[t];
}

// per-element metric of the affine map: S = det J J^{-1}, det J
template <typename T>
struct TriMet {
  T S[2][2];
  T dj;
};

template <typename T>
__device__ __forceinline__ void tri_metric(const T* g, TriMet<T>& m) {
  T J[3][3], Sm[3][3];
  const T xi[2] = {0, 0};
  jacobian<ET_TRI, T>(g, xi, J);
  m.dj = adjugate<2, T>(J, Sm);
  m.S[0][0] = Sm[0][0];
  m.S[0][1] = Sm[0][1];
  m.S[1][0] = Sm[1][0];
  m.S[1][1] = Sm[1][1];
}

// TC: the float path's operator applies on tensor cores (mma_tf32.cuh);
// otherwise scalar dot products (the only form of the FP64 path).
// TD: tile divisor; FP64 fields on small meshes take quarter tiles, so that
// their few blocks spread over the SMs (see fill_tri).
template <int P, typename T, int MODE, bool TC = false, int TD = 1>
struct KBTriLayout {
  using S = TriS<P>;
  static constexpr int NFLD = MODE == 0 ? 2 : 1;
  static constexpr bool MMA = TC && std::is_same<T, float>::value;
  // + the float path's [ET][NFLD][2][NF] buffer of L applied to q, then to f~
  static constexpr int PER_EL_T = NFLD * S::NU + 3 * NFLD * S::NF + NFLD * 2 * S::NU + S::NG + 5 + 1 +
                                  (MMA ? NFLD * 2 * S::NF : 0);
  static constexpr int BYTES_EL = PER_EL_T * (int)sizeof(T) + S::NF;
  static constexpr int ETr = 32768 / BYTES_EL;
  static constexpr int ET1 = ETr < 1 ? 1 : (ETr > 64 ? 64 : ETr);
  static constexpr int ET = ET1 / TD < 1 ? 1 : ET1 / TD;
  static constexpr size_t SMEM = (size_t)ET * BYTES_EL + sizeof(TriOpsS<P, T>) + 64;
};

template <int P, typename T, int MODE, bool TC = false, int TD = 1>
__global__ void __launch_bounds__(kThreads) kb_tri(const KArgs A) {
  using S = TriS<P>;
  using LY = KBTriLayout<P, T, MODE, TC, TD>;
  constexpr int NU = S::NU, NF = S::NF, NG = S::NG, NFLD = LY::NFLD, ET = LY::ET, N = S::N;
  constexpr int F0 = MODE == 0 ? 0 : 1;
  constexpr bool kMMA = LY::MMA;
  if (MODE == 1 && *(volatile int32_t*)&A.status[ST_PSEUDO_DONE]) return;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  TriOpsS<P, T>& op = *reinterpret_cast<TriOpsS<P, T>*>(smem_raw);
  T* base = reinterpret_cast<T*>(smem_raw + ((sizeof(TriOpsS<P, T>) + 15) & ~size_t(15)));
  T* us = base;                         // [ET][NFLD][NU]
  T* uf = us + ET * NFLD * NU;          // [ET][NFLD][NF]
  T* uo = uf + ET * NFLD * NF;
  T* cor = uo + ET * NFLD * NF;
  T* q = cor + ET * NFLD * NF;          // [ET][NFLD][2][NU]
  T* gs = q + ET * NFLD * 2 * NU;       // [ET][NG]
  T* met = gs + ET * NG;                // [ET][5]: S00 S01 S10 S11 dj
  T* nus = met + ET * 5;                // [ET]
  T* qf = nus + ET;                     // float path: [ET][NFLD][2][NF]
  unsigned char* lm = reinterpret_cast<unsigned char*>(qf + (kMMA ? ET * NFLD * 2 * NF : 0));

  const int64_t e0 = (int64_t)blockIdx.x * ET;
  const int ne = (int)min((int64_t)ET, A.E - e0);
  const int ncol = ne * NFLD;           // element-field columns of the tile
  const T* ustg = reinterpret_cast<const T*>(A.ustg);
  const T* tr = reinterpret_cast<const T*>(A.tr);
  T* fc = reinterpret_cast<T*>(A.fc);
  T* rp = reinterpret_cast<T*>(A.rp);
  const int tid = threadIdx.x;
  const BulkConst<T>& BC = bulk<T>(A);
  const PrmT<T> Pm = BC.prm;
  __shared__ T gfac_s;
  if (tid == 0) {
    const double tstage = A.use_dev_time ? A.dstate[DS_TIME] + rk_c(A.stage) * A.dt : A.t;
    gfac_s = time_factor_t<T>(A, tstage);
  }

  load_tri_ops<P, T>(tri_of<T>(A), op);
  for (int idx = tid; idx < ne * NFLD * NU; idx += blockDim.x) {
    const int el = idx / (NFLD * NU), r = idx % (NFLD * NU), fld = r / NU, i = r % NU;
    us[idx] = ustg[((e0 + el) * 2 + F0 + fld) * NU + i];
  }
  for (int idx = tid; idx < ne * NG; idx += blockDim.x) gs[idx] = geo_of<T>(A)[e0 * NG + idx];
  __syncthreads();
  for (int el = tid; el < ne; el += blockDim.x) {
    TriMet<T> m;
    tri_metric(gs + el * NG, m);
    met[el * 5 + 0] = m.S[0][0];
    met[el * 5 + 1] = m.S[0][1];
    met[el * 5 + 2] = m.S[1][0];
    met[el * 5 + 3] = m.S[1][1];
    met[el * 5 + 4] = m.dj;
  }
  const T gfac = gfac_s;
  // ---- Step 1 (u^f = L u) and partner traces
  if constexpr (kMMA) {
    warp_gemm_3xtf32<NF, NU>(
        ncol, [&](int r, int k) { return op.L[r][k]; }, [&](int c, int k) { return us[c * NU + k]; },
        [&](int c, int r, float v) { uf[c * NF + r] = v; });
    __syncthreads();
  }
  for (int idx = tid; idx < ne * NF; idx += blockDim.x) {
    const int el = idx / NF, k = idx % NF;
    const int32_t w = A.fnbr[(e0 + el) * NF + k];
    const int isL = w & 1;
    const int64_t pg = (int64_t)partner<NF>(A, w, (int32_t)((e0 + el) * NF + k)), pe = pg / NF, pk = pg % NF;
    lm[el * NF + k] = (unsigned char)isL;
#pragma unroll
    for (int fld = 0; fld < NFLD; ++fld) {
      T acc;
      if constexpr (kMMA) {
        acc = uf[(el * NFLD + fld) * NF + k];
      } else {
        const T* ul = us + (el * NFLD + fld) * NU;
        acc = 0;
#pragma unroll
        for (int j = 0; j < NU; ++j) acc += op.L[k][j] * ul[j];
        uf[(el * NFLD + fld) * NF + k] = acc;
      }
      const T o = isL ? tr[(pe * 2 + F0 + fld) * NF + pk] : acc;
      uo[(el * NFLD + fld) * NF + k] = o;
      // jump C - u^f of Step 3 (C = u_R: nonzero at L points only)
      if constexpr (kMMA) cor[(el * NFLD + fld) * NF + k] = isL ? o - acc : (T)0;
    }
  }
  __syncthreads();
  // ---- Step 3
  if constexpr (kMMA) {
    // q~_c = [D_c | LIFT n~_c] [u; C - u^f] for c = 0, 1 (rows c NU + i)
    warp_gemm_3xtf32<2 * NU, NU + NF>(
        ncol,
        [&](int r, int k) {
          const int c = r / NU, i = r % NU;
          return k < NU ? (c ? op.Ds[i][k] : op.Dr[i][k]) : op.LIFT[i][k - NU] * op.nref[k - NU][c];
        },
        [&](int c, int k) { return k < NU ? us[c * NU + k] : cor[c * NF + k - NU]; },
        [&](int c, int r, float v) { q[(c * 2 + r / NU) * NU + r % NU] = v; });
    __syncthreads();
    // q_b = sum_a S[a][b] q~_a / det J
    for (int idx = tid; idx < ncol * NU; idx += blockDim.x) {
      const int c = idx / NU, i = idx % NU;
      const T* mt = met + (c / NFLD) * 5;
      const T rdj = (T)1 / mt[4];
      const T q0 = q[(c * 2 + 0) * NU + i], q1 = q[(c * 2 + 1) * NU + i];
      q[(c * 2 + 0) * NU + i] = (mt[0] * q0 + mt[2] * q1) * rdj;
      q[(c * 2 + 1) * NU + i] = (mt[1] * q0 + mt[3] * q1) * rdj;
    }
  } else {
    for (int idx = tid; idx < ne * NU; idx += blockDim.x) {
      const int el = idx / NU, i = idx % NU;
      const T* mt = met + el * 5;
      const T rdj = (T)1 / mt[4];
#pragma unroll
      for (int fld = 0; fld < NFLD; ++fld) {
        const T* ul = us + (el * NFLD + fld) * NU;
        const T* fo = uo + (el * NFLD + fld) * NF;
        const T* ff = uf + (el * NFLD + fld) * NF;
        T q0 = 0, q1 = 0;
#pragma unroll
        for (int j = 0; j < NU; ++j) {
          q0 += op.Dr[i][j] * ul[j];
          q1 += op.Ds[i][j] * ul[j];
        }
#pragma unroll
        for (int k = 0; k < NF; ++k) {
          const T jmp = lm[el * NF + k] ? fo[k] - ff[k] : (T)0;
          const T lj = op.LIFT[i][k] * jmp;
          q0 += lj * op.nref[k][0];
          q1 += lj * op.nref[k][1];
        }
        // q_b = sum_a S[a][b] q~_a / det J
        q[((el * NFLD + fld) * 2 + 0) * NU + i] = (mt[0] * q0 + mt[2] * q1) * rdj;
        q[((el * NFLD + fld) * 2 + 1) * NU + i] = (mt[1] * q0 + mt[3] * q1) * rdj;
      }
    }
  }
  if (MODE == 1) {
    for (int el = tid; el < ne; el += blockDim.x) {
      const T* ul = us + el * NU;
      double tot = 0.0, hi = 0.0;
      for (int m = 0; m < NU; ++m) {
        T c = 0;
        for (int j = 0; j < NU; ++j) c += op.Vinv[m][j] * ul[j];
        const double v = (double)c * (double)c;
        tot += v;
        if (op.high[m]) hi += v;
      }
      double nu = 0.0;
      if (tot > 0.0 && hi > 0.0) {
        const double se = log10(hi / tot);
        const double lo = A.prm.s0 - A.prm.kappa, up = A.prm.s0 + A.prm.kappa;
        if (se < lo) nu = 0.0;
        else if (se > up) nu = A.prm.nu_max;
        else nu = 0.5 * A.prm.nu_max * (1.0 + sin(M_PI * (se - A.prm.s0) / (2.0 * A.prm.kappa)));
      }
      nus[el] = (T)nu;
    }
  }
  __syncthreads();
  if constexpr (kMMA) {
    // q^f = L q, both components of every field (Eq. extrapolateGrad)
    warp_gemm_3xtf32<NF, NU>(
        ncol * 2, [&](int r, int k) { return op.L[r][k]; }, [&](int c, int k) { return q[c * NU + k]; },
        [&](int c, int r, float v) { qf[c * NF + r] = v; });
    __syncthreads();
  }
  // ---- Step 5 on L points
  for (int idx = tid; idx < ne * NF; idx += blockDim.x) {
    const int el = idx / NF, k = idx % NF;
    if (!lm[el * NF + k]) {
#pragma unroll
      for (int fld = 0; fld < NFLD; ++fld) cor[(el * NFLD + fld) * NF + k] = 0;
      continue;
    }
    const T* mt = met + el * 5;
    T pn[2];
    pn[0] = mt[0] * op.nref[k][0] + mt[2] * op.nref[k][1];
    pn[1] = mt[1] * op.nref[k][0] + mt[3] * op.nref[k][1];
    const T pm = sqrt_(pn[0] * pn[0] + pn[1] * pn[1]);
    const T nh[2] = {pn[0] / pm, pn[1] / pm};
    if (MODE == 0) {
      T qfv[2][2];
#pragma unroll
      for (int fld = 0; fld < 2; ++fld)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if constexpr (kMMA) {
            qfv[fld][c] = qf[((el * 2 + fld) * 2 + c) * NF + k];
          } else {
            const T* ql = q + ((el * 2 + fld) * 2 + c) * NU;
            T acc = 0;
#pragma unroll
            for (int j = 0; j < NU; ++j) acc += op.L[k][j] * ql[j];
            qfv[fld][c] = acc;
          }
        }
      T v[3];
      if (A.vsf) {  // the velocity cache: v(x) at the flux point, evaluated in FP64
        const T* vc = reinterpret_cast<const T*>(A.vsf) + (e0 + el) * 2 * NF + k;
        v[0] = gfac * vc[0];
        v[1] = gfac * vc[NF];
      } else {
        T x[3];
        map_point<ET_TRI, T>(gs + el * NG, op.xf[k], x);
        velocity<2, T>(BC.vel, x, gfac, v);
      }
      const T vn = v[0] * nh[0] + v[1] * nh[1];
      const T M = fmax(sqrt_(v[0] * v[0] + v[1] * v[1]), Pm.gamma);
      const int kn = Pm.nphi ? 0 : 1;  // field whose gradient gives the interface normal
      const T gm = fmax(sqrt_(qfv[kn][0] * qfv[kn][0] + qfv[kn][1] * qfv[kn][1]), Pm.delta);
      const T pL = uf[(el * 2 + 0) * NF + k], pR = uo[(el * 2 + 0) * NF + k];
      const T sL = uf[(el * 2 + 1) * NF + k], sR = uo[(el * 2 + 1) * NF + k];
      const T sharp = Pm.gamma * pL * ((T)1 - pL) / gm;
      T fvn = 0;
#pragma unroll
      for (int c = 0; c < 2; ++c) fvn += nh[c] * M * (Pm.eps * qfv[0][c] - sharp * qfv[kn][c]);
      const bool shut = Pm.noflux && A.fnbr[(e0 + el) * NF + k] >> 1 == (e0 + el) * NF + k;  // no-flux wall
      const T Fp = shut ? (T)0 : (T)0.5 * (pL + pR) * vn - fvn + Pm.tau * (pL - pR);
      const T Fs = shut ? (T)0 : (T)0.5 * (sL + sR) * vn + Pm.tau_psi * (sL - sR);
      fc[((e0 + el) * 2 + 0) * NF + k] = Fp;
      fc[((e0 + el) * 2 + 1) * NF + k] = Fs;
      cor[(el * 2 + 0) * NF + k] = pm * Fp;
      cor[(el * 2 + 1) * NF + k] = pm * Fs;
    } else {
      T gn = 0;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        T acc;
        if constexpr (kMMA) {
          acc = qf[c * NF + k + el * 2 * NF];
        } else {
          const T* ql = q + (el * 2 + c) * NU;
          acc = 0;
#pragma unroll
          for (int j = 0; j < NU; ++j) acc += op.L[k][j] * ql[j];
        }
        gn += nh[c] * acc;
      }
      const T F = -nus[el] * gn + Pm.tau_pseudo * (uf[el * NF + k] - uo[el * NF + k]);
      fc[((e0 + el) * 2 + 1) * NF + k] = F;
      cor[el * NF + k] = pm * F;
    }
  }
  __syncthreads();
  // ---- Step 4
  for (int idx = tid; idx < ne * NU; idx += blockDim.x) {
    const int el = idx / NU, i = idx % NU;
    const T* mt = met + el * 5;
    if (MODE == 0) {
      T v[3];
      if (A.vsu) {  // the velocity cache: v(x) at the solution point, evaluated in FP64
        const T* vc = reinterpret_cast<const T*>(A.vsu) + (e0 + el) * 2 * NU + i;
        v[0] = gfac * vc[0];
        v[1] = gfac * vc[NU];
      } else {
        T xi[2], x[3];
        const T* xr = tri_of<T>(A).xu + 2 * i;  // solution point i in the reference triangle
        xi[0] = xr[0];
        xi[1] = xr[1];
        map_point<ET_TRI, T>(gs + el * NG, xi, x);
        velocity<2, T>(BC.vel, x, gfac, v);
      }
      const T qp0 = q[((el * 2 + 0) * 2 + 0) * NU + i], qp1 = q[((el * 2 + 0) * 2 + 1) * NU + i];
      const int kn = Pm.nphi ? 0 : 1;  // field whose gradient gives the interface normal
      const T qs0 = q[((el * 2 + kn) * 2 + 0) * NU + i], qs1 = q[((el * 2 + kn) * 2 + 1) * NU + i];
      const T M = fmax(sqrt_(v[0] * v[0] + v[1] * v[1]), Pm.gamma);
      const T gm = fmax(sqrt_(qs0 * qs0 + qs1 * qs1), Pm.delta);
      const T ph = us[(el * 2 + 0) * NU + i], ps = us[(el * 2 + 1) * NU + i];
      const T sharp = Pm.gamma * ph * ((T)1 - ph) / gm;
      const T f00 = ph * v[0] - M * (Pm.eps * qp0 - sharp * qs0);
      const T f01 = ph * v[1] - M * (Pm.eps * qp1 - sharp * qs1);
      const T f10 = ps * v[0], f11 = ps * v[1];
      q[((el * 2 + 0) * 2 + 0) * NU + i] = mt[0] * f00 + mt[1] * f01;
      q[((el * 2 + 0) * 2 + 1) * NU + i] = mt[2] * f00 + mt[3] * f01;
      q[((el * 2 + 1) * 2 + 0) * NU + i] = mt[0] * f10 + mt[1] * f11;
      q[((el * 2 + 1) * 2 + 1) * NU + i] = mt[2] * f10 + mt[3] * f11;
    } else {
      const T qs0 = q[(el * 2 + 0) * NU + i], qs1 = q[(el * 2 + 1) * NU + i];
      const T nu = nus[el];
      q[(el * 2 + 0) * NU + i] = mt[0] * (-nu * qs0) + mt[1] * (-nu * qs1);
      q[(el * 2 + 1) * NU + i] = mt[2] * (-nu * qs0) + mt[3] * (-nu * qs1);
      const T qm = sqrt_(qs0 * qs0 + qs1 * qs1);
      const T p0 = (T)A.psi0[(e0 + el) * NU + i];
      us[el * NU + i] = tanh_(p0 / fmax(qm, Pm.delta)) * ((T)1 - qm) * mt[4];
    }
  }
  __syncthreads();
  // ---- normal discontinuous flux and jumps
  if constexpr (kMMA) {
    warp_gemm_3xtf32<NF, NU>(
        ncol * 2, [&](int r, int k) { return op.L[r][k]; }, [&](int c, int k) { return q[c * NU + k]; },
        [&](int c, int r, float v) { qf[c * NF + r] = v; });
    __syncthreads();
    for (int idx = tid; idx < ncol * NF; idx += blockDim.x) {
      const int c = idx / NF, k = idx % NF;
      cor[idx] = cor[idx] - (op.nref[k][0] * qf[(c * 2 + 0) * NF + k] + op.nref[k][1] * qf[(c * 2 + 1) * NF + k]);
    }
  } else {
    for (int idx = tid; idx < ne * NFLD * NF; idx += blockDim.x) {
      const int el = idx / (NFLD * NF), r = idx % (NFLD * NF), fld = r / NF, k = r % NF;
      const T* f0 = q + ((el * NFLD + fld) * 2 + 0) * NU;
      const T* f1 = q + ((el * NFLD + fld) * 2 + 1) * NU;
      T a0 = 0, a1 = 0;
#pragma unroll
      for (int j = 0; j < NU; ++j) {
        a0 += op.L[k][j] * f0[j];
        a1 += op.L[k][j] * f1[j];
      }
      cor[idx] = cor[idx] - (op.nref[k][0] * a0 + op.nref[k][1] * a1);
    }
  }
  __syncthreads();
  // ---- Step 6
  if constexpr (kMMA) {
    // div~ f~ = [Dr | Ds | LIFT] [f~_0; f~_1; F~ - f~perp], into qf, then out
    warp_gemm_3xtf32<NU, 2 * NU + NF>(
        ncol,
        [&](int i, int k) { return k < NU ? op.Dr[i][k] : (k < 2 * NU ? op.Ds[i][k - NU] : op.LIFT[i][k - 2 * NU]); },
        [&](int c, int k) {
          return k < 2 * NU ? q[(c * 2 + (k >= NU)) * NU + (k < NU ? k : k - NU)] : cor[c * NF + k - 2 * NU];
        },
        [&](int c, int i, float v) { qf[c * NU + i] = v; });
    __syncthreads();
    for (int idx = tid; idx < ncol * NU; idx += blockDim.x) {
      const int el = idx / (NFLD * NU), r = idx % (NFLD * NU), fld = r / NU, i = r % NU;
      T div = qf[idx];
      if (MODE == 1) div -= us[el * NU + i];
      rp[((e0 + el) * 2 + F0 + fld) * NU + i] = div;
    }
  } else {
    for (int idx = tid; idx < ne * NFLD * NU; idx += blockDim.x) {
      const int el = idx / (NFLD * NU), r = idx % (NFLD * NU), fld = r / NU, i = r % NU;
      const T* f0 = q + ((el * NFLD + fld) * 2 + 0) * NU;
      const T* f1 = q + ((el * NFLD + fld) * 2 + 1) * NU;
      const T* cr = cor + (el * NFLD + fld) * NF;
      T div = 0;
#pragma unroll
      for (int j = 0; j < NU; ++j) div += op.Dr[i][j] * f0[j] + op.Ds[i][j] * f1[j];
#pragma unroll
      for (int k = 0; k < NF; ++k) div += op.LIFT[i][k] * cr[k];
      if (MODE == 1) div -= us[el * NU + i];
      rp[((e0 + el) * 2 + F0 + fld) * NU + i] = div;
    }
  }
  (void)N;
}

template <int P, typename T, int MODE, bool TC = false, int TD = 1>
struct KATriLayout {
  using S = TriS<P>;
  static constexpr int NFLD = MODE == 0 ? 2 : 1;
  static constexpr bool FLT = std::is_same<T, float>::value;
  static constexpr bool MMA = TC && FLT;
  static constexpr bool CONS = FLT && MODE == 0;  // mixed-path flux balance
  // + the float path's [ET][NFLD][NU] lift / increment buffer and, for the
  // flux balance, the float-float states [ET][2][NU]
  static constexpr int BYTES_EL = (NFLD * S::NU + NFLD * S::NF + S::NG + 1 + (FLT ? NFLD * S::NU : 0)) * (int)sizeof(T) +
                                  (CONS ? 2 * S::NU * 8 : 0);
  static constexpr int HEAD_EL = (NFLD * S::NU + NFLD * S::NF + S::NG + 1 + (FLT ? NFLD * S::NU : 0));  // T values before u2s
  static constexpr int ETr = 16384 / BYTES_EL;
  static constexpr int ET1 = ETr < 1 ? 1 : (ETr > 128 ? 128 : ETr);
  static constexpr int ET = ET1 / TD < 1 ? 1 : ET1 / TD;
  static constexpr size_t SMEM = (size_t)ET * BYTES_EL + sizeof(TriOpsS<P, T>) + 64 + 16;  // + u2s alignment
};

template <int P, typename T, int MODE, bool TC = false, int TD = 1>
__global__ void __launch_bounds__(kThreads) ka_tri(const KArgs A) {
  using S = TriS<P>;
  using LY = KATriLayout<P, T, MODE, TC, TD>;
  constexpr int NU = S::NU, NF = S::NF, NG = S::NG, NFLD = LY::NFLD, ET = LY::ET;
  constexpr int F0 = MODE == 0 ? 0 : 1;
  if (MODE == 1 && *(volatile int32_t*)&A.status[ST_PSEUDO_DONE]) return;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red_sh[32];
  TriOpsS<P, T>& op = *reinterpret_cast<TriOpsS<P, T>*>(smem_raw);
  T* base = reinterpret_cast<T*>(smem_raw + ((sizeof(TriOpsS<P, T>) + 15) & ~size_t(15)));
  T* ys = base;
  T* cr = ys + ET * NFLD * NU;
  T* gs = cr + ET * NFLD * NF;
  T* djs = gs + ET * NG;
  T* lf = djs + ET;                     // float path: LIFT c, then the RK increments, [ET][NFLD][NU]
  // [ET][2][NU] float-float states of the flux balance, on a 16-byte boundary
  float2* u2s = reinterpret_cast<float2*>(
      (reinterpret_cast<uintptr_t>(base + ET * LY::HEAD_EL) + 15) & ~static_cast<uintptr_t>(15));
  constexpr bool kMMA = LY::MMA;
  // Mixed path: each element's float-float solution is shifted at stage 4 so
  // that its quadrature-weighted mass change equals the RK4-weighted sum of
  // its edge fluxes, -sum_k w_k F_out,k with w_k the physical edge weight
  // shared bitwise by both sides; the global mass then changes only through
  // walls (as in ka_tensor).
  constexpr bool kCons = LY::CONS;
  __shared__ double tgt[kCons ? 2 * ET : 1];
  __shared__ float dlt[kCons ? 4 * ET : 1];

  const int64_t e0 = (int64_t)blockIdx.x * ET;
  const int ne = (int)min((int64_t)ET, A.E - e0);
  T* ustg = reinterpret_cast<T*>(A.ustg);
  T* tr = reinterpret_cast<T*>(A.tr);
  const T* fc = reinterpret_cast<const T*>(A.fc);
  const T* rp = reinterpret_cast<const T*>(A.rp);
  const int tid = threadIdx.x;
  const int stage = A.stage;

  load_tri_ops<P, T>(tri_of<T>(A), op);
  for (int idx = tid; idx < ne * NG; idx += blockDim.x) gs[idx] = geo_of<T>(A)[e0 * NG + idx];
  for (int idx = tid; idx < ne * NFLD * NU; idx += blockDim.x) {
    const int el = idx / (NFLD * NU), r = idx % (NFLD * NU), fld = r / NU, i = r % NU;
    const int64_t g = ((e0 + el) * 2 + F0 + fld) * NU + i;
    ys[idx] = stage == 0 ? ustg[g] : rp[g];
  }
  __syncthreads();
  double sq = 0.0;
  const RKConstF& rkc = A.rk;
  if (stage != 0) {
    for (int el = tid; el < ne; el += blockDim.x) {
      TriMet<T> m;
      tri_metric(gs + el * NG, m);
      djs[el] = m.dj;
    }
    for (int idx = tid; idx < ne * NF; idx += blockDim.x) {
      const int el = idx / NF, k = idx % NF;
      const int32_t w = A.fnbr[(e0 + el) * NF + k];
      if (w & 1) {
#pragma unroll
        for (int fld = 0; fld < NFLD; ++fld) cr[(el * NFLD + fld) * NF + k] = 0;
        continue;
      }
      const int64_t pg = (int64_t)partner<NF>(A, w, (int32_t)((e0 + el) * NF + k)), pe = pg / NF, pk = pg % NF;
      TriMet<T> m;
      tri_metric(gs + el * NG, m);
      const T pn0 = m.S[0][0] * op.nref[k][0] + m.S[1][0] * op.nref[k][1];
      const T pn1 = m.S[0][1] * op.nref[k][0] + m.S[1][1] * op.nref[k][1];
      const T pm = sqrt_(pn0 * pn0 + pn1 * pn1);
#pragma unroll
      for (int fld = 0; fld < NFLD; ++fld)
        cr[(el * NFLD + fld) * NF + k] = -pm * fc[(pe * 2 + F0 + fld) * NF + pk];
    }
    __syncthreads();
    if constexpr (kMMA) {
      warp_gemm_3xtf32<NU, NF>(
          ne * NFLD, [&](int r, int k) { return op.LIFT[r][k]; }, [&](int c, int k) { return cr[c * NF + k]; },
          [&](int c, int r, float v) { lf[c * NU + r] = v; });
      __syncthreads();
    }
    const bool cons = kCons && A.tacc && A.wphys && stage >= 1;
    if (cons) {
      // element flux balance T = -sum_k w_k F_out,k (float-float), RK4-accumulated in FP64
      for (int t = tid; t < ne * 2; t += blockDim.x) {
        const int el = t / 2, fld = t % 2;
        float2 bsum = make_float2(0.f, 0.f);
        for (int k = 0; k < NF; ++k) {
          const int64_t og = (e0 + el) * NF + k;
          const int32_t w = A.fnbr[og];
          const int64_t pg = (int64_t)partner<NF>(A, w, (int32_t)og);
          const float Fo = (w & 1) ? (float)fc[((e0 + el) * 2 + fld) * NF + k]
                                   : -(float)fc[((pg / NF) * 2 + fld) * NF + pg % NF];
          bsum = ff_add(bsum, ff_mul(A.wphys[og], Fo));
        }
        const double Te = -((double)bsum.x + (double)bsum.y);
        const int64_t gt = (e0 + el) * 2 + fld;
        if (stage == 1) A.tacc[gt] = Te;
        else if (stage < 4) A.tacc[gt] = A.tacc[gt] + 2.0 * Te;
        else tgt[t] = rkc.ddt6 * (A.tacc[gt] + Te);
      }
    }
    for (int idx = tid; idx < ne * NFLD * NU; idx += blockDim.x) {
      const int el = idx / (NFLD * NU), r = idx % (NFLD * NU), fld = r / NU, i = r % NU;
      T div = ys[idx];
      if constexpr (kMMA) {
        div += lf[idx];
      } else {
        const T* c = cr + (el * NFLD + fld) * NF;
#pragma unroll
        for (int k = 0; k < NF; ++k) div += op.LIFT[i][k] * c[k];
      }
      const T R = -div / djs[el];
      const int64_t g = ((e0 + el) * 2 + F0 + fld) * NU + i;
      if (stage < 0) {
        A.out[(int64_t)fld * A.E * NU + (e0 + el) * NU + i] = (double)R;
        continue;
      }
      if constexpr (kCons) {
        if (cons && stage == 4) {
          // float-float update now, the element's uniform shift below
          const float2 u = reinterpret_cast<const float2*>(A.u)[g];
          const float inc = rkc.dt6 * (reinterpret_cast<const float*>(A.acc)[g] + (float)R);
          const float s2 = u.x + inc;
          const float e2 = two_sum_lo(u.x, inc, s2) + u.y;
          const float hi = s2 + e2;
          u2s[idx] = make_float2(hi, e2 - (hi - s2));
          lf[idx] = inc;
          continue;
        }
      }
      const T yt = rk_apply(A, stage, g, R, rkc, (MODE == 1 && stage == 4) ? &sq : nullptr);
      if (!isfinite(yt)) atomicExch(&A.status[ST_STATUS], -4);
      ustg[g] = yt;
      ys[idx] = yt;
    }
    __syncthreads();
    if (kCons && cons && stage == 4) {
      for (int t = tid; t < ne * 2; t += blockDim.x) {
        const int el = t / 2;
        float2 S2 = make_float2(0.f, 0.f);
        double W = 0.0;
        for (int i = 0; i < NU; ++i) {
          const float2 wd = A.wdetf[(e0 + el) * NU + i];
          S2 = ff_add(S2, ff_mul(wd, (float)lf[t * NU + i]));
          W += (double)wd.x + (double)wd.y;
        }
        const double d = (tgt[t] - ((double)S2.x + (double)S2.y)) / W;
        const float dh = (float)d;
        dlt[2 * t] = dh;
        dlt[2 * t + 1] = (float)(d - (double)dh);
      }
      __syncthreads();
      for (int idx = tid; idx < ne * NFLD * NU; idx += blockDim.x) {
        const int el = idx / (NFLD * NU), r = idx % (NFLD * NU), fld = r / NU, i = r % NU;
        const int64_t g = ((e0 + el) * 2 + F0 + fld) * NU + i;
        const float2 u = u2s[idx];
        const float dh = dlt[2 * (el * 2 + fld)], dl = dlt[2 * (el * 2 + fld) + 1];
        const float s2 = u.x + dh;
        const float e2 = two_sum_lo(u.x, dh, s2) + (u.y + dl);
        const float hi = s2 + e2;
        reinterpret_cast<float2*>(A.u)[g] = make_float2(hi, e2 - (hi - s2));
        if (!isfinite(hi)) atomicExch(&A.status[ST_STATUS], -4);
        ustg[g] = (T)hi;
        ys[idx] = (T)hi;
      }
      __syncthreads();
    }
  }
  if (stage >= 0) {
    if constexpr (kMMA) {
      warp_gemm_3xtf32<NF, NU>(
          ne * NFLD, [&](int r, int k) { return op.L[r][k]; }, [&](int c, int k) { return ys[c * NU + k]; },
          [&](int c, int r, float v) { tr[((e0 + c / NFLD) * 2 + F0 + c % NFLD) * NF + r] = v; });
    } else {
      for (int idx = tid; idx < ne * NFLD * NF; idx += blockDim.x) {
        const int el = idx / (NFLD * NF), r = idx % (NFLD * NF), fld = r / NF, k = r % NF;
        const T* yl = ys + (el * NFLD + fld) * NU;
        T acc = 0;
#pragma unroll
        for (int j = 0; j < NU; ++j) acc += op.L[k][j] * yl[j];
        tr[((e0 + el) * 2 + F0 + fld) * NF + k] = acc;
      }
    }
  }
  if (MODE == 0 && stage == 4 && A.use_dev_time && blockIdx.x == 0 && tid == 0)
    A.dstate[DS_TIME] = A.dstate[DS_TIME] + A.dt;
  if (MODE == 1 && stage == 4) pseudo_rms_finish(A, block_sum(sq, red_sh), red_sh, A.E * NU);
}

// Spatial velocity factor v(x) (g = 1) at the solution and flux points of
// every triangle, evaluated once in double (exact zeros where the analytic
// field vanishes, as on the walls of the benchmark flows) and stored in the
// bulk type: vsu [E][2][NU], vsf [E][2][NF].
template <int P, typename T>
__global__ void k_vel_cache_tri(const KArgs A) {
  using S = TriS<P>;
  constexpr int NU = S::NU, NF = S::NF, NG = S::NG;
  const int64_t n = A.E * (NU + NF);
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < n; g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = g / (NU + NF);
    const int r = (int)(g % (NU + NF));
    const double* xr = r < NU ? A.trid.xu + 2 * r : A.trid.xf + 2 * (r - NU);
    const double xi[2] = {xr[0], xr[1]};
    double x[3], v[3];
    map_point<ET_TRI, double>(A.geo + e * NG, xi, x);
    velocity<2, double>(A.cd.vel, x, 1.0, v);
    if (r < NU) {
      T* o = reinterpret_cast<T*>(const_cast<void*>(A.vsu)) + e * 2 * NU + r;
      o[0] = (T)v[0];
      o[NU] = (T)v[1];
    } else {
      T* o = reinterpret_cast<T*>(const_cast<void*>(A.vsf)) + e * 2 * NF + (r - NU);
      o[0] = (T)v[0];
      o[NF] = (T)v[1];
    }
  }
}

}  // namespace frp
