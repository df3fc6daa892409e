// Warp-per-element kernels of the mixed path's preconditioning stage (psi alone,
// Eq. pseudotimesystem) on quadrilaterals and hexahedra, organised as the
// physical step's (kline.cuh): MODE 1 of kb_tensor and ka_tensor.
//
// The block-wide kernels spent most of their time in FP64: the modal energies
// of the resolution indicator as one thread's serial sum per element, and nine
// instructions a point for the pseudo-time residual, on a pipe of 2 lanes a
// clock.  Here the energies are float-float sums over the lanes, the indicator's
// logarithm and sine are evaluated in float-float (sensor_nu), and of the
// residual only the sum of squares is FP64, two instructions a point: in
// float-float its squares would leave the floats' range with psi.
#pragma once
#include "kline.cuh"

namespace frp {

// rows of one field whose elements are `pitch` floats apart, through a
// warp-private buffer with unit stride over the lanes (N other than 2 and 4)
template <int NU>
__device__ __forceinline__ void rows_fetch(float* dst, const float* src, int pitch, int ne, int lane) {
  for (int i = lane; i < ne * NU; i += 32) cp_async_4(dst + i, src + (i / NU) * pitch + i % NU);
}
template <int NU>
__device__ __forceinline__ void rows_flush(float* dst, const float* src, int pitch, int ne, int lane) {
  for (int i = lane; i < ne * NU; i += 32) dst[(i / NU) * pitch + i % NU] = src[i];
}

template <int DIM, int N, bool GEN>
struct KBPLine {
  using L = LL<DIM, N>;
  static constexpr int WARP_F = (2 + DIM) * L::AS * L::EPW;  // psi, modes, gradient
  static constexpr int IN_F = L::DIRECT ? 0 : (L::EPW * L::NU + 3) / 4 * 4;
  static constexpr int O_GEO = (WARP_F + 3) / 4 * 4 + IN_F;
  static constexpr int F = O_GEO + (GEN ? L::EPW * L::S::NG : 0);
  static_assert(O_GEO % 4 == 0 && F % 4 == 0, "16-byte boundaries");
};

// quotient of two float-float values
__device__ __forceinline__ float2 ff_div(float2 a, float2 b) {
  const float q = a.x / b.x;
  const float r = (__fmaf_rn(-q, b.x, a.x) + a.y) - q * b.y;
  const float l = r / b.x;
  const float h = q + l;
  return make_float2(h, l - (h - q));
}

// The power of two that brings the largest magnitude of an element's modal
// coefficients (given by its bits) to [1, 4): the ratio of the energies does not
// depend on it, the scaling is exact, and no square of a coefficient of any
// size overflows or is lost beside the largest one's.
__device__ __forceinline__ float energy_scale(unsigned bits) {
  return __int_as_float((int)(254u - min(bits >> 23, 253u)) << 23);
}
__device__ __forceinline__ unsigned abs_bits(float v) { return __float_as_uint(v) & 0x7fffffffu; }
// Maximum over the LN lanes of an element; every lane gets it.  first: the element's first lane.
template <int LN>
__device__ __forceinline__ unsigned line_max(unsigned v, int l, int first) {
  if constexpr ((LN & (LN - 1)) == 0) {
#pragma unroll
    for (int o = LN / 2; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
  } else {
    constexpr int TOP = LN > 16 ? 16 : LN > 8 ? 8 : LN > 4 ? 4 : LN > 2 ? 2 : 1;
#pragma unroll
    for (int o = TOP; o > 0; o >>= 1) {
      const unsigned t = __shfl_down_sync(0xffffffffu, v, o);
      if (l + o < LN) v = max(v, t);
    }
    return __shfl_sync(0xffffffffu, v, first);
  }
}

// nu_s of Eqs. resolutionIndicator, nu_s from the energies of the modes below
// and at the top degree, evaluated in float-float.  With r = hi / (lo + hi) and
// z = (pi / 2) (log10 r - (s0 - kappa)) / (2 kappa), the ramp
// (1 + sin(pi (log10 r - s0) / (2 kappa))) / 2 is sin^2 z.  The logarithm is the
// series 2 (t + t^3 / 3 + ...) of the significand m in [1/sqrt 2, sqrt 2),
// t = (m - 1) / (m + 1), and the sine its Taylor series up to pi / 4, both with
// the leading terms in float-float: nu_s is as close to the exact value as the
// rounded FP64 evaluation (worst 5.953e-8 to 5.958e-8, mean 2.05e-8 to 2.20e-8
// for p = 1..6, equal to six and seven digits; 99.995 % of the results are equal).
// log10 and sin in FP64 took a warp 3000 cycles of the FP64 pipe wherever one of
// its elements lies in the ramp.
__device__ __forceinline__ float sensor_nu(const PhysPrm& P, float2 lo, float2 hi, float2 nu_max) {
  const float tot = lo.x + hi.x;
  if (!(tot > 0.f) || !(hi.x > 0.f)) return 0.f;
  if (hi.x < P.ramp_lo * tot) return 0.f;  // most elements: flat or resolved
  float2 r = ff_div(hi, ff_add(lo, hi));
  if (r.x < 0x1p-126f) r = make_float2(0x1p-126f, 0.f);  // a ramp that reaches below the floats
  // r = m 2^k
  int k = (__float_as_int(r.x) >> 23) - 127;
  float mh = __int_as_float((__float_as_int(r.x) & 0x007fffff) | 0x3f800000);
  if (mh > 1.41421356f) {
    mh *= 0.5f;
    ++k;
  }
  const float sc = mh / r.x;  // a power of two
  const float2 m = make_float2(mh, r.y * sc);
  const float2 t = ff_div(ff_add(m, make_float2(-1.f, 0.f)), ff_add(m, make_float2(1.f, 0.f)));
  const float2 t3 = ff_mul2(ff_mul2(t, t), t);
  const float t2 = t.x * t.x;
  float ps = __fmaf_rn(t2, 1.f / 13.f, 1.f / 11.f);
  ps = __fmaf_rn(t2, ps, 1.f / 9.f);
  ps = __fmaf_rn(t2, ps, 1.f / 7.f);
  ps = __fmaf_rn(t2, ps, 1.f / 5.f);
  const float2 third = make_float2(0.333333343f, -9.93410776e-9f);
  const float2 half_log = ff_add(t, ff_add(ff_mul2(t3, third), make_float2(t3.x * t2 * ps, 0.f)));
  // z = C0 + k C1 + half_log C2
  float2 z = ff_add(ff_mul2(make_float2(P.ramp_c1h, P.ramp_c1l), make_float2((float)k, 0.f)),
                    ff_mul2(make_float2(P.ramp_c2h, P.ramp_c2l), half_log));
  z = ff_add(z, make_float2(P.ramp_c0h, P.ramp_c0l));
  const float2 hpi = make_float2(1.57079637f, -4.37113883e-8f);
  if (z.x <= 0.f) return 0.f;
  if (z.x >= hpi.x) return nu_max.x;
  const bool up = z.x > 0.785398163f;
  if (up) z = ff_add(hpi, make_float2(-z.x, -z.y));  // sin^2 z = 1 - sin^2(pi/2 - z)
  const float2 z2 = ff_mul2(z, z), z3 = ff_mul2(z2, z);
  float s = __fmaf_rn(z2.x, -1.f / 39916800.f, 1.f / 362880.f);
  s = __fmaf_rn(z2.x, s, -1.f / 5040.f);
  const float2 sixth = make_float2(-0.166666672f, 4.96705388e-9f), c5 = make_float2(0.00833333377f, -4.34617203e-10f);
  const float2 z35 = ff_add(sixth, ff_add(ff_mul2(z2, c5), make_float2(z2.x * z2.x * s, 0.f)));
  float2 v = ff_add(z, ff_mul2(z3, z35));
  v = ff_mul2(v, v);
  if (up) v = ff_add(make_float2(1.f, 0.f), make_float2(-v.x, -v.y));
  v = ff_mul2(v, nu_max);
  return v.x + v.y;
}

template <int DIM, int N, bool GEN, int WPB>
__global__ void __launch_bounds__(WPB * 32, (!GEN ? 24 : DIM == 3 ? 16 : 20) / WPB) kbp_line(const KArgs A) {
  using L = LL<DIM, N>;
  using K = KBPLine<DIM, N, GEN>;
  constexpr int NU = L::NU, NF = L::NF, NFP = L::NFP, LN = L::LN, EPW = L::EPW, NP = L::NP, AS = L::AS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* wsm = reinterpret_cast<float*>(smem_raw) + warp * K::F;
  float* in = wsm + (K::WARP_F + 3) / 4 * 4;
  const int es = L::FULL ? lane / LN : min(lane / LN, EPW - 1), l = lane - (lane / LN) * LN;
  const bool lane_ok = L::FULL || lane < EPW * LN;
  const int64_t e0 = ((int64_t)blockIdx.x * WPB + warp) * EPW;
  const int64_t eraw = e0 + es;
  const bool act = lane_ok && eraw < A.E;
  const int64_t e = eraw < A.E ? eraw : A.E - 1;
  const int ne = (int)max((int64_t)0, min((int64_t)EPW, A.E - e0));
  const float* trA = reinterpret_cast<const float*>(A.tr);
  const LineOps& O = A.lo;
  const PrmT<float>& P = A.cf.prm;

  // ---- loads
  if (GEN && ne > 0) tile_fetch<EPW, L::S::NG * 4>(wsm + K::O_GEO, A.geof + e0 * L::S::NG, ne, lane);
  int fl[DIM][2];
  [[maybe_unused]] int2 fw[DIM][2];
  [[maybe_unused]] int32_t w2[DIM][2];
#pragma unroll
  for (int a = 0; a < DIM; ++a)
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if constexpr (DIM == 3) fw[a][s] = __ldg(A.ffw + e * 6 + 2 * a + s);
      else w2[a][s] = __ldg(A.fnbr + e * NF + (2 * a + s) * NFP + l);
    }
  float p0[N];
  if constexpr (N % 2 == 0) {
#pragma unroll
    for (int j = 0; j < N; j += 2) {
      const double2 t = *reinterpret_cast<const double2*>(A.psi0 + e * NU + l * N + j);
      p0[j] = (float)t.x;
      p0[j + 1] = (float)t.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) p0[j] = (float)A.psi0[e * NU + l * N + j];
  }
  const float* mc = reinterpret_cast<const float*>(A.mcg) + e * kMetricRec;
  const bool diag = !GEN || __ldg(mc + 11) == 2.f;
  float sd[DIM];
#pragma unroll
  for (int a = 0; a < DIM; ++a) sd[a] = __ldg(mc + a * 4);
  const float det = __ldg(mc + 9), rdet = __ldg(mc + 10);
  if (*(volatile int32_t*)&A.status[ST_PSEUDO_DONE]) {
    if (GEN) cp_async_wait_all();  // no copy in flight outlives its block
    return;
  }
  float2 u[NP], o[DIM];
  const float* ug = reinterpret_cast<const float*>(A.ustg);
  if constexpr (L::DIRECT) grow_get<N>(ug + (e * 2 + 1) * NU + l * N, u);
  else rows_fetch<NU>(in, ug + (e0 * 2 + 1) * NU, 2 * NU, ne, lane);
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    float t[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int k = (2 * a + s) * NFP + l;
      if constexpr (DIM == 3) {
        const int32_t po = face_link<N, NF>(A, fw[a][s], e, 2 * a + s, l % N, l / N, fl[a][s]);
        t[s] = (fl[a][s] & (kFwL | kFwWall)) == kFwL ? trA[po + NF] : 0.f;
      } else {
        t[s] = trA[e * 2 * NF + NF + k];
        fl[a][s] = (w2[a][s] & 1) | ((w2[a][s] >> 1) == (int32_t)(e * NF + k) ? kFwWall : 0);
      }
    }
    o[a] = make_float2(t[0], t[1]);
  }
  if constexpr (!L::DIRECT) {
    cp_async_wait_all();
    __syncwarp();
    grow_get<N>(in + es * NU + l * N, u);
  }
  if (GEN) cp_async_wait_all();

  constexpr int FA = AS * EPW;
  float* U = wsm + es * AS;
  float* C = U + FA;       // modal coefficients
  float* Q = U + 2 * FA;   // [a]: + a FA

  // ---- Steps 1-3 and the modal transform, axis 0 from registers
  float2 tr[DIM], q[DIM][NP], qe[DIM];
  float sc[DIM];
#pragma unroll
  for (int a = 0; a < DIM; ++a) sc[a] = diag ? __fmul_rn(sd[a], rdet) : 1.f;
  float cm[N];  // modes along the last axis of the lane's line
  {
    float v[N];
    unpair<N>(u, v);
    float2 c[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      c[p] = mul2(O.V[0][p], dup2(v[0]));
#pragma unroll
      for (int m = 1; m < N; ++m) c[p] = fma2(O.V[m][p], dup2(v[m]), c[p]);
    }
    if (lane_ok) {
      row_put<NP, L::V4>(U + pline<DIM, N>(0, l), u);
      row_put<NP, L::V4>(C + pline<DIM, N>(0, l), c);
    }
  }
  __syncwarp();
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    float v[N];
    if (a == 0) unpair<N>(u, v);
    else if (a == 1) line_get<N, pstride<DIM, N>(1)>(U + pline<DIM, N>(1, l), v);
    else line_get<N, pstride<DIM, N>(2)>(U + pline<DIM, N>(2, l), v);
    const float2 t = line_ends<N>(O, v);
    tr[a] = t;
    float2 ot = o[a];
    ot.x = (fl[a][0] & (kFwL | kFwWall)) == kFwL ? ot.x : t.x;
    ot.y = (fl[a][1] & (kFwL | kFwWall)) == kFwL ? ot.y : t.y;
    o[a] = ot;
    float2 d[NP];
    line_deriv<N>(O, v, O.gL, O.gR, sub2(ot, t), d);
#pragma unroll
    for (int p = 0; p < NP; ++p) d[p] = mul2(d[p], dup2(sc[a]));
    float s[N];
    unpair<N>(d, s);
    qe[a] = line_ends<N>(O, s);
    if (a == 0) {
#pragma unroll
      for (int p = 0; p < NP; ++p) q[0][p] = d[p];
    } else if (lane_ok) {
      float* dst = Q + a * FA + pline<DIM, N>(a, l);
      if (a == 1) line_put<N, pstride<DIM, N>(1)>(dst, d);
      else line_put<N, pstride<DIM, N>(2)>(dst, d);
    }
    if (a > 0) {
      if (a == 2) __syncwarp();  // axis 1's modes are in
      float w[N];
      float* cl = C + pline<DIM, N>(a, l);
      if (a == 1) line_get<N, pstride<DIM, N>(1)>(cl, w);
      else line_get<N, pstride<DIM, N>(2)>(cl, w);
      float2 c[NP];
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        c[p] = mul2(O.V[0][p], dup2(w[0]));
#pragma unroll
        for (int m = 1; m < N; ++m) c[p] = fma2(O.V[m][p], dup2(w[m]), c[p]);
      }
      if (a < DIM - 1) {
        if (lane_ok) line_put<N, pstride<DIM, N>(1)>(cl, c);
      } else {
        unpair<N>(c, cm);
      }
    }
  }
  // ---- resolution indicator: energies of the modes below the top degree (a
  //      lane's line holds modes (its two indices, 0..N-1)) and at it
  float nu;
  {
    const int src = L::FULL ? es * LN : min(es * LN, 31);
    unsigned big = 0;
#pragma unroll
    for (int m = 0; m < N; ++m) big = max(big, abs_bits(cm[m]));
    const float unit = energy_scale(line_max<LN>(big, l, src));
#pragma unroll
    for (int m = 0; m < N; ++m) cm[m] *= unit;
    const bool top = DIM == 3 ? (l % N == N - 1 || l / N == N - 1) : l == N - 1;
    float2 b = make_float2(0.f, 0.f), t;
#pragma unroll
    for (int m = 0; m < N - 1; ++m) {
      const float p = __fmul_rn(cm[m], cm[m]);
      b = ff_add(b, make_float2(p, __fmaf_rn(cm[m], cm[m], -p)));
    }
    {
      const float p = __fmul_rn(cm[N - 1], cm[N - 1]);
      t = make_float2(p, __fmaf_rn(cm[N - 1], cm[N - 1], -p));
    }
    float2 hi = top ? ff_add(t, b) : t, lo = top ? make_float2(0.f, 0.f) : b;
    if (!lane_ok) hi = lo = make_float2(0.f, 0.f);
    line_tree<LN>(lo, hi, l);
    const float2 h0 = make_float2(__shfl_sync(0xffffffffu, hi.x, src + LineTree<LN>::LB),
                                  __shfl_sync(0xffffffffu, hi.y, src + LineTree<LN>::LB));
    nu = 0.f;
    if (lane_ok && l == 0) {
      float2 nm = make_float2(A.prm.nu_h, A.prm.nu_l);
      if (A.ep) {
        const double d = A.ep[e].nu_max;
        nm.x = (float)d;
        nm.y = (float)(d - (double)nm.x);
      }
      nu = sensor_nu(A.prm, lo, h0, nm);
    }
    nu = __shfl_sync(0xffffffffu, nu, src);
  }
  __syncwarp();
#pragma unroll
  for (int a = 1; a < DIM; ++a) row_get<NP, L::V4>(Q + a * FA + pline<DIM, N>(0, l), q[a]);

  const int lc1 = DIM == 3 ? l % N : l, lc2 = DIM == 3 ? l / N : 0;
  const float* geo = wsm + K::O_GEO + es * L::S::NG;
  float2 xi[3];
  xi[1] = dup2(A.cf.ops.x[lc1]);
  xi[2] = dup2(A.cf.ops.x[lc2]);
  if (GEN && !diag) {
    // physical gradient, kept in registers and in the rows
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      float2 Sm[3][3], r[3];
      xi[0] = O.xp[p];
      const float2 rdj = rcp2(metric_all<DIM>(geo, xi, Sm));
#pragma unroll
      for (int b = 0; b < DIM; ++b) {
        r[b] = mul2(Sm[0][b], q[0][p]);
#pragma unroll
        for (int a = 1; a < DIM; ++a) r[b] = fma2(Sm[a][b], q[a][p], r[b]);
        r[b] = mul2(r[b], rdj);
      }
#pragma unroll
      for (int b = 0; b < DIM; ++b) q[b][p] = r[b];
    }
    if (lane_ok) {
#pragma unroll
      for (int b = 0; b < DIM; ++b) row_put<NP, L::V4>(Q + b * FA + pline<DIM, N>(0, l), q[b]);
    }
  }
  if (GEN) __syncwarp();

  // ---- Step 5
  const float2 nnu = dup2(-nu);
  float2 cor[DIM];
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    const float2 dp = sub2(tr[a], o[a]);
    float2 F;
    if (diag) {
      F = fma2(dup2(__fmul_rn(fabsf(sd[a]), P.tau_pseudo)), dp,
               mul2(mul2(make_float2(-sd[a], sd[a]), nnu), qe[a]));
    } else if (GEN) {
      float2 xf[3], Sr[3];
      {
        int i = 0;
#pragma unroll
        for (int b = 0; b < DIM; ++b) {
          if (b == a) {
            xf[b] = make_float2(-1.f, 1.f);
          } else {
            xf[b] = dup2(A.cf.ops.x[i == 0 ? (DIM == 2 ? l : l % N) : l / N]);
            ++i;
          }
        }
      }
      metric_row<DIM>(geo, a, xf, Sr);
      float2 gn = dup2(0.f), pm2 = dup2(0.f);
#pragma unroll
      for (int c = 0; c < DIM; ++c) {
        float v[N];
        if (a == 0) unpair<N>(q[c], v);
        else if (a == 1) line_get<N, pstride<DIM, N>(1)>(Q + c * FA + pline<DIM, N>(1, l), v);
        else line_get<N, pstride<DIM, N>(2)>(Q + c * FA + pline<DIM, N>(2, l), v);
        const float2 pn = mul2(make_float2(-1.f, 1.f), Sr[c]);
        gn = fma2(line_ends<N>(O, v), pn, gn);
        pm2 = fma2(pn, pn, pm2);
      }
      const float2 pm = make_float2(sqrtf(pm2.x), sqrtf(pm2.y));
      F = fma2(mul2(pm, dup2(P.tau_pseudo)), dp, mul2(nnu, gn));
    }
    const bool l0 = fl[a][0] & kFwL, l1 = fl[a][1] & kFwL;
    F = make_float2(l0 ? F.x : 0.f, l1 ? F.y : 0.f);
    cor[a] = F;
    if (act) {
      const int k0 = 2 * a * NFP + l;
      float* fcE = reinterpret_cast<float*>(A.fc) + e * 2 * NF + NF;
      if (l0) fcE[k0] = F.x;
      if (l1) fcE[k0 + NFP] = F.y;
      if constexpr (FaceScatter<DIM>::v) {
#pragma unroll
        for (int s = 0; s < 2; ++s)
          if ((fl[a][s] & (kFwL | kFwWall)) == kFwL) {
            const int32_t pg = partner<NF>(A, w2[a][s], (int32_t)(e * NF + k0 + s * NFP));
            reinterpret_cast<float*>(A.fc)[(int64_t)(pg / NF) * 2 * NF + NF + pg % NF] = s ? F.y : F.x;
          }
      }
    }
  }
  if (GEN) __syncwarp();  // the faces have read the gradient rows

  // ---- Step 4 and the smeared-sign source
  float2 fx[NP], src[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    float2 g2 = mul2(q[0][p], q[0][p]);
#pragma unroll
    for (int c = 1; c < DIM; ++c) g2 = fma2(q[c][p], q[c][p], g2);
    const float2 qm = make_float2(sqrtf(g2.x), sqrtf(g2.y));
    float2 dj = dup2(det), t[3];
    if (diag) {
#pragma unroll
      for (int a = 0; a < DIM; ++a) t[a] = mul2(mul2(dup2(sd[a]), nnu), q[a][p]);
    } else if (GEN) {
      float2 Sm[3][3];
      xi[0] = O.xp[p];
      dj = metric_all<DIM>(geo, xi, Sm);
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        t[a] = mul2(Sm[a][0], q[0][p]);
#pragma unroll
        for (int c = 1; c < DIM; ++c) t[a] = fma2(Sm[a][c], q[c][p], t[a]);
        t[a] = mul2(t[a], nnu);
      }
    }
    fx[p] = t[0];
#pragma unroll
    for (int a = 1; a < DIM; ++a) q[a][p] = t[a];
    const float s0 = tanhf(p0[2 * p] / fmaxf(qm.x, P.delta));
    const float s1 = 2 * p + 1 < N ? tanhf(p0[2 * p + 1 < N ? 2 * p + 1 : 0] / fmaxf(qm.y, P.delta)) : 0.f;
    src[p] = mul2(mul2(make_float2(s0, s1), sub2(dup2(1.f), qm)), dj);
  }
  if (lane_ok) {
#pragma unroll
    for (int a = 1; a < DIM; ++a) row_put<NP, L::V4>(Q + a * FA + pline<DIM, N>(0, l), q[a]);
  }
  __syncwarp();

  // ---- Step 6
  float2 dv[NP];
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    float v[N];
    float* s = Q + a * FA + pline<DIM, N>(a, l);
    if (a == 0) unpair<N>(fx, v);
    else if (a == 1) line_get<N, pstride<DIM, N>(1)>(s, v);
    else line_get<N, pstride<DIM, N>(2)>(s, v);
    const float2 c = fma2(line_ends<N>(O, v), make_float2(1.f, -1.f), cor[a]);
    float2 d[NP];
    line_deriv<N>(O, v, O.ngL, O.gR, c, d);
    if (a == 0) {
#pragma unroll
      for (int p = 0; p < NP; ++p) dv[p] = d[p];
    } else if (lane_ok) {
      if (a == 1) line_put<N, pstride<DIM, N>(1)>(s, d);
      else line_put<N, pstride<DIM, N>(2)>(s, d);
    }
  }
  __syncwarp();
#pragma unroll
  for (int a = 1; a < DIM; ++a) {
    float2 t[NP];
    row_get<NP, L::V4>(Q + a * FA + pline<DIM, N>(0, l), t);
#pragma unroll
    for (int p = 0; p < NP; ++p) dv[p] = add2(dv[p], t[p]);
  }
  // the source, of order one where the divergence is small, last: one rounding of its size (first, the two
  // sums that follow round at its size too, and psi after 20 iterations was 4 % further off on 32^3 hexes p = 4)
#pragma unroll
  for (int p = 0; p < NP; ++p) dv[p] = sub2(dv[p], src[p]);
  float* rp = reinterpret_cast<float*>(A.rp);
  if constexpr (L::DIRECT) {
    if (act) grow_put<N>(rp + (e * 2 + 1) * NU + l * N, dv);
  } else {
    if (lane_ok) grow_put<N>(in + es * NU + l * N, dv);
    __syncwarp();
    rows_flush<NU>(rp + (e0 * 2 + 1) * NU, in, 2 * NU, ne, lane);
  }
}

// ---- update kernel ---------------------------------------------------------------
template <int DIM, int N, bool GEN>
struct KAPLine {
  using L = LL<DIM, N>;
  static constexpr int ROWS_F = (L::AS * L::EPW + 3) / 4 * 4;
  static constexpr int COR_F = ((DIM - 1) * 2 * L::OTH * L::RS * L::EPW + 3) / 4 * 4;
  // input and output buffer of the strided forms: the rate (later the stage value), accumulator, solution pairs
  static constexpr int C = (L::EPW * L::NU + 3) / 4 * 4;
  static constexpr int IN_F = L::DIRECT ? 0 : 4 * C;
  static constexpr int O_GEO = ROWS_F + COR_F + IN_F;
  static constexpr int F = O_GEO + (GEN ? L::EPW * L::S::NG : 0);
  static_assert(O_GEO % 4 == 0 && F % 4 == 0, "16-byte boundaries");
};

// SF: stage 1..4, or 0 to recompute the traces of psi alone.  GEN false: every
// element is affine.
//
// Stage 4 leaves one partial of the residual a block, so its grid is resident
// and every warp walks over tiles (one tile a warp and 8,000 partials cost
// stage 4 of 64,000 hexes p = 3 58.6 us where the other stages take 24); the
// other stages make one pass.
template <int DIM, int N, bool GEN, int WPB, int SF>
__global__ void __launch_bounds__(WPB * 32, 24 / WPB) kap_line(const KArgs A) {
  using L = LL<DIM, N>;
  using K = KAPLine<DIM, N, GEN>;
  constexpr int NU = L::NU, NF = L::NF, NFP = L::NFP, LN = L::LN, EPW = L::EPW, NP = L::NP;
  if (*(volatile int32_t*)&A.status[ST_PSEUDO_DONE]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* R0 = reinterpret_cast<float*>(smem_raw) + warp * K::F;
  float* C0 = R0 + K::ROWS_F;
  float* in = C0 + K::COR_F;
  const int es = L::FULL ? lane / LN : min(lane / LN, EPW - 1), l = lane - (lane / LN) * LN;
  const bool lane_ok = L::FULL || lane < EPW * LN;
  float* ustg = reinterpret_cast<float*>(A.ustg);
  float* acc = reinterpret_cast<float*>(A.acc);
  float2* U = reinterpret_cast<float2*>(A.u);
  const float* fcA = reinterpret_cast<const float*>(A.fc);
  const LineOps& O = A.lo;
  [[maybe_unused]] double sum = 0.0;  // stage 4: squared residuals

#pragma unroll 1
  for (int64_t e0 = ((int64_t)blockIdx.x * WPB + warp) * EPW; e0 < A.E;
       e0 += SF == 4 ? (int64_t)gridDim.x * WPB * EPW : A.E) {
  const int64_t eraw = e0 + es;
  const bool act = lane_ok && eraw < A.E;
  const int64_t e = eraw < A.E ? eraw : A.E - 1;
  const int ne = (int)min((int64_t)EPW, A.E - e0);

  // ---- loads
  float2 y[NP], u[N];
  float ac[N];
  const float* src = SF == 0 ? ustg : reinterpret_cast<const float*>(A.rp);
  const int64_t r = (e * 2 + 1) * NU + l * N;
  if constexpr (L::DIRECT) {
    grow_get<N>(src + r, y);
    if constexpr (SF >= 1) {
#pragma unroll
      for (int j = 0; j < N; j += 2) {
        const float4 t = *reinterpret_cast<const float4*>(U + r + j);
        u[j] = make_float2(t.x, t.y);
        u[j + 1] = make_float2(t.z, t.w);
      }
    }
    if constexpr (SF >= 2) {
      float2 t[NP];
      grow_get<N>(acc + r, t);
      unpair<N>(t, ac);
    }
  } else {
    const int64_t r0 = (e0 * 2 + 1) * NU;
    rows_fetch<NU>(in, src + r0, 2 * NU, ne, lane);
    if constexpr (SF >= 2) rows_fetch<NU>(in + K::C, acc + r0, 2 * NU, ne, lane);
    if constexpr (SF >= 1)
      for (int i = lane; i < ne * NU; i += 32) cp_async_8(in + 2 * K::C + 2 * i, U + r0 + (i / NU) * 2 * NU + i % NU);
  }
  if (GEN && SF >= 1 && ne > 0) tile_fetch<EPW, L::S::NG * 4>(R0 + K::O_GEO, A.geof + e0 * L::S::NG, ne, lane);
  const float* mc = reinterpret_cast<const float*>(A.mcg) + e * kMetricRec;
  const float rdet = __ldg(mc + 10);
  const bool aff = !GEN || (DIM == 3 && __ldg(mc + 11) != 0.f);
  int fl[DIM][2];
  float2 F[DIM];
  [[maybe_unused]] int32_t w2[DIM][2];
  if constexpr (DIM == 3) {
    int2 fw[DIM][2];
#pragma unroll
    for (int a = 0; a < DIM; ++a)
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) fw[a][sd] = __ldg(A.ffw + e * 6 + 2 * a + sd);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      float t[2] = {0.f, 0.f};
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        const int32_t po = face_link<N, NF>(A, fw[a][sd], e, 2 * a + sd, l % N, l / N, fl[a][sd]);
        if (SF >= 1 && !(fl[a][sd] & kFwL)) t[sd] = fcA[po + NF];
      }
      F[a] = make_float2(t[0], t[1]);
    }
  } else {
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      float t[2] = {0.f, 0.f};
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        const int k = (2 * a + sd) * NFP + l;
        const int32_t og = (int32_t)(e * NF + k);
        w2[a][sd] = A.fnbr[og];
        fl[a][sd] = (w2[a][sd] & 1) | ((w2[a][sd] >> 1) == og ? kFwWall : 0);
        if constexpr (SF >= 1) {
          t[sd] = fcA[e * 2 * NF + NF + k];
          if (fl[a][sd] & kFwL) t[sd] = 0.f;
        }
      }
      F[a] = make_float2(t[0], t[1]);
    }
  }
  if constexpr (!L::DIRECT || GEN) cp_async_wait_all();
  if constexpr (!L::DIRECT) {
    __syncwarp();
    const int rl = es * NU + l * N;
    grow_get<N>(in + rl, y);
    if constexpr (SF >= 2)
#pragma unroll
      for (int j = 0; j < N; ++j) ac[j] = in[K::C + rl + j];
    if constexpr (SF >= 1)
#pragma unroll
      for (int j = 0; j < N; ++j) u[j] = reinterpret_cast<const float2*>(in + 2 * K::C)[rl + j];
  }

  [[maybe_unused]] double sq = 0.0;  // stage 4: sum of the squared changes
  if constexpr (SF >= 1) {
    const RKConstF& rk = A.ep ? A.ep[e].rkp : A.rk;
    const int lc1 = DIM == 3 ? l % N : l, lc2 = DIM == 3 ? l / N : 0;
    // R ends lift minus the partner's F~ (F is zero at L ends)
#pragma unroll
    for (int a = 1; a < DIM; ++a)
      if (lane_ok) {
        float* d = C0 + (((a - 1) * 2 * EPW + es) * L::OTH + lc2) * L::RS + lc1;
        d[0] = F[a].x;
        d[EPW * L::OTH * L::RS] = F[a].y;
      }
    __syncwarp();
#pragma unroll
    for (int p = 0; p < NP; ++p) y[p] = nfma2(O.ngL[p], dup2(F[0].x), nfma2(O.gR[p], dup2(F[0].y), y[p]));
#pragma unroll
    for (int a = 1; a < DIM; ++a) {
      const int me = a == 1 ? lc1 : lc2, other = DIM == 3 ? (a == 1 ? lc2 : lc1) : 0;
      const float gl = A.cf.ops.gLd[me], gr = -A.cf.ops.gRd[me];
      const float* s = C0 + (((a - 1) * 2 * EPW + es) * L::OTH + other) * L::RS;
      float2 r0[NP], r1[NP];
      row_get<NP, L::V4>(s, r0);
      row_get<NP, L::V4>(s + EPW * L::OTH * L::RS, r1);
#pragma unroll
      for (int p = 0; p < NP; ++p) y[p] = fma2(dup2(gl), r0[p], fma2(dup2(gr), r1[p], y[p]));
    }
    float bad = 0.f;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      float2 rdj;
      if (aff) {
        rdj = dup2(rdet);
      } else {
        float2 xi[3], Sm[3][3];
        xi[0] = O.xp[p];
        xi[1] = dup2(A.cf.ops.x[lc1]);
        xi[2] = dup2(A.cf.ops.x[lc2]);
        rdj = rcp2(metric_all<DIM>(R0 + K::O_GEO + es * L::S::NG, xi, Sm));
      }
      const float2 R = mul2(make_float2(-y[p].x, -y[p].y), rdj);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int j = 2 * p + i;
        if (j >= N) {
          y[p].y = 0.f;
          continue;
        }
        const float Rj = i ? R.y : R.x;
        const float2 uu = u[j];
        float yn;
        if constexpr (SF == 1) {
          ac[j] = Rj;
          yn = uu.x + __fmaf_rn(rk.half_dt, Rj, uu.y);
        } else if constexpr (SF == 2 || SF == 3) {
          ac[j] = __fmaf_rn(2.f, Rj, ac[j]);
          yn = uu.x + __fmaf_rn(SF == 2 ? rk.half_dt : rk.dt, Rj, uu.y);
        } else {
          const float inc = rk.dt6 * (ac[j] + Rj);
          const float s2 = uu.x + inc;
          const float e2 = two_sum_lo(uu.x, inc, s2) + uu.y;
          yn = s2 + e2;
          const float lo = e2 - (yn - s2);
          // the change as a float-float value, squared in FP64
          const float ch = yn - uu.x;
          const double d = widen(ch) + widen(two_sum_lo(yn, -uu.x, ch) + (lo - uu.y));
          sq = fma(d, d, sq);
          u[j] = make_float2(yn, lo);
        }
        bad = __fmaf_rn(yn, 0.f, bad);
        if (i) y[p].y = yn;
        else y[p].x = yn;
      }
    }
    if (act && bad != 0.f) atomicExch(&A.status[ST_STATUS], -4);
    if constexpr (L::DIRECT) {
      if (act) {
        grow_put<N>(ustg + r, y);
        if constexpr (SF < 4) {
          float2 t[NP];
#pragma unroll
          for (int p = 0; p < NP; ++p) t[p] = make_float2(ac[2 * p], ac[2 * p + 1]);
          grow_put<N>(acc + r, t);
        } else {
#pragma unroll
          for (int j = 0; j < N; j += 2)
            *reinterpret_cast<float4*>(U + r + j) = make_float4(u[j].x, u[j].y, u[j + 1].x, u[j + 1].y);
        }
      }
    } else {
      if (lane_ok) {
        const int rl = es * NU + l * N;
        grow_put<N>(in + rl, y);
#pragma unroll
        for (int j = 0; j < N; ++j) {
          if constexpr (SF < 4) in[K::C + rl + j] = ac[j];
          else reinterpret_cast<float2*>(in + 2 * K::C)[rl + j] = u[j];
        }
      }
      __syncwarp();
      const int64_t r0 = (e0 * 2 + 1) * NU;
      rows_flush<NU>(ustg + r0, in, 2 * NU, ne, lane);
      if constexpr (SF < 4) rows_flush<NU>(acc + r0, in + K::C, 2 * NU, ne, lane);
      else
        for (int i = lane; i < ne * NU; i += 32)
          U[r0 + (i / NU) * 2 * NU + i % NU] = reinterpret_cast<const float2*>(in + 2 * K::C)[i];
    }
  }

  // ---- traces of the new stage value
  if (lane_ok) row_put<NP, L::V4>(R0 + es * L::AS + pline<DIM, N>(0, l), y);
  __syncwarp();
  float* tr = reinterpret_cast<float*>(A.tr);
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    float v[N];
    const float* s = R0 + es * L::AS + pline<DIM, N>(a, l);
    if (a == 0) unpair<N>(y, v);
    else if (a == 1) line_get<N, pstride<DIM, N>(1)>(s, v);
    else line_get<N, pstride<DIM, N>(2)>(s, v);
    const float2 t = line_ends<N>(O, v);
    if (!act) continue;
#pragma unroll
    for (int sd = 0; sd < 2; ++sd) {
      const int k = (2 * a + sd) * NFP + l;
      const int w = fl[a][sd];
      if (!(!(w & kFwL) || (w & kFwWall))) continue;
      if constexpr (FaceScatter<DIM>::v) {
        const int32_t pg = partner<NF>(A, w2[a][sd], (int32_t)(e * NF + k));
        tr[(int64_t)(pg / NF) * 2 * NF + NF + pg % NF] = sd ? t.y : t.x;
      } else {
        tr[(e * 2 + 1) * NF + k] = sd ? t.y : t.x;
      }
    }
  }

  if constexpr (SF == 4) {
    // 1 / dtau^2 times the lane's squared changes
    const RKConstF& rk = A.ep ? A.ep[e].rkp : A.rk;
    if (act) sum = fma(sq, rk.rdt * rk.rdt, sum);
    __syncwarp();  // the tile's buffers are read
  }
  }  // tiles

  if constexpr (SF == 4) {
    // RMS of the pseudo-time residual
    __shared__ double part[WPB];
    __shared__ double red_sh[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) part[warp] = sum;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
      for (int w = 0; w < WPB; ++w) s += part[w];
    pseudo_rms_finish(A, s, red_sh, A.E * NU);
  }
}

}  // namespace frp
