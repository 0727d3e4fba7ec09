// Fused TMOP element kernel: one group of threads (16, 32 or 64) per element.
//
//   gather  x (and v) of the element's n^d nodes into shared memory
//   forward A(q) = sum_i x_i grad phi_i(q)            (eq. (2.2), sum factorised)
//   point   T = A W^-1, mu / P / dP                   (Table 3.1, Section 3.4)
//   adjoint y_i += sum_q w_q det W [S W^-t grad phi_i] (gradient formula of Section 3.4)
//   scatter FP64 atomics into the nodal output, fixed dofs skipped
//
// OP_ENERGY instead accumulates w_q det W mu and min det A in FP64 and writes
// one partial per block (reduced in a second, fixed-order pass);
// OP_ENERGY_GRAD does both: the gradient, and the energy partials from the
// mu it evaluates anyway.
#pragma once
#include "tmop_device.cuh"
#include "tmop_fixed.cuh"
#include "tmop_kparams.h"

namespace tmop {

template <int D, int N, int Q1>
struct Shape {
  static constexpr int NDOF = (D == 2) ? N * N : N * N * N;
  static constexpr int QP = (D == 2) ? Q1 * Q1 : Q1 * Q1 * Q1;
};

template <int a, int b> struct cmax { static constexpr int value = a > b ? a : b; };

// Shared-memory words (of type R) per warp for NC gathered components.
template <int D, int N, int Q1, int NC>
struct Buf {
  static constexpr int B0 = (D == 2) ? cmax<NC * N * N, 2 * NC * Q1 * Q1>::value
                                     : cmax<NC * N * N * N, 3 * NC * N * Q1 * Q1>::value;
  static constexpr int B1 = (D == 2) ? 2 * NC * N * Q1
                                     : cmax<2 * NC * N * N * Q1, 3 * NC * Q1 * Q1 * Q1>::value;
};

// Words of type R rounded up to a whole number of 16-byte units, so every
// per-warp buffer starts on a 16-byte boundary (bulk-copy destinations).
template <class R>
constexpr int round16(int words) {
  return ((words * (int)sizeof(R) + 15) / 16) * 16 / (int)sizeof(R);
}

template <int D, int N, int Q1, class R, int OP, bool WIDE = false>
struct ElemCfg {
  // 3D Hessian action: x and v are contracted one after the other and only
  // A(x) is kept (buffer B2) while v runs through the stage buffers, so the
  // stage buffers hold D components; 2D contracts both at once (2D
  // components, no B2).
  static constexpr bool HV = OP == OP_HESS || OP == OP_GRAD_HESS;  // contracts x and v
  static constexpr bool SPLIT = HV && D == 3;
  static constexpr int NC = (HV && !SPLIT) ? 2 * D : D;
  static constexpr int B0 = round16<R>(Buf<D, N, Q1, NC>::B0);
  static constexpr int B1 = round16<R>(Buf<D, N, Q1, NC>::B1);
  static constexpr int B2 = SPLIT ? round16<R>(D * D * Shape<D, N, Q1>::QP) : 0;
  static constexpr int PER_WARP = (int)sizeof(R) * (B0 + B1 + B2);
  // Threads per element. The FP64 3D kernels with 4 or more points per
  // direction run two warps on an element, in a block of its own, as many
  // blocks per SM as shared memory holds: the contractions run on the integer
  // pipes beside the FP64 pipe, and with one warp per element only 2-3 warps
  // per scheduler hide their latency (48^3 order-3 hexes, gradient + Hessian
  // action: 8.30 ms with one warp, 6.87 with two). In 2D a stage has 6 to 24 lines, one per thread:
  // on meshes that fill the chip (WIDE, use_wide) half a warp per element leaves fewer
  // of them idle (150 x 117 order-4 quads, 6^2 points, gradient + Hessian
  // action: 266 us with a warp, 195 us with half, 197 us with a quarter); on
  // small ones, where an element's latency counts, a warp is faster (8^2
  // order-2 quads, Newton: 5.22 against 5.51 ms).
  static constexpr bool FX3 = D == 3 && sizeof(R) == 8;
  static constexpr bool HAS_WIDE = D == 2 && sizeof(R) == 8 && OP != OP_ENERGY;
  static constexpr int GT = (HAS_WIDE && WIDE) ? 16
                            : (FX3 && Q1 >= 4 && OP != OP_ENERGY && OP != OP_LINEARIZE) ? 64
                                                                                       : 32;
  // Elements in flight per block: up to 8 within ~200 KB of shared memory;
  // the FP64 3D energy as two blocks of 6 per SM where they fit
  static constexpr bool TWO = FX3 && OP == OP_ENERGY && 12 * PER_WARP <= 200 * 1024;
  static constexpr int FIT = 200 * 1024 / PER_WARP;
  static constexpr int WARPS = GT == 64 ? 1 : (TWO ? 6 : (FIT >= 8 ? 8 : (FIT < 1 ? 1 : FIT)));
  // Blocks per SM that bound the registers (0: no bound): 6 (168 registers)
  // for the kernels that hold T and dT, 7 or 8 (128) for the others; 5 for the
  // one-pass kernel at 5 points per axis, where 6 spills. 48^3 order-3 hexes (5
  // points per axis), gradient + Hessian action: 4.61 ms with 8, 3.83 with 6,
  // 3.70 with 5; 24^3, stored-Hessian product 227 us with 8, 242 with 10; energy
  // + gradient 232 us with 9, 227 with 7.
  static constexpr int WANT = HV ? (OP == OP_GRAD_HESS && Q1 == 5 ? 5 : 6) : (OP == OP_HESS_PA ? 8 : 7);
  static constexpr int MINB = GT == 64 ? (FIT >= WANT ? WANT : FIT) : (TWO ? 2 : 0);
  // after the 1D tables: the product weight w_q0 w_q1 (w_q2) of every point
  static constexpr int WQ_OFF = 2 * kMaxQ * kMaxN + kMaxQ;
  static constexpr int TABLE = round16<R>(WQ_OFF + Shape<D, N, Q1>::QP);
  static constexpr size_t smem_bytes() { return sizeof(R) * (TABLE + WARPS * (B0 + B1 + B2)); }
};

// Second term of a composite metric at one point: T2 = A W2^-1 and, for a
// direction dA, dT2 = dA W2^-1 (Section 4.2, eq. (4.1)).
template <int D, class R>
__device__ __forceinline__ void times_w2(const KBase& p, const R* M, R* out) {
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int b = 0; b < D; ++b) {
      R s = R(0);
#pragma unroll
      for (int c = 0; c < D; ++c) s = fma(M[a * D + c], R(p.Winv2[c * D + b]), s);
      out[a * D + b] = s;
    }
}

// The FP32 kernels take the second derivative of mu302 and mu98 from
// forward-mode dual numbers: the closed forms' rounding is larger there (order-1
// hexes, mu302: 1.6e-7 against 1.3e-7 of FP64). In FP64 it is smaller
// (Metric302, and MetricLin for mu98: 1.8e-15 against 2.9e-15 on order-2
// hexes), and the 45 entries of mu302 at 24^3 5^3 points take 1.9 ms, not 15.6.
template <class R>
__device__ __forceinline__ bool metric_dual(int id) { return sizeof(R) == 4 && (id == 302 || id == 98); }

// dP of metric `id` at T in direction dT
template <int D, class R>
__device__ __forceinline__ bool metric_dP(int id, const R* T, const R* dT, R* S) {
  if constexpr (sizeof(R) == 4) {
    if (metric_dual<R>(id)) {
      Dual<R> Td[D * D], Pd[D * D], mud;
#pragma unroll
      for (int i = 0; i < D * D; ++i) Td[i] = Dual<R>{T[i], dT[i]};
      const bool ok = metric_P<D>(id, Td, mud, Pd);
#pragma unroll
      for (int i = 0; i < D * D; ++i) S[i] = Pd[i].d;
      return ok;
    }
  }
  if constexpr (D == 3 && sizeof(R) == 8) {
    if (id == 302) {
      Metric302<R> L;
      const bool ok = L.init(T, R(1));
      if (ok) L.dP(dT, S);
      return ok;
    }
  }
  MetricLin<D, R> L;
  const bool ok = L.init(id, T);
  if (ok) L.dP(dT, S);
  return ok;
}

template <int D, int N, int Q1, class R, int OP, bool WIDE>
__global__ void __launch_bounds__(ElemCfg<D, N, Q1, R, OP, WIDE>::WARPS * ElemCfg<D, N, Q1, R, OP, WIDE>::GT,
                                  ElemCfg<D, N, Q1, R, OP, WIDE>::MINB)
    elem_kernel(const typename KArg<R>::type p) {
  using Cfg = ElemCfg<D, N, Q1, R, OP, WIDE>;
  constexpr int NDOF = Shape<D, N, Q1>::NDOF, QP = Shape<D, N, Q1>::QP, DD = D * D;
  constexpr int WARPS = Cfg::WARPS, GT = Cfg::GT;   // elements per block, threads per element
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R* sB = reinterpret_cast<R*>(smem_raw);
  R* sG = sB + kMaxQ * kMaxN;
  R* sw = sG + kMaxQ * kMaxN;
  const int lane = threadIdx.x % GT, warp = threadIdx.x / GT;   // thread of the element's group, group of the block
  const int bar = 1 + warp;
  R* P0 = sB + Cfg::TABLE + warp * (Cfg::B0 + Cfg::B1 + Cfg::B2);
  R* P1 = P0 + Cfg::B0;
  R* P2 = P1 + Cfg::B1;  // A(x) of the split 3D Hessian action

  // FP64: contractions in fixed point (tmop_fixed.cuh), tables from the
  // parameter block; FP32: tables in shared memory (2D) or registers (3D)
  constexpr bool FX = sizeof(R) == 8;
  if constexpr (!FX) {
    for (int t = threadIdx.x; t < Q1 * N; t += blockDim.x) {
      sB[t] = R(p.B[t]);
      sG[t] = R(p.G[t]);
    }
  }
  for (int t = threadIdx.x; t < Q1; t += blockDim.x) sw[t] = R(p.w1[t]);
  // point weights, rounded as (w_q0 w_q1) w_q2 in R: two multiplies per point
  // fewer on GB300's narrow FP64 pipe
  R* sWq = sB + Cfg::WQ_OFF;
  for (int t = threadIdx.x; t < QP; t += blockDim.x) {
    R w = R(p.w1[t % Q1]) * R(p.w1[(t / Q1) % Q1]);
    if constexpr (D == 3) w *= R(p.w1[t / (Q1 * Q1)]);
    sWq[t] = w;
  }
  constexpr int GW = GT > 32 ? GT / 32 : 1;   // warps per element
  // mu303 with W = I: the pointwise stage of these FP64 3D kernels in fixed point (fx_point303)
  constexpr bool FX303 = FX && D == 3 && OP != OP_LINEARIZE && OP != OP_HESS_PA;
  constexpr bool FXPA = FX && D == 3 && OP == OP_HESS_PA;   // and the product of the stored Hessians (fx_stored_product)
  constexpr int NKEY = FXPA ? D : (OP == OP_GRAD_HESS ? 2 : 1);
  constexpr int NKQ = (FXPA || (FX303 && OP != OP_ENERGY)) ? NKEY * QP : 1;
  __shared__ short s_kq[NKQ > 1 ? WARPS : 1][NKQ];   // exponents of the points' results
  __shared__ int s_key[NKQ > 1 ? WARPS : 1][GW * NKEY];
  __shared__ unsigned s_mag[WARPS][GW * 2 * D];   // per warp and component: largest magnitudes of the group's warps
  R Wi[DD];
#pragma unroll
  for (int i = 0; i < DD; ++i) Wi[i] = R(p.Winv[i]);
  // FP32 3D kernels: the 1D tables in registers for the register-blocked stages
  constexpr bool RB = (D == 3) && sizeof(R) == 4;
  R tB[Q1 * N], tG[Q1 * N];
  if constexpr (RB) {
#pragma unroll
    for (int t = 0; t < Q1 * N; ++t) {
      tB[t] = R(p.B[t]);
      tG[t] = R(p.G[t]);
    }
  }
  __syncthreads();

  double accF = 0.0, accMin = INFINITY;
  // elements in flight per block (FP64, small meshes: fewer than WARPS, launch_elem_impl)
  const int warps = FX ? (int)blockDim.x / GT : WARPS;
  const int nwarps_total = gridDim.x * warps;
  // (the product from compact records, OP_HESS_PA_C, is pac_kernel in tmop_pa_compact.cu)
  constexpr bool PA_APPLY = OP == OP_HESS_PA;
  constexpr bool EG = OP == OP_ENERGY_GRAD;                // gradient + energy partials
  constexpr bool GRADLIKE = OP == OP_GRADIENT || EG;
  constexpr int NSH = PA_APPLY ? D * D * (D * D + 1) / 2 : 1;
  static_assert(OP != OP_HESS_PA_C, "OP_HESS_PA_C runs in pac_kernel");
  static_assert(OP != OP_GRAD_HESS || sizeof(R) == 8, "the fused gradient + Hessian action is FP64");
  // its second 3D adjoint runs its stage 2 in the A(x) buffer
  static_assert(!(OP == OP_GRAD_HESS && D == 3) || 2 * D * N * N * Q1 <= Cfg::B2, "B2 too small");
  static_assert(OP != OP_LINEARIZE_C || D == 3, "compact records are 3D");
  static_assert(!FX || Cfg::NC * FxNodal<D, N>::CS <= Cfg::B0, "B0 too small for the padded nodal fields");
  NodeMap<N> nodes(p.elem_nodes, p.sx, p.sy, D == 3 ? N - 1 : 1);
  const int ecount = p.elist ? p.ecount : p.nelem;
  for (int ei = blockIdx.x * warps + warp; ei < ecount; ei += nwarps_total) {
    const int e = p.elist ? __ldg(p.elist + ei) : ei;
    nodes.element(e, NDOF);
    // Partially assembled product: the stored values of this lane's first
    // point are loaded now, so their latency overlaps the gather and the
    // v-contraction. (With two warps per element the registers they take cost
    // more than they hide: 273 against 227 us on 24^3 order-3 hexes; a prefetch
    // of the element's block into L2 instead: 236 us.)
    constexpr bool HPRE = PA_APPLY && GT <= 32;
    R hpre[HPRE ? NSH : 1];
    if constexpr (HPRE) {
      if (lane < Shape<D, N, Q1>::QP) {
        const R* H0 = static_cast<const R*>(p.pa) + (size_t)e * p.pa_stride + lane;
#pragma unroll
        for (int t = 0; t < NSH; ++t) hpre[t] = __ldg(H0 + (size_t)t * Shape<D, N, Q1>::QP);
      }
    }
    // ---- gather. The coordinates are taken relative to the element's first
    // node (in FP64) before they are rounded (FP32) or given the element's
    // common exponent (FP64): A is translation invariant (sum_i grad phi_i =
    // 0), and this keeps the relative error of A at the level of eps instead
    // of eps |x| / h.
    double xref[D];
    unsigned mag[FX ? Cfg::NC : 1] = {};   // FP64: largest magnitude (high word) per gathered component
    auto nodal = [&](int c, int t) { return FX ? FxNodal<D, N>::at(c, t) : c * NDOF + t; };
    if constexpr (!PA_APPLY) {
      const int g0 = nodes(0);
#pragma unroll
      for (int c = 0; c < D; ++c) xref[c] = __ldg(p.x + (size_t)c * p.nnode + g0);
    }
    for (int t = lane; t < NDOF; t += GT) {
      const int g = nodes(t);
      if constexpr (PA_APPLY) {
        // the partially assembled product needs only the direction v
#pragma unroll
        for (int c = 0; c < D; ++c) {
          const size_t dof = (size_t)c * p.nnode + g;
          const bool fx = p.fixed && __ldg(p.fixed + dof);
          const R vv = fx ? R(0) : (p.v32 ? R(__ldg(p.v32 + dof)) : from_f64<R>(__ldg(p.v + dof)));
          P0[nodal(c, t)] = vv;
          if constexpr (FX) mag[c] = max(mag[c], fx_mag(vv));
        }
        continue;
      }
#pragma unroll
      for (int c = 0; c < D; ++c) {
        const double xv = __ldg(p.x + (size_t)c * p.nnode + g) - xref[c];
        P0[nodal(c, t)] = from_f64<R>(xv);
        if constexpr (FX) mag[c] = max(mag[c], fx_mag(xv));
      }
      if constexpr (Cfg::HV && !Cfg::SPLIT) {
#pragma unroll
        for (int c = 0; c < D; ++c) {
          const size_t dof = (size_t)c * p.nnode + g;
          const bool fx = p.fixed && __ldg(p.fixed + dof);
          const double vv = fx ? 0.0 : __ldg(p.v + dof);
          P0[nodal(D + c, t)] = from_f64<R>(vv);
          if constexpr (FX) mag[D + c] = max(mag[D + c], fx_mag(vv));
        }
      }
    }
    // the split Hessian action's v, loaded behind x and masked
    constexpr int VPRE = (Cfg::SPLIT && FX) ? (NDOF + GT - 1) / GT : 0;
    double vpre[VPRE > 0 ? VPRE * D : 1];
#pragma unroll
    for (int k = 0; k < VPRE; ++k) {
      const int t = lane + k * GT;
      if (t >= NDOF) break;
      const int g = nodes(t);
#pragma unroll
      for (int c = 0; c < D; ++c) {
        const size_t dof = (size_t)c * p.nnode + g;
        const double vv = __ldg(p.v + dof);
        vpre[k * D + c] = (p.fixed && __ldg(p.fixed + dof)) ? 0.0 : vv;
      }
    }
    int em[FX ? Cfg::NC : 1];
    int emx[FX ? D : 1];   // the split Hessian action's exponents of x
    bool fx303 = false;    // mu303 with W = I: pointwise stage in fixed point
    if constexpr (FX) fx_group_exp<GT, Cfg::NC>(mag, em, s_mag[warp], bar);
    else __syncwarp();
    if constexpr (FX303) {
      // one exponent for all components (at most 2 bits lost to one of them),
      // where the scalars stay inside the FP64 range (kFx303X)
      const int lo = min(em[0], min(em[1], em[2])), hi = max(em[0], max(em[1], em[2]));
      fx303 = p.metric == 303 && p.wkind == WK_IDENTITY && !p.metric2 &&
              hi >= 1023 - kFx303X && hi <= 1023 + kFx303X && hi - lo <= 2;
      if (fx303) em[0] = em[1] = em[2] = hi;
    }
    // ---- forward contraction: A (and dA) at every point
    if constexpr (Cfg::SPLIT && FX) {
      // A(x) into P2 (P2 also serves as the first stage buffer), then v into
      // P1, by one copy of the code
#pragma unroll 1
      for (int f = 0;; ++f) {
        fwd3_fx<N, Q1, D, GT>(p.fx, em, P0, f == 0 ? P2 : P1, lane, bar);
        if (f) break;
#pragma unroll
        for (int c = 0; c < D; ++c) {
          mag[c] = 0;
          emx[c] = em[c];
        }
#pragma unroll
        for (int k = 0; k < VPRE; ++k) {
          const int t = lane + k * GT;
          if (t >= NDOF) break;
#pragma unroll
          for (int c = 0; c < D; ++c) {
            P0[nodal(c, t)] = vpre[k * D + c];
            mag[c] = max(mag[c], fx_mag(vpre[k * D + c]));
          }
        }
        fx_group_exp<GT, D>(mag, em, s_mag[warp], bar);
        if (fx303) {
          const int hi = max(em[0], max(em[1], em[2]));
          fx303 = hi >= 1023 - kFx303V && hi <= 1023 + kFx303V;
          if (fx303) em[0] = em[1] = em[2] = hi;
        }
      }
    } else if constexpr (Cfg::SPLIT) {
      fwd3_rb<N, Q1, D, R>(tB, tG, P0, P2, lane);
      for (int t = lane; t < NDOF; t += GT) {
        const int g = nodes(t);
#pragma unroll
        for (int c = 0; c < D; ++c) {
          const size_t dof = (size_t)c * p.nnode + g;
          const bool fx = p.fixed && __ldg(p.fixed + dof);
          P0[c * NDOF + t] = fx ? R(0) : from_f64<R>(__ldg(p.v + dof));
        }
      }
      __syncwarp();
      fwd3_rb<N, Q1, D, R>(tB, tG, P0, P1, lane);
    } else if constexpr (D == 2) {
      if constexpr (FX) fwd2_fx<N, Q1, Cfg::NC, GT>(p.fx, em, P0, P1, lane, bar);
      else fwd2<N, Q1, Cfg::NC, R>(sB, sG, P0, P1, lane);
    } else {
      if constexpr (FX) fwd3_fx<N, Q1, Cfg::NC, GT>(p.fx, em, P0, P1, lane, bar);
      else fwd3_rb<N, Q1, Cfg::NC, R>(tB, tG, P0, P1, lane);
    }
    R* Abuf = Cfg::SPLIT ? P2 : ((D == 2) ? P0 : P1);     // A: [D][D][QP]
    R* dAbuf = Cfg::SPLIT ? P1 : Abuf + DD * QP;         // dA (Hessian action)
    R* Rbuf = Cfg::SPLIT ? P1 : Abuf;                    // per-point output of the adjoint
    // ---- pointwise
    double emin = INFINITY;
    // FP64 3D: A and dA are in fixed point
    constexpr bool RAW = FX && D == 3;
    FxScale sA[RAW ? D : 1], sV[RAW ? D : 1];
    if constexpr (RAW) {
#pragma unroll
      for (int c = 0; c < D; ++c) {
        sA[c] = fx_scale(Cfg::SPLIT ? emx[c] : em[c], p.fx.xin, p.fx.gexp);
        sV[c] = fx_scale(em[c], p.fx.xin, p.fx.gexp);
      }
    }
    auto load = [&](const R* buf, const FxScale* sc, int i, int q) -> R {
      if constexpr (RAW) return fx_to_f64(reinterpret_cast<const fx_t*>(buf)[i * QP + q], sc[i / D]);
      else return buf[i * QP + q];
    };
    int key[D];
#pragma unroll
    for (int k = 0; k < D; ++k) key[k] = kFxKeyMin;
    // FP64: largest magnitude (high word) per component of the fields the
    // adjoint map takes (OP_GRAD_HESS: the gradient's, then the Hessian action's)
    unsigned rmag[FX ? 2 * D : 1] = {};
    constexpr int NS = DD * (DD + 1) / 2;
    // the exponents of a point's results in fixed point (k: 0 the gradient's
    // fields, NKEY - 1 the Hessian action's)
    auto record = [&](int k, int q, const FxPoint& pt) {
      key[k] = max(key[k], fx_point_key(pt));
      s_kq[warp][k * QP + q] = (short)(pt.zero() ? -16000 : pt.E);
    };
    unsigned thin_pts = 0;   // the thread's points of a fixed-point element that took the FP64 stage
    for (int q = lane; q < QP; q += GT) {
      if constexpr (OP == OP_HESS_PA) {
        // y = H dA with the stored symmetric A-space Hessian (already scaled by w det W)
        const R* H = static_cast<const R*>(p.pa) + (size_t)e * p.pa_stride + q;
        // all NS loads are issued before the first use, so their latencies overlap
        R h[NS];
        if (HPRE && q == lane) {
#pragma unroll
          for (int t = 0; t < NS; ++t) h[t] = hpre[HPRE ? t : 0];
        } else {
#pragma unroll
          for (int t = 0; t < NS; ++t) h[t] = __ldg(H + (size_t)t * QP);
        }
        if constexpr (FXPA) {
          const short4 ex = __ldg(p.pa_exp + (size_t)e * QP + q);
          FxPoint pt[D];
          fx_stored_product<QP>(reinterpret_cast<fx_t*>(Abuf) + q, h, ex, sA, pt);
          const bool bad = ex.w == kPaNan || sA[0].nan || sA[1].nan || sA[2].nan;   // NaN everywhere
#pragma unroll
          for (int a = 0; a < D; ++a) {
            key[a] = max(key[a], bad ? kFxNan : fx_point_key(pt[a]));
            s_kq[warp][a * QP + q] = (short)(pt[a].zero() ? -16000 : pt[a].E);
          }
          continue;
        }
        R dA[DD], y[DD];
#pragma unroll
        for (int i = 0; i < DD; ++i) {
          dA[i] = load(Abuf, sA, i, q);
          y[i] = R(0);
        }
        int s = 0;
#pragma unroll
        for (int r = 0; r < DD; ++r)
#pragma unroll
          for (int c = r; c < DD; ++c, ++s) {
            y[r] = fma(h[s], dA[c], y[r]);
            if (c != r) y[c] = fma(h[s], dA[r], y[c]);
          }
#pragma unroll
        for (int i = 0; i < DD; ++i) {
          Abuf[i * QP + q] = y[i];
          if constexpr (FX) rmag[i / D] = max(rmag[i / D], fx_mag(y[i]));
        }
        continue;
      }
      if constexpr (FX303) {
        fx_t* Tq = reinterpret_cast<fx_t*>(Abuf) + q;
        int up = 0;
        bool thin = true;
        if (fx303) {
          // (one choice per warp: a warp that took both stages would pay for both;
          // the lanes of the last points alone)
          const int n = QP - (q - (int)(threadIdx.x & 31));
          thin = __any_sync(n < 32 ? (1u << n) - 1u : 0xffffffffu, fx_thin<QP>(Tq, up));
          if (OP == OP_GRAD_HESS && thin) thin_pts |= 1u << (q / GT);
        }
        if (!thin) {
          FxPoint pt[2];
          double mu, tau;
          const double s = sWq[q] * p.detW;
          const bool ok = fx_point303<QP, GRADLIKE || OP == OP_GRAD_HESS, Cfg::HV>(
              Tq, reinterpret_cast<fx_t*>(dAbuf) + q, up, sA[0].kb, sV[0].kb, s, pt[0], pt[NKEY - 1], mu, tau);
          if constexpr (OP != OP_ENERGY) {
#pragma unroll
            for (int k = 0; k < NKEY; ++k) record(k, q, pt[k]);
          }
          if constexpr (EG || OP == OP_ENERGY) {
            emin = fmin(emin, tau);
            if (ok) accF += s * mu;
            else accF = INFINITY;
          }
          continue;
        }
      }
      R A[DD];
#pragma unroll
      for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = 0; b < D; ++b) A[a * D + b] = load(Abuf, sA, a * D + b, q);
      const R wq = sWq[q];
      R detW = R(p.detW);
      if (p.wkind == WK_PER_QP) {
        const double* Wq = p.Winv_qp + ((size_t)e * QP + q) * DD;
#pragma unroll
        for (int i = 0; i < DD; ++i) Wi[i] = R(__ldg(Wq + i));
        detW = R(__ldg(p.detW_qp + (size_t)e * QP + q));
      }
      R T[DD];
      if (p.wkind == WK_IDENTITY) {
#pragma unroll
        for (int i = 0; i < DD; ++i) T[i] = A[i];
      } else {
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
          for (int b = 0; b < D; ++b) {
            R s = R(0);
#pragma unroll
            for (int c = 0; c < D; ++c) s = fma(A[a * D + c], Wi[c * D + b], s);
            T[a * D + b] = s;
          }
      }
      if constexpr (OP == OP_GRAD_HESS) {
        // s P and s dP[dT] at the same point (s = w det W): one evaluation of
        // the metric's terms for both. For an (|T|^2, det T) metric
        // P = 2 mu_1 T + mu_t C, i.e. s P = cA T + ct C with MetricAct's scaled
        // coefficients (mu14 = |T - I|^2 is the exception: its P from metric_P);
        // mu302 from the terms of Metric302.
        const R s = wq * detW;
        R dA[DD], dT[DD], Sg[DD], Sh[DD];
#pragma unroll
        for (int i = 0; i < DD; ++i) dA[i] = load(dAbuf, sV, i, q);
        if (p.wkind == WK_IDENTITY) {
#pragma unroll
          for (int i = 0; i < DD; ++i) dT[i] = dA[i];
        } else {
#pragma unroll
          for (int a = 0; a < D; ++a)
#pragma unroll
            for (int b = 0; b < D; ++b) {
              R acc = R(0);
#pragma unroll
              for (int c = 0; c < D; ++c) acc = fma(dA[a * D + c], Wi[c * D + b], acc);
              dT[a * D + b] = acc;
            }
        }
        bool ok;
        if (D == 3 && p.metric == 302) {   // (FP64 kernels only)
          if constexpr (D == 3) {
            Metric302<R> L;
            ok = L.init(T, s);
            if (ok) {
              L.dP(dT, Sh);
#pragma unroll
              for (int i = 0; i < DD; ++i) Sg[i] = L.P(i);
            }
          }
        } else {
          MetricAct<D, R> L;
          ok = L.init(p.metric, T, s);
          if (ok) {
            L.dP(dT, Sh);
            if (p.metric == 14) {
              R mu;
              metric_P<D>(p.metric, T, mu, Sg, s);
            } else {
#pragma unroll
              for (int i = 0; i < DD; ++i) Sg[i] = fma(L.cA, L.x(i), L.ct * L.C[i]);
            }
          }
        }
        // R = S W^-t for both: the Hessian action's in place of dA, the
        // gradient's in place of A
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
          for (int b = 0; b < D; ++b) {
            R rg = R(0), rh = R(0);
            if (p.wkind == WK_IDENTITY) {
              rg = Sg[a * D + b];
              rh = Sh[a * D + b];
            } else {
#pragma unroll
              for (int c = 0; c < D; ++c) {
                rg = fma(Sg[a * D + c], Wi[b * D + c], rg);
                rh = fma(Sh[a * D + c], Wi[b * D + c], rh);
              }
            }
            rg = ok ? rg : R(0);
            rh = ok ? rh : R(0);
            Abuf[(a * D + b) * QP + q] = rg;
            dAbuf[(a * D + b) * QP + q] = rh;
            rmag[a] = max(rmag[a], fx_mag(rg));
            rmag[D + a] = max(rmag[D + a], fx_mag(rh));
          }
        continue;
      }
      if constexpr (OP == OP_LINEARIZE_C) {
        // compact record: T and w det W times the partials of mu in (|T|^2, det T)
        R* H = static_cast<R*>(p.pa) + (size_t)e * p.pa_stride + q;
        const R s = wq * detW;
        MetricLin<D, R> L;
        const bool ok = L.init(p.metric, T);
#pragma unroll
        for (int i = 0; i < DD; ++i) H[(size_t)i * QP] = T[i];
        H[(size_t)(DD + 0) * QP] = ok ? s * L.m1 : R(0);
        H[(size_t)(DD + 1) * QP] = ok ? s * L.mt : R(0);
        H[(size_t)(DD + 2) * QP] = ok ? s * L.m11 : R(0);
        H[(size_t)(DD + 3) * QP] = ok ? s * L.m1t : R(0);
        H[(size_t)(DD + 4) * QP] = ok ? s * L.mtt : R(0);
        continue;
      }
      if constexpr (OP == OP_LINEARIZE) {
        // column kl of the A-space Hessian: direction dA = E_kl, dT = E_kl W^-1,
        // R = w det W (d^2mu/dT^2 : dT) W^-t; the upper triangle is stored
        R* H = static_cast<R*>(p.pa) + (size_t)e * p.pa_stride + q;
        const R s = wq * detW;
        // FP64 3D: the entries are packed for the fixed-point product as soon as a
        // point has them all, which writes them once and leaves the integer work
        // beside the FP64 pipe's (a packing kernel of its own: 2.45 ms on 32^3
        // order-3 hexes, 2.39 so; 2.15 without packing)
        constexpr bool PACK = FX && D == 3;
        R hp[PACK ? 45 : 1];
        bool ok = true;
        auto put = [&](int i, R v) {
          if constexpr (PACK) hp[i] = v;
          else H[(size_t)i * QP] = ok ? v : R(0);
        };
        MetricLin<D, R> L;
        const bool lin = sizeof(R) == 4 ? !metric_dual<R>(p.metric) : p.metric != 302;
        if (lin) ok = L.init(p.metric, T);
        if constexpr (D == 3 && sizeof(R) == 8) {
          if (!lin && p.wkind == WK_IDENTITY && !p.metric2) {
            // mu302 with W = I, in closed form: with G = T^t T, M = I1 T - T G
            // (= dK/dT / 2), a = 2 s K / (9 tau^2), b = 2 s I1 / (9 tau^2),
            // c = 2 s I1 K / (9 tau^3) as in Metric302,
            //   H[(a,b),(c,d)] = (a + b I1) d_ac d_bd + (da_cd + 2 b T_cd) T_ab + db_cd M_ab - dc_cd C_ab
            //                    - b (d_ac G_bd + d_bd (T T^t)_ac + T_ad T_cb) - c dC_ab/dT_cd,
            // da, db, dc the derivatives of a, b, c by T_cd (nine directions of
            // dP took 15.6 ms, 1.9 now, on 24^3 order-3 hexes)
            Metric302<R> Q;
            ok = Q.init(T, s);
            R G[9], TT[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
              const int r = i / 3, c = i % 3;
              G[i] = fma(T[r], T[c], fma(T[3 + r], T[3 + c], T[6 + r] * T[6 + c]));
              TT[i] = fma(T[3 * r], T[3 * c], fma(T[3 * r + 1], T[3 * c + 1], T[3 * r + 2] * T[3 * c + 2]));
            }
            int off3 = 0;
#pragma unroll
            for (int kl = 0; kl < 9; ++kl) {
              const int c = kl / 3, d = kl % 3;
              const R dt = R(-2) * Q.it * Q.C[kl];
              const R pT = fma(R(2) * Q.f, Q.N[kl], fma(Q.a, dt, R(2) * Q.b * T[kl]));
              const R pM = fma(R(2) * Q.f, T[kl], Q.b * dt);
              const R pC = -Q.it * fma(R(2), fma(Q.a, T[kl], Q.b * Q.N[kl]), R(-3) * Q.c * Q.C[kl]);
#pragma unroll
              for (int mn = kl; mn < 9; ++mn) {
                const int a = mn / 3, b = mn % 3;
                R v = fma(pT, T[mn], fma(pM, Q.N[mn], pC * Q.C[mn]));
                R u = T[a * 3 + d] * T[c * 3 + b];
                if (a == c) u += G[b * 3 + d];
                if (b == d) u += TT[a * 3 + c];
                v = fma(-Q.b, u, v);
                if (mn == kl) v += fma(Q.b, Q.I1, Q.a);
                if (a != c && b != d) {
                  const int ee = 3 - a - c, ff = 3 - b - d;
                  const bool plus = (c == (a + 1) % 3) == (d == (b + 1) % 3);
                  v = fma(plus ? -Q.c : Q.c, T[ee * 3 + ff], v);
                }
                put(off3 + mn - kl, v);
              }
              off3 += 9 - kl;
            }
            if constexpr (PACK) fx_pack_point(hp, ok, H, QP, p.pa_exp + (size_t)e * QP + q);
            continue;
          }
        }
        if constexpr (D == 3) {
          if (lin && p.wkind == WK_IDENTITY && !p.metric2) {
            // W = I, an (|T|^2, det T) metric: the 45 entries in closed form,
            //   H[(a,b),(c,d)] = 2 mu_1 d_ac d_bd + (4 mu_11 T_cd + 2 mu_1t C_cd) T_ab
            //                    + (2 mu_1t T_cd + mu_tt C_cd) C_ab + mu_t dC_ab/dT_cd,
            // with dC_ab/dT_cd = +-T_ef (e, f the indices other than a, c and
            // b, d; zero if a = c or b = d): ~4 operations per entry where the
            // directional derivative costs ~100 per column. In FP64, whose pipe
            // bounds this kernel, two multiply-adds per entry on top of the
            // constant term: 2.39 -> 2.26 ms on 32^3 order-3 hexes.
            const R m1 = s * L.m1, mt = s * L.mt, m11 = s * L.m11, m1t = s * L.m1t, mtt = s * L.mtt;
            R mT[PACK ? 9 : 1];
            if constexpr (PACK) {
#pragma unroll
              for (int i = 0; i < 9; ++i) mT[i] = mt * T[i];
            }
            int off3 = 0;
#pragma unroll
            for (int kl = 0; kl < 9; ++kl) {
              const int c = kl / 3, d = kl % 3;
              const R Pc = fma(R(4) * m11, L.x(kl), R(2) * m1t * L.C[kl]);
              const R Qc = fma(R(2) * m1t, L.x(kl), mtt * L.C[kl]);
#pragma unroll
              for (int mn = kl; mn < 9; ++mn) {
                const int a = mn / 3, b = mn % 3;
                const int ee = 3 - a - c, ff = 3 - b - d;
                const bool plus = (c == (a + 1) % 3) == (d == (b + 1) % 3);
                R v;
                if constexpr (PACK) {
                  if (mn == kl) v = fma(Qc, L.C[mn], R(2) * m1);
                  else if (a != c && b != d) v = fma(Qc, L.C[mn], plus ? mT[ee * 3 + ff] : -mT[ee * 3 + ff]);
                  else v = Qc * L.C[mn];
                  v = fma(Pc, L.x(mn), v);
                } else {
                  v = fma(Pc, L.x(mn), Qc * L.C[mn]);
                  if (mn == kl) v += R(2) * m1;
                  if (a != c && b != d) v = fma(plus ? mt : -mt, T[ee * 3 + ff], v);
                }
                put(off3 + mn - kl, v);
              }
              off3 += 9 - kl;
            }
            if constexpr (PACK) fx_pack_point(hp, ok, H, QP, p.pa_exp + (size_t)e * QP + q);
            continue;
          }
        }
        int off = 0;
#pragma unroll 1
        for (int kl = 0; kl < DD; ++kl) {
          const int k = kl / D, l = kl % D;
          R dT[DD], S[DD];
#pragma unroll
          for (int a = 0; a < D; ++a)
#pragma unroll
            for (int b = 0; b < D; ++b)
              dT[a * D + b] = a == k ? (p.wkind == WK_IDENTITY ? R(l == b) : Wi[l * D + b]) : R(0);
          if (lin) {
            if (ok) L.dP(dT, S);
          } else if constexpr (sizeof(R) == 4) {
            Dual<R> Td[DD], Pd[DD], mud;
#pragma unroll
            for (int i = 0; i < DD; ++i) Td[i] = Dual<R>{T[i], dT[i]};
            ok = metric_P<D>(p.metric, Td, mud, Pd);
#pragma unroll
            for (int i = 0; i < DD; ++i) S[i] = Pd[i].d;
          } else {
            ok = metric_dP<D>(p.metric, T, dT, S);
          }
          // second term: dT2 = E_kl W2^-1
          R S2[DD];
          bool ok2 = false;
          R s2 = R(0);
          if (p.metric2) {
            R T2[DD], dT2[DD];
            times_w2<D>(p, A, T2);
#pragma unroll
            for (int a = 0; a < D; ++a)
#pragma unroll
              for (int b = 0; b < D; ++b) dT2[a * D + b] = a == k ? R(p.Winv2[l * D + b]) : R(0);
            ok2 = metric_dP<D>(p.metric2, T2, dT2, S2);
            s2 = wq * R(p.detW2) * (p.eta2 ? R(__ldg(p.eta2 + (size_t)e * QP + q)) : R(1));
          }
#pragma unroll
          for (int mn = 0; mn < DD; ++mn) {
            if (mn < kl) continue;
            const int m = mn / D, nn = mn % D;
            R r = R(0);
            if (p.wkind == WK_IDENTITY) {
              r = S[mn];
            } else {
#pragma unroll
              for (int c = 0; c < D; ++c) r = fma(S[m * D + c], Wi[nn * D + c], r);
            }
            R val = ok ? s * r : R(0);
            if (ok2) {
              R r2 = R(0);
#pragma unroll
              for (int c = 0; c < D; ++c) r2 = fma(S2[m * D + c], R(p.Winv2[nn * D + c]), r2);
              val = fma(s2, r2, val);
            }
            H[(size_t)(off + mn - kl) * QP] = val;
          }
          off += DD - kl;
        }
        if constexpr (PACK) {   // (read back: the loop's index is not a constant)
          R hb[45];
#pragma unroll
          for (int i = 0; i < 45; ++i) hb[i] = H[(size_t)i * QP];
          fx_pack_point(hb, true, H, QP, p.pa_exp + (size_t)e * QP + q);
        }
        continue;
      }
      if constexpr (OP == OP_ENERGY) {
        double Ad[DD];
#pragma unroll
        for (int i = 0; i < DD; ++i) Ad[i] = double(A[i]);
        const double dA = det_m<D>(Ad);
        emin = fmin(emin, dA);
        R mu;
        R Pd[DD];
        if (metric_P<D>(p.metric, T, mu, Pd)) accF += double(wq * detW) * double(mu);
        else accF = INFINITY;
        if (p.metric2) {
          R T2[DD], mu2;
          times_w2<D>(p, A, T2);
          const double eta = p.eta2 ? __ldg(p.eta2 + (size_t)e * QP + q) : 1.0;
          if (metric_P<D>(p.metric2, T2, mu2, Pd)) accF += double(wq) * p.detW2 * eta * double(mu2);
          else accF = INFINITY;
        }
      } else {
        // S below is already scaled by s = w det W (folded into the metric's
        // coefficients)
        const R s = wq * detW;
        R S[DD], dA[DD];
        bool ok;
        if constexpr (GRADLIKE) {
          R mu;
          ok = metric_P<D>(p.metric, T, mu, S, s);
          if constexpr (EG) {   // the energy of OP_ENERGY from the same point
            double Ad[DD];
#pragma unroll
            for (int i = 0; i < DD; ++i) Ad[i] = double(A[i]);
            emin = fmin(emin, det_m<D>(Ad));
            if (ok) accF += double(wq * detW) * double(mu);
            else accF = INFINITY;
          }
        } else {
          R dT[DD];
#pragma unroll
          for (int i = 0; i < DD; ++i) dA[i] = load(dAbuf, sV, i, q);
          if (p.wkind == WK_IDENTITY) {
#pragma unroll
            for (int i = 0; i < DD; ++i) dT[i] = dA[i];
          } else {
#pragma unroll
            for (int a = 0; a < D; ++a)
#pragma unroll
              for (int b = 0; b < D; ++b) {
                R acc = R(0);
#pragma unroll
                for (int c = 0; c < D; ++c) acc = fma(dA[a * D + c], Wi[c * D + b], acc);
                dT[a * D + b] = acc;
              }
          }
          if (metric_dual<R>(p.metric)) {
            Dual<R> Td[DD], Pd[DD], mud;
#pragma unroll
            for (int i = 0; i < DD; ++i) Td[i] = Dual<R>{T[i], dT[i]};
            ok = metric_P<D>(p.metric, Td, mud, Pd);
#pragma unroll
            for (int i = 0; i < DD; ++i) S[i] = s * Pd[i].d;
          } else if (D == 3 && sizeof(R) == 8 && p.metric == 302) {
            if constexpr (D == 3 && sizeof(R) == 8) {
              Metric302<R> L;
              ok = L.init(T, s);
              if (ok) L.dP(dT, S);
            }
          } else {
            MetricAct<D, R> L;
            ok = L.init(p.metric, T, s);
            if (ok) L.dP(dT, S);
          }
        }
        // R = s S W^-t (S already carries s), stored in place of A at this point
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
          for (int b = 0; b < D; ++b) {
            R r = R(0);
            if (p.wkind == WK_IDENTITY) {
              r = S[a * D + b];
            } else {
#pragma unroll
              for (int c = 0; c < D; ++c) r = fma(S[a * D + c], Wi[b * D + c], r);
            }
            r = ok ? r : R(0);
            Rbuf[(a * D + b) * QP + q] = r;
            if constexpr (FX) rmag[a] = max(rmag[a], fx_mag(r));
          }
        if (p.metric2) {
          // + eta w det W2 S2 W2^-t (S2 = P2 or dP2 at T2 = A W2^-1)
          R T2[DD], S2[DD];
          times_w2<D>(p, A, T2);
          bool ok2;
          if constexpr (GRADLIKE) {
            R mu2;
            ok2 = metric_P<D>(p.metric2, T2, mu2, S2);
            if constexpr (EG) {
              const double eta = p.eta2 ? __ldg(p.eta2 + (size_t)e * QP + q) : 1.0;
              if (ok2) accF += double(wq) * p.detW2 * eta * double(mu2);
              else accF = INFINITY;
            }
          } else {
            R dT2[DD];
            times_w2<D>(p, dA, dT2);
            ok2 = metric_dP<D>(p.metric2, T2, dT2, S2);
          }
          if (ok2) {
            const R s2 = wq * R(p.detW2) * (p.eta2 ? R(__ldg(p.eta2 + (size_t)e * QP + q)) : R(1));
#pragma unroll
            for (int a = 0; a < D; ++a)
#pragma unroll
              for (int b = 0; b < D; ++b) {
                R r2 = R(0);
#pragma unroll
                for (int c = 0; c < D; ++c) r2 = fma(S2[a * D + c], R(p.Winv2[b * D + c]), r2);
                r2 = fma(s2, r2, Rbuf[(a * D + b) * QP + q]);
                Rbuf[(a * D + b) * QP + q] = r2;
                if constexpr (FX) rmag[a] = max(rmag[a], fx_mag(r2));
              }
          }
        }
        if constexpr (FX303) {
          if (fx303) record(0, q, fx_point_pack<QP>(Rbuf + q));
        }
      }
    }
    if constexpr (FX303 && OP == OP_GRAD_HESS) {
      // (after the loop, which then keeps its registers for the metrics: 32^3
      // order-2 hexes with mu98 782 us with the packing inside, 765 so; for the
      // other operations inside: 48^3 order-3 gradient 1.73 ms after it, 1.65 so)
#pragma unroll 1
      for (int q = lane; thin_pts; q += GT, thin_pts >>= 1)
        if (thin_pts & 1u) {
          record(0, q, fx_point_pack<QP>(Abuf + q));
          record(NKEY - 1, q, fx_point_pack<QP>(dAbuf + q));
        }
    }
    if constexpr (OP == OP_LINEARIZE || OP == OP_LINEARIZE_C) {
      group_sync<GT>(bar);
    } else if constexpr (OP == OP_ENERGY) {
      accMin = fmin(accMin, emin);
      if (p.elem_min) {
#pragma unroll
        for (int o = (GT < 32 ? GT : 32) / 2; o > 0; o >>= 1)
          emin = fmin(emin, __shfl_xor_sync(group_mask<GT>(), emin, o));
        if (lane == 0) p.elem_min[e] = emin;
      }
    } else if constexpr (OP == OP_GRAD_HESS) {
      // ---- two adjoint contractions: 3D, the Hessian action's fields (P1)
      // into y, then the gradient's (P2) into g, each through P0 and its own
      // buffer; 2D, both at once (components 0..D-1 the gradient's fields,
      // D..2D-1 the Hessian action's)
      if constexpr (D == 2) {
        // P0 holds the gradient's fields (in place of A), then the Hessian action's (dA)
        int er[2 * D];
        fx_group_exp<GT, 2 * D>(rmag, er, s_mag[warp], bar);
        adj2_fx<N, Q1, 2 * D, GT>(p.fx, er, P0, P1, lane, bar);
        for (int t = lane; t < NDOF; t += GT) {
          const int gn = nodes(t);
#pragma unroll
          for (int c = 0; c < D; ++c) {
            const size_t dof = (size_t)c * p.nnode + gn;
            if (p.fixed && __ldg(p.fixed + dof)) continue;
            atomicAdd(p.g + dof, P0[nodal(c, t)]);
            atomicAdd(p.y + dof, P0[nodal(D + c, t)]);
          }
        }
      } else {
        int er2[2 * D];
        if (FX303 && fx303) fx_group_max<GT, NKEY>(key, s_key[warp], bar);
        else fx_group_exp<GT, 2 * D>(rmag, er2, s_mag[warp], bar);
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
          R* Rin = pass == 0 ? P1 : P2;
          double* out = pass == 0 ? p.y : p.g;
          int er[D];
#pragma unroll
          for (int c = 0; c < D; ++c) er[c] = pass == 0 ? er2[D + c] : er2[c];
          if (FX303 && fx303) {
            const int k = pass == 0 ? 1 : 0, L = pass == 0 ? key[1] : key[0];
            const int Ls[3] = {L, L, L};
            er[0] = er[1] = er[D - 1] = fx_point_emax(L);
            adj3_fx<N, Q1, D, GT, true>(p.fx, er, P0, Rin, lane, bar, s_kq[warp] + k * QP, 0, Ls);
          } else {
            adj3_fx<N, Q1, D, GT>(p.fx, er, P0, Rin, lane, bar);
          }
          for (int t = lane; t < NDOF; t += GT) {
            const int gn = nodes(t);
#pragma unroll
            for (int c = 0; c < D; ++c) {
              const size_t dof = (size_t)c * p.nnode + gn;
              if (p.fixed && __ldg(p.fixed + dof)) continue;
              atomicAdd(out + dof, P0[nodal(c, t)]);
            }
          }
          group_sync<GT>(bar);
        }
      }
    } else {
      if constexpr (EG) accMin = fmin(accMin, emin);
      // ---- adjoint contraction and scatter
      if constexpr (FX) {
        int er[D];
        if (FXPA || (FX303 && fx303)) {
          if constexpr (FXPA || FX303) {
            fx_group_max<GT, NKEY>(key, s_key[warp], bar);
            if constexpr (!FXPA) key[1] = key[2] = key[0];
#pragma unroll
            for (int c = 0; c < D; ++c) er[c] = fx_point_emax(key[c]);
            adj3_fx<N, Q1, D, GT, true>(p.fx, er, P0, P1, lane, bar, s_kq[warp], FXPA ? QP : 0, key);
          }
        } else {
          fx_group_exp<GT, D>(rmag, er, s_mag[warp], bar);
          if constexpr (D == 2) adj2_fx<N, Q1, D, GT>(p.fx, er, P0, P1, lane, bar);
          else adj3_fx<N, Q1, D, GT>(p.fx, er, P0, P1, lane, bar);
        }
      } else if constexpr (D == 2) {
        __syncwarp();
        adj2<N, Q1, D, R>(sB, sG, P0, P1, lane);
      } else {
        __syncwarp();
        adj3_rb<N, Q1, D, R>(tB, tG, P0, P1, lane);
      }
      for (int t = lane; t < NDOF; t += GT) {
        const int g = nodes(t);
#pragma unroll
        for (int c = 0; c < D; ++c) {
          const size_t dof = (size_t)c * p.nnode + g;
          if (p.fixed && __ldg(p.fixed + dof)) continue;
          // (one colour per launch in the deterministic mode: no other
          // element of the launch adds to this node, so each node gets one
          // add per launch, in colour order)
          if (PA_APPLY && p.y32) atomicAdd(p.y32 + dof, float(P0[nodal(c, t)]));   // FP32 Krylov vectors
          else atomicAdd(p.y + dof, to_f64(P0[nodal(c, t)]));
        }
      }
    }
    group_sync<GT>(bar);
  }

  if constexpr (OP == OP_ENERGY || EG) {
    constexpr int BW = (WARPS * GT + 31) / 32;
    __shared__ double redF[BW], redM[BW];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      accF += __shfl_xor_sync(0xffffffffu, accF, o);
      accMin = fmin(accMin, __shfl_xor_sync(0xffffffffu, accMin, o));
    }
    if (threadIdx.x % 32 == 0) { redF[threadIdx.x / 32] = accF; redM[threadIdx.x / 32] = accMin; }
    __syncthreads();
    if (threadIdx.x == 0) {
      double f = 0.0, m = INFINITY;
      for (int w = 0; w < (FX ? (int)blockDim.x / 32 : BW); ++w) { f += redF[w]; m = fmin(m, redM[w]); }
      p.part_F[blockIdx.x] = f;
      p.part_min[blockIdx.x] = m;
    }
  }
}

// Host-side launcher for one instantiation.
template <int D, int N, int Q1, class R, int OP, bool WIDE>
int launch_elem_impl(const KParams& p, int grid, void* stream) {
  using Cfg = ElemCfg<D, N, Q1, R, OP, WIDE>;
  const int w = (p.nelem + grid - 1) / grid;
  const int threads = sizeof(R) == 4 ? Cfg::WARPS * Cfg::GT
                                     : ((w < Cfg::WARPS ? w : Cfg::WARPS) * Cfg::GT + 31) / 32 * 32;
  elem_kernel<D, N, Q1, R, OP, WIDE><<<grid, threads, Cfg::smem_bytes(), (cudaStream_t)stream>>>(p);
  return (int)cudaGetLastError();
}

// Occupancy-derived grid size, and the opt-in for > 48 KB of shared memory.
template <int D, int N, int Q1, class R, int OP, bool WIDE>
int prepare_elem_impl(int nelem, int* grid) {
  using Cfg = ElemCfg<D, N, Q1, R, OP, WIDE>;
  const size_t smem = Cfg::smem_bytes();
  const void* f = (const void*)elem_kernel<D, N, Q1, R, OP, WIDE>;
  cudaError_t err = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return (int)err;
  int per_sm = 0, dev = 0, sms = 0;
  err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, Cfg::WARPS * Cfg::GT, smem);
  if (err != cudaSuccess) return (int)err;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (per_sm < 1) return (int)cudaErrorInvalidConfiguration;
  // FP64, fewer full blocks than SMs: the elements are spread over all SMs in
  // smaller blocks instead, since the warps of a block share one narrow FP64
  // pipe.
  const int need = (nelem + Cfg::WARPS - 1) / Cfg::WARPS;
  const int full = per_sm * sms;
  if (sizeof(R) == 8 && need < sms) {
    const int w = (nelem + sms - 1) / sms;
    *grid = (nelem + w - 1) / w;
  } else {
    *grid = need < full ? need : full;
  }
  return 0;
}

// The WIDE form where it exists and every one of GB300's 152 SMs has a full
// block of 8 elements (a constant, so that prepare and launch agree).
constexpr int kWideElements = 152 * 8;
template <int D, int N, int Q1, class R, int OP>
bool use_wide(int nelem) {
  return ElemCfg<D, N, Q1, R, OP>::HAS_WIDE && nelem >= kWideElements;
}

template <int D, int N, int Q1, class R, int OP>
int launch_elem(const KParams& p, int grid, void* stream) {
  constexpr bool W = ElemCfg<D, N, Q1, R, OP>::HAS_WIDE;
  return use_wide<D, N, Q1, R, OP>(p.nelem) ? launch_elem_impl<D, N, Q1, R, OP, W>(p, grid, stream)
                                            : launch_elem_impl<D, N, Q1, R, OP, false>(p, grid, stream);
}

template <int D, int N, int Q1, class R, int OP>
int prepare_elem(int nelem, int* grid) {
  constexpr bool W = ElemCfg<D, N, Q1, R, OP>::HAS_WIDE;
  return use_wide<D, N, Q1, R, OP>(nelem) ? prepare_elem_impl<D, N, Q1, R, OP, W>(nelem, grid)
                                          : prepare_elem_impl<D, N, Q1, R, OP, false>(nelem, grid);
}

}  // namespace tmop
