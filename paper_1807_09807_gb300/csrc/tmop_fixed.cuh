// FP64 tensor-product contractions in 64-bit fixed point.
//
// Why: an FP64 multiply-add takes GB300's FP64 pipe 17 cycles per warp and SM
// (an add or a multiply 20), a 32 x 32 + 64 -> 64 bit IMAD.WIDE the integer
// pipe 4 cycles per warp and scheduler, i.e. 1 per SM, and the two pipes run
// beside one another (measured). A contraction is a sum of products of field
// values with constant table entries, so its operands can share one exponent
// per element and component: written as integers of ~57 bits relative to the
// largest value, a multiply-add is three IMAD.WIDE with no carry handling, and
// the result is as accurate as FP64 arithmetic (whose intermediate sums round
// at 2^-53 of their magnitude; the dropped parts here lie at ~2^-57 of the
// largest value). The same holds for the products of matrix entries in the
// pointwise stage of mu303 (fx_point303) where T's entries are of one size, of
// which only the scalars stay in FP64. 48^3 order-3 hexes, gradient + Hessian
// action: 11.13 ms with FP64 contractions, 5.53 ms with these, 3.82 ms with the
// pointwise products too (FP64 instructions per element and warp 1490, 654, 98).
//
// Numbers: a value v of a component whose largest magnitude is below 2^E is
// held as round-toward-zero(v 2^(X - E)), X = xin (forward) or rin (adjoint)
// chosen on the host so that no sum of a map can leave 61 bits (fx_tables). A
// table entry c, |c| <= 1, is c 2^60 = ch 2^30 + cl with |cl| <= 2^29; a
// value is split as h 2^30 + l, 0 <= l < 2^30. A dot keeps H = sum ch h and
// M = sum (ch l + cl h); its value is H + (M >> 30), and cl l 2^-60 (at most
// 1 unit per term) is dropped. G (derivatives) carries a factor 2^-gexp.
//
// The 1D tables are centro-symmetric (B) and centro-antisymmetric (G), so
// each line of values is first split into sums and differences of mirror
// pairs, which halves the multiplications: B and G have each an even and an
// odd table over half of the points and half of the nodes.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "tmop_device.cuh"
#include "tmop_kparams.h"

namespace tmop {

typedef long long fx_t;

// An element is worked on by GT threads: part of a warp, a warp or several.
// The lanes of the group within its warp:
template <int GT>
__device__ __forceinline__ unsigned group_mask() {
  if constexpr (GT >= 32) return 0xffffffffu;
  else return ((1u << GT) - 1u) << (threadIdx.x & 31 & ~(GT - 1));
}
// Barrier of the group (named barrier `bar` where it is several warps).
template <int GT>
__device__ __forceinline__ void group_sync(int bar) {
  if constexpr (GT <= 32) __syncwarp(group_mask<GT>());
  else asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(GT) : "memory");
}

__device__ __forceinline__ unsigned fx_mag(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// The exponents used: not below 64, so that a component of zeros (or of
// magnitudes below 2^-1016 and less) becomes zeros and the exponent field of a
// result cannot fall below 1.
__device__ __forceinline__ int fx_floor(unsigned e) { return e < 64u ? 64 : (int)e; }

// Exponent fields of the largest magnitudes (high words m) of NC components
// among the group's threads, with the barrier that makes the group's
// shared-memory writes before it visible. s: [warps of the group][NC] words,
// rewritten only after a later barrier of the group.
template <int GT, int NC>
__device__ __forceinline__ void fx_group_exp(const unsigned* m, int* e, unsigned* s, int bar) {
  if constexpr (GT <= 32) {
#pragma unroll
    for (int c = 0; c < NC; ++c) e[c] = fx_floor(__reduce_max_sync(group_mask<GT>(), m[c]) >> 20);
    group_sync<GT>(bar);
  } else {
    constexpr int G = GT / 32;
    const int w = (threadIdx.x >> 5) % G;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const unsigned r = __reduce_max_sync(0xffffffffu, m[c]);
      if ((threadIdx.x & 31) == 0) s[w * NC + c] = r;
    }
    group_sync<GT>(bar);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      unsigned r = s[c];
#pragma unroll
      for (int k = 1; k < G; ++k) r = max(r, s[k * NC + c]);
      e[c] = fx_floor(r >> 20);
    }
  }
}

// v -> fixed point with `lsh` + 53 bits below 2^(emax - 1022), emax >= the
// exponent field of v and >= 64.
__device__ __forceinline__ fx_t fx_from_f64(double v, int emax, int lsh) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  unsigned long long m = (((unsigned long long)mh << 32) | lo) << lsh;
  asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(emax - (int)((hi >> 20) & 0x7ffu)));   // clamps at 64
  const long long neg = (int)hi >> 31;   // (the exact negative: -0.0 and what is shifted out become 0)
  return ((fx_t)m ^ neg) - neg;
}

// Scale of a component's values: the exponent field of a value whose leading
// bit is bit b is b + kb. A component with a non-finite value (or one above
// 2^1013, whose results might not be finite) becomes NaN.
struct FxScale {
  int kb;
  unsigned nan;
};
__device__ __forceinline__ unsigned fx_nan(int emax) { return emax >= 2036 ? 0x7ff80000u : 0u; }
__device__ __forceinline__ FxScale fx_scale(int emax, int bits, int gexp) {
  return {1 + gexp + emax - bits, fx_nan(emax)};
}

// |y| < 2^62 -> FP64, rounded to nearest (values below 2^31 in magnitude are
// exact but for their last bit). Without branches, so that several
// conversions overlap.
__device__ __forceinline__ double fx_to_f64(fx_t y, const FxScale& s) {
  const int neg = (int)(y >> 32) >> 31;
  // (the complement for the negative: off by one unit of ~2^-57)
  unsigned uh = (unsigned)((int)(y >> 32) ^ neg), ul = (unsigned)((int)y ^ neg);
  const bool low = uh == 0;            // the leading bit is in the low word
  uh = low ? ul >> 1 : uh;
  ul = low ? ul << 31 : ul;
  unsigned b;                          // leading bit of uh, <= 30
  asm("bfind.u32 %0, %1;" : "=r"(b) : "r"(uh));
  unsigned long long u = ((((unsigned long long)uh << 32) | ul) << (30 - b)) + 0x200u;   // leading bit 62; round the
  u >>= 10;                                                                               // 10 low bits
  const unsigned f = (b << 20) + ((unsigned)(s.kb + (low ? 0 : 31)) << 20);              // the leading bit adds one
  unsigned hi = (unsigned)(u >> 32) + f;
  hi = uh == 0 ? 0u : hi;
  return __hiloint2double((int)(hi | ((unsigned)neg & 0x80000000u) | s.nan), (int)(unsigned)u);
}

// 30-bit limbs of a value
struct Limbs {
  int h, l;
};
__device__ __forceinline__ Limbs fx_split(fx_t v) { return {(int)(v >> 30), (int)v & 0x3fffffff}; }

struct FxAcc {
  long long H, M;
};
__device__ __forceinline__ void fx_mac(FxAcc& a, const Limbs& v, int ch, int cl) {
  // (written out: the compiler's own form of the sign-extended product takes
  // twice the instructions)
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.H) : "r"(v.h), "r"(ch));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.M) : "r"(v.l), "r"(ch));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.M) : "r"(v.h), "r"(cl));
}
__device__ __forceinline__ fx_t fx_value(const FxAcc& a) { return a.H + (a.M >> 30); }

// Mirror sums and differences of a line of L values, as limbs.
template <int L>
struct FxLine {
  static constexpr int LH = L / 2, LE = (L + 1) / 2;
  Limbs p[LE], m[LH > 0 ? LH : 1];
  __device__ __forceinline__ void set(const fx_t* v) {
#pragma unroll
    for (int i = 0; i < LH; ++i) {
      p[i] = fx_split(v[i] + v[L - 1 - i]);
      m[i] = fx_split(v[i] - v[L - 1 - i]);
    }
    if constexpr (L % 2) p[LH] = fx_split(v[LH]);
  }
};

// nodes -> points along one line: out(q, value), with B or with G
template <int N, int Q1, bool DERIV, class OUT>
__device__ __forceinline__ void fx_forward(const FxTab& T, const FxLine<N>& x, OUT&& out) {
  constexpr int NH = N / 2, NE = (N + 1) / 2, QH = Q1 / 2, QE = (Q1 + 1) / 2;
#pragma unroll
  for (int q = 0; q < QE; ++q) {
    FxAcc s{0, 0}, d{0, 0};   // parts of q and of its mirror point with equal and with opposite sign
    if constexpr (DERIV) {
#pragma unroll
      for (int i = 0; i < NH; ++i) fx_mac(s, x.m[i], T.GoH[q * 3 + i], T.GoL[q * 3 + i]);
    } else {
#pragma unroll
      for (int i = 0; i < NE; ++i) fx_mac(s, x.p[i], T.BeH[q * 3 + i], T.BeL[q * 3 + i]);
    }
    if (q < QH) {
      if constexpr (DERIV) {
#pragma unroll
        for (int i = 0; i < NE; ++i) fx_mac(d, x.p[i], T.GeH[q * 3 + i], T.GeL[q * 3 + i]);
      } else {
#pragma unroll
        for (int i = 0; i < NH; ++i) fx_mac(d, x.m[i], T.BoH[q * 3 + i], T.BoL[q * 3 + i]);
      }
      const fx_t a = fx_value(s), b = fx_value(d);
      out(q, a + b);
      out(Q1 - 1 - q, a - b);
    } else {
      out(q, fx_value(s));
    }
  }
}

// points -> nodes along one line: out(i, value) of B^t b (+ G^t g when the
// line has a derivative part)
template <int N, int Q1, bool HASB, bool HASG, class OUT>
__device__ __forceinline__ void fx_adjoint(const FxTab& T, const FxLine<Q1>& b, const FxLine<Q1>& g, OUT&& out) {
  constexpr int NH = N / 2, NE = (N + 1) / 2, QH = Q1 / 2, QE = (Q1 + 1) / 2;
#pragma unroll
  for (int i = 0; i < NE; ++i) {
    FxAcc e{0, 0}, o{0, 0};
    if constexpr (HASB) {
#pragma unroll
      for (int q = 0; q < QE; ++q) fx_mac(e, b.p[q], T.BeH[q * 3 + i], T.BeL[q * 3 + i]);
    }
    if constexpr (HASG) {
#pragma unroll
      for (int q = 0; q < QH; ++q) fx_mac(e, g.m[q], T.GeH[q * 3 + i], T.GeL[q * 3 + i]);
    }
    if (i < NH) {
      if constexpr (HASB) {
#pragma unroll
        for (int q = 0; q < QH; ++q) fx_mac(o, b.m[q], T.BoH[q * 3 + i], T.BoL[q * 3 + i]);
      }
      if constexpr (HASG) {
#pragma unroll
        for (int q = 0; q < QE; ++q) fx_mac(o, g.p[q], T.GoH[q * 3 + i], T.GoL[q * 3 + i]);
      }
      const fx_t ve = fx_value(e), vo = fx_value(o);
      out(i, ve + vo);
      out(N - 1 - i, ve - vo);
    } else {
      out(i, fx_value(e));
    }
  }
}

// Nodal fields sit in shared memory with the x index slowest, [c][i][(l,) j],
// rows padded by N words: the lanes of the x stage (one line each) then read
// consecutive words.
template <int D, int N>
struct FxNodal {
  static constexpr int ROWS = D == 2 ? N : N * N, LS = ROWS + N, CS = N * LS;
  static __device__ __forceinline__ int at(int c, int t) { return c * CS + (t % N) * LS + t / N; }   // local node t
};

// 3D forward map of NC components. P0: X (FxNodal, double) -> P1: [NC][2][N][N][Q]
// -> P0: [NC][3][N][Q][Q] -> P1: A[NC][3][Q][Q][Q] (fixed point at fx_scale(em,
// xin, gexp): the pointwise stage converts them, one point per thread). em:
// exponent field of the largest magnitude of each component. `lane`: the
// thread's number among the GT of its group.
template <int N, int Q1, int NC, int GT>
__device__ __forceinline__ void fwd3_fx(const FxTab& T, const int (&em)[NC], double* P0d, double* P1d, int lane, int bar) {
  constexpr int NNQ = N * N * Q1, NQQ = N * Q1 * Q1, QQ = Q1 * Q1, QQQ = Q1 * Q1 * Q1;
  fx_t *P0 = reinterpret_cast<fx_t*>(P0d), *P1 = reinterpret_cast<fx_t*>(P1d);
  auto pick = [&](int c) {
    int e = em[0];
#pragma unroll
    for (int k = 1; k < NC; ++k) e = c == k ? em[k] : e;
    return e;
  };
#pragma unroll 1
  for (int t = lane; t < NC * N * N; t += GT) {               // (c, l, j): lines along x
    const int c = t / (N * N), lj = t % (N * N), e = pick(c);
    fx_t v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = fx_from_f64(P0d[c * FxNodal<3, N>::CS + i * FxNodal<3, N>::LS + lj], e, T.xin - 53);
    FxLine<N> x;
    x.set(v);
    fx_t* o = P1 + (c * 2) * NNQ + lj * Q1;
    fx_forward<N, Q1, false>(T, x, [&](int q, fx_t y) { o[q] = y; });
    fx_forward<N, Q1, true>(T, x, [&](int q, fx_t y) { o[NNQ + q] = y; });
  }
  group_sync<GT>(bar);
#pragma unroll 1
  for (int t = lane; t < NC * N * Q1; t += GT) {              // (c, l, q0): lines along y
    const int q0 = t % Q1, l = (t / Q1) % N, c = t / (Q1 * N);
    const fx_t* s = P1 + (c * 2) * NNQ + l * N * Q1 + q0;
    fx_t* o = P0 + (c * 3) * NQQ + l * QQ + q0;
    fx_t v[N];
    FxLine<N> x;
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = s[j * Q1];
    x.set(v);
    fx_forward<N, Q1, false>(T, x, [&](int q, fx_t y) { o[q * Q1] = y; });
    fx_forward<N, Q1, true>(T, x, [&](int q, fx_t y) { o[NQQ + q * Q1] = y; });
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = s[NNQ + j * Q1];
    x.set(v);
    fx_forward<N, Q1, false>(T, x, [&](int q, fx_t y) { o[2 * NQQ + q * Q1] = y; });
  }
  group_sync<GT>(bar);
#pragma unroll 1
  for (int t = lane; t < NC * QQ; t += GT) {                  // (c, q1, q0): lines along z
    const int c = t / QQ, q01 = t % QQ;
    const fx_t* s = P0 + (c * 3) * NQQ + q01;
    fx_t* o = P1 + (c * 3) * QQQ + q01;
    fx_t v[N];
    FxLine<N> x;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {   // (kept rolled: the kernels' code has to stay in the instruction caches)
#pragma unroll
      for (int l = 0; l < N; ++l) v[l] = s[(2 - k) * NQQ + l * QQ];
      x.set(v);
      fx_forward<N, Q1, false>(T, x, [&](int q, fx_t y) { o[k * QQQ + q * QQ] = y; });
    }
#pragma unroll
    for (int l = 0; l < N; ++l) v[l] = s[l * QQ];
    x.set(v);
    fx_forward<N, Q1, true>(T, x, [&](int q, fx_t y) { o[2 * QQQ + q * QQ] = y; });
  }
  group_sync<GT>(bar);
}

// y shifted left by sh bits (right, with its sign, for sh < 0)
__device__ __forceinline__ fx_t fx_align(fx_t y, int sh) {
  const int r = min(max(-sh, 0), 63), l = max(sh, 0);
  return (fx_t)((unsigned long long)y << l) >> r;
}

// 3D adjoint map. P1: R[NC][3][Q][Q][Q] (double) -> P0: [NC][3][N][Q][Q] ->
// P1: [NC][2][N][N][Q] -> P0: Y (FxNodal, double).
// RAW: R is in fixed point instead, point q of component c at exponent
// kq[c kst + q] (FxPoint::E) in an element whose largest key is L[c].
template <int N, int Q1, int NC, int GT, bool RAW = false>
__device__ __forceinline__ void adj3_fx(const FxTab& T, const int (&em)[NC], double* P0d, double* P1d, int lane, int bar,
                                        const short* kq = nullptr, int kst = 0, const int* L = nullptr) {
  constexpr int NNQ = N * N * Q1, NQQ = N * Q1 * Q1, QQ = Q1 * Q1, QQQ = Q1 * Q1 * Q1;
  fx_t *P0 = reinterpret_cast<fx_t*>(P0d), *P1 = reinterpret_cast<fx_t*>(P1d);
  auto pick = [&](int c) {
    int e = em[0];
#pragma unroll
    for (int k = 1; k < NC; ++k) e = c == k ? em[k] : e;
    return e;
  };
  auto pickL = [&](int c) {
    int l = L[0];
#pragma unroll
    for (int k = 1; k < NC; ++k) l = c == k ? L[k] : l;
    return l;
  };
#pragma unroll 1
  for (int t = lane; t < NC * QQ; t += GT) {                  // (c, q1, q0): lines along z
    const int c = t / QQ, q01 = t % QQ, e = pick(c), sh = T.rin - 53;
    const double* s = P1d + (c * 3) * QQQ + q01;
    fx_t* o = P0 + (c * 3) * NQQ + q01;
    fx_t v[Q1];
    FxLine<Q1> x;
    int al[RAW ? Q1 : 1];
    if constexpr (RAW) {
#pragma unroll
      for (int q = 0; q < Q1; ++q) al[q] = kq[c * kst + q * QQ + q01] - pickL(c) + T.rin - 33;
    }
    auto in = [&](int i, int q) -> fx_t {
      if constexpr (RAW) return fx_align(reinterpret_cast<const fx_t*>(s)[i], al[q]);
      else return fx_from_f64(s[i], e, sh);
    };
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
#pragma unroll
      for (int q = 0; q < Q1; ++q) v[q] = in(k * QQQ + q * QQ, q);
      x.set(v);
      fx_adjoint<N, Q1, true, false>(T, x, x, [&](int l, fx_t y) { o[k * NQQ + l * QQ] = y; });
    }
#pragma unroll
    for (int q = 0; q < Q1; ++q) v[q] = in(2 * QQQ + q * QQ, q);
    x.set(v);
    fx_adjoint<N, Q1, false, true>(T, x, x, [&](int l, fx_t y) { o[2 * NQQ + l * QQ] = y; });
  }
  group_sync<GT>(bar);
#pragma unroll 1
  for (int t = lane; t < NC * N * Q1; t += GT) {              // (c, l, q0): lines along y
    const int q0 = t % Q1, l = (t / Q1) % N, c = t / (Q1 * N);
    const fx_t* s = P0 + (c * 3) * NQQ + l * QQ + q0;
    fx_t* o = P1 + (c * 2) * NNQ + l * N * Q1 + q0;
    fx_t v[Q1];
    FxLine<Q1> x, g;
#pragma unroll
    for (int q = 0; q < Q1; ++q) v[q] = s[q * Q1];
    x.set(v);
    fx_adjoint<N, Q1, true, false>(T, x, x, [&](int j, fx_t y) { o[j * Q1] = y; });             // pairs with G in x
#pragma unroll
    for (int q = 0; q < Q1; ++q) v[q] = s[NQQ + q * Q1];
    g.set(v);
#pragma unroll
    for (int q = 0; q < Q1; ++q) v[q] = s[2 * NQQ + q * Q1];
    x.set(v);
    fx_adjoint<N, Q1, true, true>(T, x, g, [&](int j, fx_t y) { o[NNQ + j * Q1] = y; });        // pairs with B in x
  }
  group_sync<GT>(bar);
#pragma unroll 1
  for (int t = lane; t < NC * N * N; t += GT) {               // (c, l, j): lines along x
    const int c = t / (N * N), lj = t % (N * N);
    const FxScale sc = fx_scale(pick(c), T.rin, T.gexp);
    const fx_t* s = P1 + (c * 2) * NNQ + lj * Q1;
    double* o = P0d + c * FxNodal<3, N>::CS + lj;
    fx_t v[Q1];
    FxLine<Q1> x, g;
#pragma unroll
    for (int q = 0; q < Q1; ++q) v[q] = s[q];
    g.set(v);
#pragma unroll
    for (int q = 0; q < Q1; ++q) v[q] = s[NNQ + q];
    x.set(v);
    fx_adjoint<N, Q1, true, true>(T, x, g, [&](int i, fx_t y) { o[i * FxNodal<3, N>::LS] = fx_to_f64(y, sc); });
  }
  group_sync<GT>(bar);
}

// 2D forward map. P0: X (FxNodal) -> P1: [NC][2][N][Q] -> P0: A[NC][2][Q][Q]
template <int N, int Q1, int NC, int GT>
__device__ __forceinline__ void fwd2_fx(const FxTab& T, const int (&em)[NC], double* P0d, double* P1d, int lane, int bar) {
  constexpr int NQ = N * Q1, QQ = Q1 * Q1;
  fx_t* P1 = reinterpret_cast<fx_t*>(P1d);
  auto pick = [&](int c) {
    int e = em[0];
#pragma unroll
    for (int k = 1; k < NC; ++k) e = c == k ? em[k] : e;
    return e;
  };
#pragma unroll 1
  for (int t = lane; t < NC * N; t += GT) {                   // (c, j): lines along x
    const int c = t / N, j = t % N, e = pick(c);
    fx_t v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = fx_from_f64(P0d[c * FxNodal<2, N>::CS + i * FxNodal<2, N>::LS + j], e, T.xin - 53);
    FxLine<N> x;
    x.set(v);
    fx_t* o = P1 + (c * 2) * NQ + j * Q1;
    fx_forward<N, Q1, false>(T, x, [&](int q, fx_t y) { o[q] = y; });
    fx_forward<N, Q1, true>(T, x, [&](int q, fx_t y) { o[NQ + q] = y; });
  }
  group_sync<GT>(bar);
#pragma unroll 1
  for (int t = lane; t < NC * Q1; t += GT) {                  // (c, q0): lines along y
    const int q0 = t % Q1, c = t / Q1;
    const FxScale sc = fx_scale(pick(c), T.xin, T.gexp);
    const fx_t* s = P1 + (c * 2) * NQ + q0;
    double* o = P0d + (c * 2) * QQ + q0;
    fx_t v[N];
    FxLine<N> x;
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = s[NQ + j * Q1];
    x.set(v);
    fx_forward<N, Q1, false>(T, x, [&](int q, fx_t y) { o[q * Q1] = fx_to_f64(y, sc); });        // d/dxi_0
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = s[j * Q1];
    x.set(v);
    fx_forward<N, Q1, true>(T, x, [&](int q, fx_t y) { o[QQ + q * Q1] = fx_to_f64(y, sc); });    // d/dxi_1
  }
  group_sync<GT>(bar);
}

// 2D adjoint map. P0: R[NC][2][Q][Q] -> P1: [NC][2][N][Q] -> P0: Y (FxNodal)
template <int N, int Q1, int NC, int GT>
__device__ __forceinline__ void adj2_fx(const FxTab& T, const int (&em)[NC], double* P0d, double* P1d, int lane, int bar) {
  constexpr int NQ = N * Q1, QQ = Q1 * Q1;
  fx_t* P1 = reinterpret_cast<fx_t*>(P1d);
  auto pick = [&](int c) {
    int e = em[0];
#pragma unroll
    for (int k = 1; k < NC; ++k) e = c == k ? em[k] : e;
    return e;
  };
#pragma unroll 1
  for (int t = lane; t < NC * Q1; t += GT) {                  // (c, q0): lines along y
    const int q0 = t % Q1, c = t / Q1, e = pick(c), sh = T.rin - 53;
    const double* s = P0d + (c * 2) * QQ + q0;
    fx_t* o = P1 + (c * 2) * NQ + q0;
    fx_t v[Q1];
    FxLine<Q1> x;
#pragma unroll
    for (int q = 0; q < Q1; ++q) v[q] = fx_from_f64(s[q * Q1], e, sh);
    x.set(v);
    fx_adjoint<N, Q1, true, false>(T, x, x, [&](int j, fx_t y) { o[j * Q1] = y; });             // pairs with G in x
#pragma unroll
    for (int q = 0; q < Q1; ++q) v[q] = fx_from_f64(s[QQ + q * Q1], e, sh);
    x.set(v);
    fx_adjoint<N, Q1, false, true>(T, x, x, [&](int j, fx_t y) { o[NQ + j * Q1] = y; });        // pairs with B in x
  }
  group_sync<GT>(bar);
#pragma unroll 1
  for (int t = lane; t < NC * N; t += GT) {                   // (c, j): lines along x
    const int c = t / N, j = t % N;
    const FxScale sc = fx_scale(pick(c), T.rin, T.gexp);
    const fx_t* s = P1 + (c * 2) * NQ + j * Q1;
    double* o = P0d + c * FxNodal<2, N>::CS + j;
    fx_t v[Q1];
    FxLine<Q1> x, g;
#pragma unroll
    for (int q = 0; q < Q1; ++q) v[q] = s[q];
    g.set(v);
#pragma unroll
    for (int q = 0; q < Q1; ++q) v[q] = s[NQ + q];
    x.set(v);
    fx_adjoint<N, Q1, true, true>(T, x, g, [&](int i, fx_t y) { o[i * FxNodal<2, N>::LS] = fx_to_f64(y, sc); });
  }
  group_sync<GT>(bar);
}

// High word of a value's magnitude (of its complement for a negative one).
__device__ __forceinline__ unsigned fx_word(fx_t y) { return (unsigned)((int)(y >> 32) ^ ((int)(y >> 32) >> 31)); }

// Bits to shift the nine entries of a point up by: to |entries| < 2^59 by the
// largest one, or none (< 2^59.4 by fx_tables). By the point's own largest
// entry: products of entries have a fixed number of bits, so at a point whose T
// is r times smaller than the element's largest one would lose r^2 of the
// cofactors and r^3 of det T to that one's scale (order-3 hexes graded to r =
// 100: det T to 1e-11).
template <int ST>
__device__ __forceinline__ int fx_room(const fx_t* T) {
  unsigned top = 0;   // (the same leading bit as the largest magnitude)
#pragma unroll
  for (int i = 0; i < 9; ++i) top |= fx_word(T[i * ST]);
  return max(__clz((int)top) - 5, 0);
}

// Bits to shift a point's T up by (up), and whether it has a row or a column
// more than about four times smaller than its largest entry, which sends the
// point to the FP64 stage (fx_point_pack): products of the small entries of an
// element long in one direction (aspect r) lose r^2 to the scale of the long
// ones, where FP64 loses r to the map (order-3 hexes of aspect 1000: gradient to
// 2e-11 in fixed point, 4e-13 in FP64). Point by point and not by the element:
// 16^3 order-4 hexes with nodes moved by a tenth of their spacing, gradient +
// Hessian action 328 us, 390 with the whole element in FP64, 291 without the test.
template <int ST>
__device__ __forceinline__ bool fx_thin(const fx_t* T, int& up) {
  unsigned w[6] = {};   // rows, columns
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const unsigned m = fx_word(T[i * ST]);
    w[i / 3] |= m;
    w[3 + i % 3] |= m;
  }
  const unsigned top = w[0] | w[1] | w[2];
  up = max(__clz((int)top) - 5, 0);
  return min(min(min(w[0], w[1]), min(w[2], w[3])), min(w[4], w[5])) < top >> 2;
}

// mu303 at one point in fixed point (W = I): s P (GRAD, in place of T) and s dP
// in direction V (HESS, in place of V), s = w det W, with
//   P = cA T + ct C,  dP = cA V + bT T + bC C + ct dC[V]   (MetricAct),
// where only the scalars (from |T|^2, det T, T:V and C:V) are FP64: one FP64
// operation takes as long as ~17 IMAD.WIDE. T, V: entries [3][3] at stride ST,
// of one scale each (FxScale::kb kT, kV), shifted up by what the point has to
// spare (fx_room).
// Magnitudes: |T|, |V|, |C| < 2^59, |dC| < 2^60, coefficients < 2^59 under a
// common exponent per point, so all sums of limb products are < 2^63 and the
// results < 2^61; a product loses ~2^-56 of the largest one.
// A result is y 2^(E - 2044); E and the bits of the magnitudes per point are
// returned for the adjoint map, which gives the element one exponent.
struct FxPoint {
  int E;                       // exponent of the point's results
  unsigned hi = 0, lo = 0;     // the magnitudes' words, or-ed: the leading bit of the largest one
  // (Both words: where the terms of P or of a product cancel, as near an ideal
  // mesh, all entries can lie below 2^32 and still hold 25 good bits.)
  __device__ __forceinline__ void add(fx_t y) {
    const int neg = (int)(y >> 32) >> 31;
    hi |= (unsigned)((int)(y >> 32) ^ neg);
    lo |= (unsigned)((int)y ^ neg);
  }
  __device__ __forceinline__ bool zero() const { return (hi | lo) == 0; }
};
// Elements whose x - x_0 has a largest component within 2^-kFx303X and
// 2^kFx303X (and v within 2^-kFx303V and 2^kFx303V) take this stage, the others
// the FP64 one. At a point |T| can be 2^57 smaller than the element's, and det T
// 2^58 smaller than |T|^3: with |T| within 2^-101 and 2^46, tau lies within
// 2^-361 and 2^138, so cA and ct, the gradient's scalars, within 2^-100 and
// 2^400. Those of dP can leave the range at such a point where v is large, as
// they do in FP64: results are then NaN (dP's E below).
constexpr int kFx303X = 40, kFx303V = 610;
constexpr int kFxNan = 32000;   // E of a point whose results are not finite
template <int ST, bool GRAD, bool HESS>
__device__ __forceinline__ bool fx_point303(fx_t* T, fx_t* V, int upT, int kT, int kV, double s, FxPoint& pg,
                                            FxPoint& ph, double& mu, double& tau) {
  Limbs a[9], c[9], v[HESS ? 9 : 1];
  const int upV = HESS ? fx_room<ST>(V) : 0;
  kT -= upT;
  kV -= upV;
  const int kC = 2 * kT + 60 - 1023;
  long long H = 0, M = 0;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    a[i] = fx_split((fx_t)((unsigned long long)T[i * ST] << upT));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(H) : "r"(a[i].h), "r"(a[i].h));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(M) : "r"(a[i].h), "r"(a[i].l));
  }
  const double I1 = fx_to_f64(H + (M >> 29), {kC, 0u});
  auto minor = [](const Limbs* x, const Limbs* y, int i, FxAcc& p, FxAcc& m) {   // x_p y_q and x_m y_n of entry i
    const int r1 = 3 * ((i / 3 + 1) % 3), r2 = 3 * ((i / 3 + 2) % 3), c1 = (i % 3 + 1) % 3, c2 = (i % 3 + 2) % 3;
    fx_mac(p, x[r1 + c1], y[r2 + c2].h, y[r2 + c2].l);
    fx_mac(m, x[r1 + c2], y[r2 + c1].h, y[r2 + c1].l);
  };
  FxAcc at{0, 0};
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    FxAcc p{0, 0}, m{0, 0};
    minor(a, a, i, p, m);
    c[i] = fx_split((p.H - m.H) + ((p.M - m.M) >> 30));
    if (i < 3) fx_mac(at, a[i], c[i].h, c[i].l);
  }
  tau = fx_to_f64(fx_value(at), {kT + kC + 60 - 1023, 0u});
  const bool ok = tau > 0.0;
  double t = 0.0, d = 0.0;
  if constexpr (HESS) {
    long long Ht = 0, Ma = 0, Mb = 0, Hd = 0, Mc = 0, Md = 0;   // (9 cross terms per sum)
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      v[i] = fx_split((fx_t)((unsigned long long)V[i * ST] << upV));
      asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(Ht) : "r"(a[i].h), "r"(v[i].h));
      asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(Ma) : "r"(a[i].h), "r"(v[i].l));
      asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(Mb) : "r"(a[i].l), "r"(v[i].h));
      asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(Hd) : "r"(c[i].h), "r"(v[i].h));
      asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(Mc) : "r"(c[i].h), "r"(v[i].l));
      asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(Md) : "r"(c[i].l), "r"(v[i].h));
    }
    t = fx_to_f64(Ht + (Ma >> 30) + (Mb >> 30), {kT + kV + 60 - 1023, 0u});
    d = fx_to_f64(Hd + (Mc >> 30) + (Md >> 30), {kC + kV + 60 - 1023, 0u});
  }
  // the scalars, as in MetricAct::init and dP
  const double r = rcbrt_nr(ok ? tau : 1.0), r2 = r * r, it = r2 * r;
  const double cA = ok ? ((2.0 / 3.0) * s) * r2 : 0.0;
  const double c1t = cA * ((-2.0 / 3.0) * it);
  const double ct = c1t * (0.5 * I1);
  mu = fma((1.0 / 3.0) * I1, r2, -1.0);
  auto ex = [](double x) { return (int)((unsigned)__double2hiint(x) >> 20 & 0x7ffu); };
  if constexpr (GRAD) {
    const int E = max(ex(cA) + kT, ex(ct) + kC);
    const Limbs gT = fx_split(fx_from_f64(cA, E - kT, 6)), gC = fx_split(fx_from_f64(ct, E - kC, 6));
    pg = {E};
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      FxAcc z{0, 0};
      fx_mac(z, a[i], gT.h, gT.l);
      fx_mac(z, c[i], gC.h, gC.l);
      const fx_t y = ok ? fx_value(z) : 0;
      T[i * ST] = y;
      pg.add(y);
    }
  }
  if constexpr (HESS) {
    const double ctt = (ct * it) * (-5.0 / 3.0);
    const double bT = c1t * d, bC = fma(c1t, t, ctt * d);
    const int kD = kT + kV + 60 - 1023;
    const int E = max(max(ex(cA) + kV, ex(bT) + kT), max(ex(bC) + kC, ex(ct) + kD));
    const bool finite = max(ex(bT), ex(bC)) < 2047;
    const Limbs hV = fx_split(fx_from_f64(cA, E - kV, 6)), hT = fx_split(fx_from_f64(bT, E - kT, 6));
    const Limbs hC = fx_split(fx_from_f64(bC, E - kC, 6)), hD = fx_split(fx_from_f64(ct, E - kD, 6));
    ph = {E};
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      FxAcc p{0, 0}, n{0, 0}, z{0, 0};
      minor(v, a, i, p, n);
      minor(a, v, i, p, n);
      const Limbs dc = fx_split((p.H - n.H) + ((p.M - n.M) >> 30));
      fx_mac(z, dc, hD.h, hD.l);
      fx_mac(z, v[i], hV.h, hV.l);
      fx_mac(z, a[i], hT.h, hT.l);
      fx_mac(z, c[i], hC.h, hC.l);
      const fx_t y = ok ? fx_value(z) : 0;
      V[i * ST] = y;
      ph.add(y);
    }
    if (!finite) ph = {kFxNan, 1u << 30};
  }
  return ok;
}

// A point's nine results from the FP64 stage, in place: doubles to integers
// below 2^59 under one exponent, as fx_point303 leaves them.
template <int ST>
__device__ __forceinline__ FxPoint fx_point_pack(double* R) {
  unsigned m = 0;
#pragma unroll
  for (int i = 0; i < 9; ++i) m = max(m, fx_mag(R[i * ST]));
  const int e = fx_floor(m >> 20);
  FxPoint pt = {e + 2044 - 1022 - 59};
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const fx_t y = fx_from_f64(R[i * ST], e, 6);
    reinterpret_cast<fx_t*>(R)[i * ST] = y;
    pt.add(y);
  }
  if (fx_nan(e)) pt = {kFxNan, 1u << 30};
  return pt;
}

// Largest values of NK keys over the group, with a barrier (as fx_group_exp).
template <int GT, int NK>
__device__ __forceinline__ void fx_group_max(int* key, int* s, int bar) {
#pragma unroll
  for (int k = 0; k < NK; ++k) key[k] = __reduce_max_sync(group_mask<GT>(), key[k]);
  if constexpr (GT > 32) {
    constexpr int G = GT / 32;
    const int w = (threadIdx.x >> 5) % G;
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
      for (int k = 0; k < NK; ++k) s[w * NK + k] = key[k];
    }
    group_sync<GT>(bar);
#pragma unroll
    for (int k = 0; k < NK; ++k)
#pragma unroll
      for (int w2 = 0; w2 < G; ++w2) key[k] = max(key[k], s[w2 * NK + k]);
  } else {
    group_sync<GT>(bar);
  }
}

// ---------------------------------------------------------------- stored Hessians
// The FP64 3D stored Hessians are packed for the fixed-point product by the
// linearisation (fx_pack_point): the 45 entries H_(r,c) of a point, r = 3 a + b, as
//   H_(r,c) = (h 2^30 + l) 2^(E + s_a + s_c - 57),  |h| <= 2^27, 0 <= l < 2^30,
// (h, l) in the place of the double's high and low word, and {s_0, s_1, s_2, E}
// beside them; s_a is half the exponent of block (a, a), so that directions
// along which elements are long or short keep their digits.
// (The least of their digits are not missed: an error of 2^-57 of a block's
// largest entry stays below what FP64 rounding of dA, relative to the largest
// nodal value of v, does through that entry. On elements of aspect 1 to 1000, in
// rows or columns, the product's error from it is 1e-17 to 7e-15 where FP64
// arithmetic has 1e-16 to 1e-12.)
constexpr int kPaNan = 32767, kPaZero = -20000;   // E of a point with a non-finite entry, of one without any

// Packs the 45 entries h of a point to H[i st], their exponents to *ex; ok: the
// point's T has a Hessian (else zeros).
__device__ __forceinline__ void fx_pack_point(const double (&h)[45], bool ok, double* H, int st, short4* ex) {
  // largest entries of the blocks: their high words, then exponents (|entry| < 2^m)
  unsigned w[3][3] = {};
#pragma unroll
  for (int r = 0; r < 9; ++r)
#pragma unroll
    for (int c = r; c < 9; ++c)
      w[r / 3][c / 3] = max(w[r / 3][c / 3], fx_mag(h[r * 9 - r * (r - 1) / 2 + c - r]));
  int m[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int c = a; c < 3; ++c) m[a][c] = (int)(w[a][c] >> 20) - 1022;
  const int top = max(max(max(m[0][0], m[1][1]), max(m[2][2], m[0][1])), max(m[0][2], m[1][2]));
  // half the exponents of the diagonal blocks, or one for all where they do
  // not bound the others (an indefinite point can have a small one)
  int s[3] = {m[0][0] >> 1, m[1][1] >> 1, m[2][2] >> 1};
  const bool even = m[0][1] > s[0] + s[1] + 8 || m[0][2] > s[0] + s[2] + 8 || m[1][2] > s[1] + s[2] + 8 ||
                    min(m[0][0], min(m[1][1], m[2][2])) < -900;
  if (even) s[0] = s[1] = s[2] = top >> 1;
  int E = -100000;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int c = a; c < 3; ++c) E = max(E, m[a][c] - s[a] - s[c]);
  const bool zero = !ok || top < -900;            // (nothing above 2^-900)
  const int base = zero ? 4096 : E + 1022;        // (zero: everything is shifted out)
#pragma unroll
  for (int r = 0; r < 9; ++r)
#pragma unroll
    for (int c = r; c < 9; ++c) {
      const int i = r * 9 - r * (r - 1) / 2 + c - r;
      const Limbs l = fx_split(fx_from_f64(h[i], base + s[r / 3] + s[c / 3], 4));
      H[(size_t)i * st] = __hiloint2double(l.h, l.l);
    }
  *ex = make_short4((short)s[0], (short)s[1], (short)s[2], (short)(zero ? kPaZero : (top >= 1025 ? kPaNan : E)));
}

// y = H dA at one point: h the packed entries, ex their exponents; A: dA in
// fixed point at stride ST (rows' scales kb), shifted up by what the point has
// to spare (fx_room); the rows are first brought to one exponent under the
// scaling of H. y replaces dA; pt: per row.
template <int ST>
__device__ __forceinline__ void fx_stored_product(fx_t* A, const double* h, short4 ex, const FxScale* sA, FxPoint* pt) {
  const int s[3] = {ex.x, ex.y, ex.z}, up = fx_room<ST>(A);
  int m[3], mx = -100000;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    m[a] = sA[a].kb + s[a];
    mx = max(mx, m[a]);
  }
  Limbs d[9];
#pragma unroll
  for (int i = 0; i < 9; ++i)
    d[i] = fx_split((fx_t)((unsigned long long)A[i * ST] << up) >> min(mx - m[i / 3], 63));
#pragma unroll
  for (int a = 0; a < 3; ++a) pt[a] = {s[a] + ex.w + mx - up + 1024};
#pragma unroll
  for (int r = 0; r < 9; ++r) {
    FxAcc z{0, 0};   // 9 terms: |H| < 9 2^56, |M| < 9 (2^59 + 2^57) < 2^63
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      const int lo = r < c ? r : c, hi = r < c ? c : r, t = lo * 9 - lo * (lo - 1) / 2 + hi - lo;
      fx_mac(z, d[c], __double2hiint(h[t]), __double2loint(h[t]));
    }
    const fx_t y = fx_value(z);
    A[r * ST] = y;
    pt[r / 3].add(y);
  }
}

// The key whose maximum over the points gives the element's exponent (L; with
// kFxNan one that fx_scale takes for not finite), and the exponent field of the largest magnitude (as fx_group_exp's) from it. Not
// below kFxKeyMin, whose field is fx_floor's 64: what lies below (fields that
// are zero, products that underflow) becomes zero, and the exponent field of a
// result cannot leave its range.
constexpr int kFxKeyMin = 64 + 2044 - 1022 - 33;
__device__ __forceinline__ int fx_point_key(const FxPoint& p) {
  unsigned b;   // leading bit of the word
  asm("bfind.u32 %0, %1;" : "=r"(b) : "r"(p.hi ? p.hi : p.lo));
  return p.zero() ? kFxKeyMin : p.E + (int)b - (p.hi ? 0 : 32);
}
__device__ __forceinline__ int fx_point_emax(int L) { return L + 33 - 2044 + 1022; }
}  // namespace tmop
