// FP64 tensor-product contractions in 64-bit fixed point.
//
// Why: GB300 executes 2 FP64 operations per SM and clock, and 64 IMAD.WIDE
// (32 x 32 + 64 -> 64 bit) per SM and clock (measured: 1.90 and 56.7 lane
// operations at the 2.07 GHz maximum clock), with the integer pipe running
// beside the FP64 pipe (one DFMA and 16 IMAD.WIDE take no longer than the
// DFMA alone). A contraction is a sum of products of field values with
// constant table entries, so its operands share one exponent per element and
// component: written as integers of ~57 bits relative to the largest value,
// a multiply-add is three IMAD.WIDE with no carry handling, and the result
// is as accurate as FP64 arithmetic (whose intermediate sums round at 2^-53
// of their magnitude; the dropped parts here lie at ~2^-57 of the largest
// value). The FP64 pipe keeps the pointwise metric work only.
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

// Exponent fields of the largest magnitudes (high words m) of NC components
// among the group's threads, with the barrier that makes the group's
// shared-memory writes before it visible. s: [warps of the group][NC] words,
// rewritten only after a later barrier of the group.
template <int GT, int NC>
__device__ __forceinline__ void fx_group_exp(const unsigned* m, int* e, unsigned* s, int bar) {
  if constexpr (GT <= 32) {
#pragma unroll
    for (int c = 0; c < NC; ++c) e[c] = (int)(__reduce_max_sync(group_mask<GT>(), m[c]) >> 20);
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
      e[c] = (int)(r >> 20);
    }
  }
}

// v -> fixed point with `lsh` + 53 bits below 2^(emax - 1022), emax >= the
// exponent field of v (emax < 64: the value is irrelevant, see fx_to_f64).
__device__ __forceinline__ fx_t fx_from_f64(double v, int emax, int lsh) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  unsigned long long m = (((unsigned long long)mh << 32) | lo) << lsh;
  asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(emax - (int)((hi >> 20) & 0x7ffu)));   // clamps at 64
  return (fx_t)(m ^ (unsigned long long)(long long)((int)hi >> 31));   // (complement: off by one unit)
}

// Scale of a component's results: the exponent field of a result whose
// leading bit is bit b is b + kb. Components with a non-finite value become
// NaN, those below 2^-958 zero; these, and the exponents near the ends of the
// FP64 range, take the slow conversion (lim = all ones).
struct FxScale {
  int kb;
  unsigned lim;
  int emax;
};
__device__ __forceinline__ FxScale fx_scale(int emax, int bits, int gexp) {
  FxScale s;
  s.kb = 1 + gexp + emax - bits;
  s.lim = (emax > 1900 || emax < 150) ? 0xffffffffu : 0u;
  s.emax = emax;
  return s;
}

__device__ __forceinline__ double fx_to_f64(fx_t y, const FxScale& s) {
  const int neg = (int)(y >> 32) >> 31;
  // (the complement for the negative: off by one unit of ~2^-57)
  unsigned long long u = (unsigned long long)y ^ (unsigned long long)(long long)neg;
  const unsigned uh = (unsigned)(u >> 32);
  if (uh <= s.lim) {   // small against the component's largest value, or an extreme exponent
    const int k = s.kb - 1023, k1 = k / 2, k2 = k - k1;
    const double v = (double)y * __hiloint2double((1023 + k1) << 20, 0) * __hiloint2double((1023 + k2) << 20, 0);
    if (s.emax == 0x7ff) return __longlong_as_double(0x7ff8000000000000LL);
    return s.emax < 64 ? 0.0 : v;
  }
  unsigned b;                          // leading bit of uh, <= 29: |y| < 2^62
  asm("bfind.u32 %0, %1;" : "=r"(b) : "r"(uh));
  u = (u << (30 - b)) + 0x200u;        // leading bit 62; round the 10 low bits
  u >>= 10;
  const unsigned hi = (unsigned)(u >> 32) + (b << 20) + ((unsigned)(31 + s.kb) << 20);   // the leading bit adds one
  return __hiloint2double((int)(hi | ((unsigned)neg & 0x80000000u)), (int)(unsigned)u);
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
// -> P0: [NC][3][N][Q][Q] -> P1: A[NC][3][Q][Q][Q] (double). em: exponent
// field of the largest magnitude of each component. `lane`: the thread's
// number among the GT of its group.
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
    const FxScale sc = fx_scale(pick(c), T.xin, T.gexp);
    const fx_t* s = P0 + (c * 3) * NQQ + q01;
    double* o = P1d + (c * 3) * QQQ + q01;
    fx_t v[N];
    FxLine<N> x;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {   // (kept rolled: the kernels' code has to stay in the instruction caches)
#pragma unroll
      for (int l = 0; l < N; ++l) v[l] = s[(2 - k) * NQQ + l * QQ];
      x.set(v);
      fx_forward<N, Q1, false>(T, x, [&](int q, fx_t y) { o[k * QQQ + q * QQ] = fx_to_f64(y, sc); });
    }
#pragma unroll
    for (int l = 0; l < N; ++l) v[l] = s[l * QQ];
    x.set(v);
    fx_forward<N, Q1, true>(T, x, [&](int q, fx_t y) { o[2 * QQQ + q * QQ] = fx_to_f64(y, sc); });
  }
  group_sync<GT>(bar);
}

// 3D adjoint map. P1: R[NC][3][Q][Q][Q] (double) -> P0: [NC][3][N][Q][Q] ->
// P1: [NC][2][N][N][Q] -> P0: Y (FxNodal, double).
template <int N, int Q1, int NC, int GT>
__device__ __forceinline__ void adj3_fx(const FxTab& T, const int (&em)[NC], double* P0d, double* P1d, int lane, int bar) {
  constexpr int NNQ = N * N * Q1, NQQ = N * Q1 * Q1, QQ = Q1 * Q1, QQQ = Q1 * Q1 * Q1;
  fx_t *P0 = reinterpret_cast<fx_t*>(P0d), *P1 = reinterpret_cast<fx_t*>(P1d);
  auto pick = [&](int c) {
    int e = em[0];
#pragma unroll
    for (int k = 1; k < NC; ++k) e = c == k ? em[k] : e;
    return e;
  };
#pragma unroll 1
  for (int t = lane; t < NC * QQ; t += GT) {                  // (c, q1, q0): lines along z
    const int c = t / QQ, q01 = t % QQ, e = pick(c), sh = T.rin - 53;
    const double* s = P1d + (c * 3) * QQQ + q01;
    fx_t* o = P0 + (c * 3) * NQQ + q01;
    fx_t v[Q1];
    FxLine<Q1> x;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
#pragma unroll
      for (int q = 0; q < Q1; ++q) v[q] = fx_from_f64(s[k * QQQ + q * QQ], e, sh);
      x.set(v);
      fx_adjoint<N, Q1, true, false>(T, x, x, [&](int l, fx_t y) { o[k * NQQ + l * QQ] = y; });
    }
#pragma unroll
    for (int q = 0; q < Q1; ++q) v[q] = fx_from_f64(s[2 * QQQ + q * QQ], e, sh);
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

}  // namespace tmop
