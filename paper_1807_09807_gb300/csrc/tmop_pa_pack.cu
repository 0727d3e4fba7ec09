// The FP64 3D stored Hessians (45 doubles per point, OP_LINEARIZE) in the form
// of the fixed-point product (fx_stored_product in tmop_fixed.cuh), in place.
// One thread per point, the points of an element on consecutive lanes: one
// read and one write of the array (48^3 order-3 hexes, 5^3 points: 10 GB), once
// per linearisation, against the 45 conversions per point that every product
// would repeat.
#include <cuda_runtime.h>

#include "tmop_fixed.cuh"

namespace tmop {

namespace {

__global__ void __launch_bounds__(128) k_pa_pack(double* __restrict__ pa, int stride, short4* __restrict__ ex,
                                                 long long npoint, int Q) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < npoint;
       t += (long long)gridDim.x * blockDim.x) {
    const long long e = t / Q;
    double* H = pa + (size_t)e * stride + (t - e * Q);
    double h[45];
#pragma unroll
    for (int i = 0; i < 45; ++i) h[i] = H[(size_t)i * Q];
    // exponents of the largest entries of the blocks (|entry| < 2^m)
    int m[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int c = 0; c < 3; ++c) m[a][c] = -1022;
#pragma unroll
    for (int r = 0; r < 9; ++r)
#pragma unroll
      for (int c = r; c < 9; ++c) {
        const int x = (int)((fx_mag(h[r * 9 - r * (r - 1) / 2 + c - r]) >> 20)) - 1022;
        m[r / 3][c / 3] = max(m[r / 3][c / 3], x);
      }
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
    const bool zero = top < -900;   // (nothing above 2^-900)
#pragma unroll
    for (int r = 0; r < 9; ++r)
#pragma unroll
      for (int c = r; c < 9; ++c) {
        const int i = r * 9 - r * (r - 1) / 2 + c - r;
        const fx_t v = zero ? 0 : fx_from_f64(h[i], E + s[r / 3] + s[c / 3] + 1022, 4);
        const Limbs l = fx_split(v);
        H[(size_t)i * Q] = __hiloint2double(l.h, l.l);
      }
    ex[t] = make_short4((short)s[0], (short)s[1], (short)s[2],
                        (short)(top >= 1025 ? kPaNan : (zero ? kPaZero : E)));
  }
}

}  // namespace

int pa_pack(double* pa, int stride, short4* ex, int nelem, int Q, void* stream) {
  const long long n = (long long)nelem * Q, want = (n + 127) / 128;
  k_pa_pack<<<(int)(want < 152 * 16 ? want : 152 * 16), 128, 0, (cudaStream_t)stream>>>(pa, stride, ex, n, Q);
  return (int)cudaGetLastError();
}

}  // namespace tmop
