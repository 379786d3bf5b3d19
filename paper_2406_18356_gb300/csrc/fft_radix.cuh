// Short DFTs in registers and the shared-memory padding of the FFT kernels.
#pragma once

#include "common.cuh"

namespace ms {

// cos(2 pi k / 16), k < 8
__device__ __forceinline__ double c16(int k) {
  switch (k) {
    case 0: return 1.0;
    case 1: return 0.92387953251128674;
    case 2: return 0.70710678118654752;
    case 3: return 0.38268343236508977;
    case 4: return 0.0;
    case 5: return -0.38268343236508977;
    case 6: return -0.70710678118654752;
    default: return -0.92387953251128674;
  }
}
// sin(t) = cos(pi/2 - t), and cos is even
__device__ __forceinline__ double s16(int k) { return c16(k <= 4 ? 4 - k : k - 4); }

__host__ __device__ constexpr int padi(int i) { return i + (i >> 4); }

// x * W_16^k (forward: W = exp(-2 pi i / 16); inverse: its conjugate), k < 8
// a compile-time constant after unrolling
template <typename R, bool INV>
__device__ __forceinline__ C2<R> mul_w16(C2<R> x, int k) {
  if (k == 0) return x;
  C2<R> y;
  if (k == 4) {   // -i (forward) or +i (inverse)
    y.x = INV ? -x.y : x.y;
    y.y = INV ? x.x : -x.x;
    return y;
  }
  const R c = (R)c16(k), sn = (R)s16(k);
  y.x = INV ? x.x * c - x.y * sn : x.x * c + x.y * sn;
  y.y = INV ? x.y * c + x.x * sn : x.y * c - x.x * sn;
  return y;
}

template <int LOG> __host__ __device__ constexpr int brev_c(int i) {
  int r = 0;
  for (int bit = 0; bit < LOG; ++bit) r |= ((i >> bit) & 1) << (LOG - 1 - bit);
  return r;
}
template <typename R, bool INV>
__device__ __forceinline__ void bfly(C2<R>& a, C2<R>& b, int k) {
  const C2<R> bq = mul_w16<R, INV>(b, k);
  const C2<R> aq = a;
  a.x = aq.x + bq.x;
  a.y = aq.y + bq.y;
  b.x = aq.x - bq.x;
  b.y = aq.y - bq.y;
}
// Rd-point DFT (Rd = 2, 4, 8, 16) of v in registers: bit-reversed copy, then
// log2(Rd) radix-2 decimation-in-time stages; butterfly q of stage st pairs
// i0 = (q / h) 2h + q mod h with i0 + h (h = 2^st) under the twiddle
// W_2h^(q mod h) = W_16^((q mod h) 16 / 2h)
template <typename R, int Rd, bool INV>
__device__ __forceinline__ void dft_reg(C2<R> (&v)[Rd]) {
  constexpr int LOG = Rd == 2 ? 1 : (Rd == 4 ? 2 : (Rd == 8 ? 3 : 4));
  C2<R> t[Rd];
#pragma unroll
  for (int i = 0; i < Rd; ++i) t[i] = v[brev_c<LOG>(i)];
#pragma unroll
  for (int st = 0; st < LOG; ++st) {
#pragma unroll
    for (int q = 0; q < Rd / 2; ++q) {
      const int h = 1 << st;
      const int j = q & (h - 1);
      const int i0 = ((q >> st) << (st + 1)) + j;
      bfly<R, INV>(t[i0], t[i0 + h], j * (16 / (2 * h)));
    }
  }
#pragma unroll
  for (int i = 0; i < Rd; ++i) v[i] = t[i];
}

}  // namespace ms
