// Transforms of the 2d row and column passes on power-of-two sides (8 <= n <= 1024): a batch of
// sequences in shared memory, in place, radix 4 (one radix-2 stage at the end when log2 n is
// odd, twiddle-free).  Forward by decimation in frequency, natural order in and digit-reversed
// positions out; the inverse runs the stages backwards, so nothing is permuted and a stage
// costs one barrier and one pass over shared memory.  Callers translate positions to modes
// where they read or write global memory.
//
// The passes are bound by latency (a stage is a shared load, a chain of dependent double-float
// or float64 operations, a shared store and a barrier), then by the float64 pipe.  Against
// Stockham stages with two barriers each and twiddles gathered from a table in global memory,
// double-float at 512 x 512 (one GB300): a column pass over two planes 20.0 -> 14.8 us, a row
// pass over one pair 15.5 -> 12.7 us; RK4 runs at 256 x 256 in float64 1.22 and at 512 x 512
// mixed 1.08 times as fast (ratios of paired runs: the same build differs by a fifth between
// machines).
#pragma once
#include "sgn_2d_dev.cuh"

namespace sgn {
namespace d2 {

// Swizzle of a position: the 16-byte bank (low three bits) is XORed with a GF(2)-linear function
// of bits 3..9 chosen so that eight lanes of a stage (bits of any radix-4 or radix-2 digit and
// the bits next to it) and eight lanes that walk the modes (the topmost digits) each touch
// eight different banks.
__device__ __forceinline__ int sw2(int a) {
  const int m = a >> 3, u = (m ^ (m >> 4)) & 15;
  return a ^ (int)((0x0356217447126530ull >> (4 * u)) & 7);
}

// Stride of TW columns of ny: the columns lie 8 / TW 16-byte banks apart.
template <int TW>
__host__ __device__ constexpr int col_stride(int ny) { return TW == 1 ? ny : ny + 8 / TW; }

// digits of two bits, reversed (bits even)
__device__ __forceinline__ int dig_rev(int x, int bits) {
  const unsigned r = __brev((unsigned)x) >> (32 - bits);
  return (int)(((r & 0x55555555u) << 1) | ((r >> 1) & 0x55555555u));
}
// position of mode k of a length-2^l transform, and mode at position p
__device__ __forceinline__ int pos_of(int k, int l) {
  const int odd = l & 1, b = l - odd;
  return (dig_rev(k & ((1 << b) - 1), b) << odd) | (k >> b);
}
__device__ __forceinline__ int mode_at(int p, int l) {
  const int odd = l & 1, b = l - odd;
  return dig_rev(p >> odd, b) | ((p & odd) << b);
}

// Twiddles in shared memory, n entries: the stage of element distance sg has e^{-2 pi i s j/(4 sg)}
// at n - 4 sg + (s - 1) sg + j (s = 1..3, j < sg), so the lanes of a warp read consecutive entries.
template <typename T>
__device__ __forceinline__ void fill_tw2(cplx<T>* tab, int l, const cplx<T>* __restrict__ tw) {
  const int n = 1 << l;
  for (int m = threadIdx.x; m < n - 2; m += blockDim.x) {
    const int f = 31 - __clz(n - m - 1), ls = f - ((f ^ l) & 1);
    const int r = m - n + (4 << ls);
    const int s = (r >> ls) + 1, j = r & ((1 << ls) - 1);
    tab[m] = tw[(j * s) << (kTwiddleLog2 - 2 - ls)];
  }
}

template <typename T, bool INV>
__device__ __forceinline__ void dft4(cplx<T>& a0, cplx<T>& a1, cplx<T>& a2, cplx<T>& a3) {
  const cplx<T> s02 = a0 + a2, d02 = a0 - a2, s13 = a1 + a3, d13 = a1 - a3;
  const cplx<T> r13 = INV ? mul_pi(d13) : mul_mi(d13);
  a0 = s02 + s13;
  a1 = d02 + r13;
  a2 = s02 - s13;
  a3 = d02 - r13;
}

// The radix-4 stage of element distance 2^ls, and its barrier.
template <typename T, bool INV>
__device__ __forceinline__ void stage4(cplx<T>* buf, int l, int nb, int stride,
                                       const cplx<T>* tab, int ls) {
  const int lb = l - 2, sg = 1 << ls;
  const cplx<T>* w = tab + (1 << l) - 4 * sg;
  const int d1 = sw2(sg), d2 = sw2(2 * sg);
#pragma unroll 1
  for (int g = threadIdx.x; g < (nb << lb); g += blockDim.x) {
    const int x = g & ((1 << lb) - 1), i = x & (sg - 1);
    cplx<T>* s = buf + (g >> lb) * stride;
    const int a = sw2(((x ^ i) << 2) | i);
    cplx<T> a0 = s[a], a1 = s[a ^ d1], a2 = s[a ^ d2], a3 = s[a ^ d1 ^ d2];
    if (INV && ls > 0) {
      a1 = cmul_tw(a1, w[i], true);
      a2 = cmul_tw(a2, w[sg + i], true);
      a3 = cmul_tw(a3, w[2 * sg + i], true);
    }
    dft4<T, INV>(a0, a1, a2, a3);
    if (!INV && ls > 0) {
      a1 = cmul_tw(a1, w[i], false);
      a2 = cmul_tw(a2, w[sg + i], false);
      a3 = cmul_tw(a3, w[2 * sg + i], false);
    }
    s[a] = a0;
    s[a ^ d1] = a1;
    s[a ^ d2] = a2;
    s[a ^ d1 ^ d2] = a3;
  }
  __syncthreads();
}

// nb sequences of length 2^l, sequence s at buf + s * stride (element a at sw2(a)).  Every thread
// of the block calls it, after a barrier; it returns after one.
template <typename T, bool INV>
__device__ __forceinline__ void fft2d(cplx<T>* buf, int l, int nb, int stride,
                                      const cplx<T>* tab) {
  const int q = l >> 1, odd = l & 1, lp = l - 1;
  auto pairs = [&]() {
#pragma unroll 1
    for (int g = threadIdx.x; g < (nb << lp); g += blockDim.x) {
      cplx<T>* s = buf + (g >> lp) * stride;
      const int a = sw2((g & ((1 << lp) - 1)) << 1);
      const cplx<T> x = s[a], y = s[a ^ 1];
      s[a] = x + y;
      s[a ^ 1] = x - y;
    }
    __syncthreads();
  };
  if (INV && odd) pairs();
#pragma unroll 1
  for (int j = 0; j < q; ++j)
    stage4<T, INV>(buf, l, nb, stride, tab, INV ? odd + 2 * j : l - 2 - 2 * j);
  if (!INV && odd) pairs();
}

// Derivative along the sequences: forward, times i kn m (m the signed mode, 0 for n/2), inverse;
// kn = 2 pi / (L n) takes the inverse's normalisation in.  A sequence a + i b of two real
// fields becomes a' + i b'.  The last forward stage, the product and the first inverse stage
// touch the same elements and stay in registers.
template <typename T>
__device__ __forceinline__ void deriv2d(cplx<T>* buf, int l, int nb, int stride,
                                        const cplx<T>* tab, T kn) {
  const int q = l >> 1, odd = l & 1, h = 1 << (l - 1), h2 = h >> 1;
#pragma unroll 1
  for (int j = 0; j < q - 1 + odd; ++j) stage4<T, false>(buf, l, nb, stride, tab, l - 2 - 2 * j);
  auto ik = [&](cplx<T> v, int m) { return mul_ik(v, from_int<T>(m) * kn); };
  if (odd) {
    const int lp = l - 1;
#pragma unroll 1
    for (int g = threadIdx.x; g < (nb << lp); g += blockDim.x) {
      cplx<T>* s = buf + (g >> lp) * stride;
      const int p = (g & ((1 << lp) - 1)) << 1, a = sw2(p), m = mode_at(p, l);
      const cplx<T> x = s[a], y = s[a ^ 1];
      const cplx<T> X = ik(x + y, m), Y = ik(x - y, m ? m - h : 0);
      s[a] = X + Y;
      s[a ^ 1] = X - Y;
    }
  } else {
    const int lb = l - 2, d1 = sw2(1), d2 = sw2(2);
#pragma unroll 1
    for (int g = threadIdx.x; g < (nb << lb); g += blockDim.x) {
      cplx<T>* s = buf + (g >> lb) * stride;
      const int p = (g & ((1 << lb) - 1)) << 2, a = sw2(p), m = mode_at(p, l);
      cplx<T> a0 = s[a], a1 = s[a ^ d1], a2 = s[a ^ d2], a3 = s[a ^ d1 ^ d2];
      dft4<T, false>(a0, a1, a2, a3);
      a0 = ik(a0, m);
      a1 = ik(a1, m + h2);
      a2 = ik(a2, m ? m - h : 0);
      a3 = ik(a3, m - h2);
      dft4<T, true>(a0, a1, a2, a3);
      s[a] = a0;
      s[a ^ d1] = a1;
      s[a ^ d2] = a2;
      s[a ^ d1 ^ d2] = a3;
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int j = 1 - odd; j < q; ++j) stage4<T, true>(buf, l, nb, stride, tab, odd + 2 * j);
}

// C2R of one packed pair: z <- A + i B at the modes' positions from two half rows.
template <typename T>
__device__ __forceinline__ void load_c2r_pair(cplx<T>* z, const cplx<T>* A, const cplx<T>* B,
                                              int l) {
  const int n = 1 << l, h = n >> 1;
  for (int m = threadIdx.x; m <= h; m += blockDim.x) {
    const cplx<T> a = A[m], b = B[m];
    z[sw2(pos_of(m, l))] = mk(a.x - b.y, a.y + b.x);
    if (m > 0 && m < h) z[sw2(pos_of(n - m, l))] = mk(a.x + b.y, b.x - a.y);
  }
}

// R2C split of a packed row Y = FFT(a + i b) (modes at their positions): A[m] = (Y_m + conj
// Y_{n-m})/2, B[m] = (Y_m - conj Y_{n-m})/(2i), m = 0..n/2.
template <typename T>
__device__ __forceinline__ void split_r2c_pair(const cplx<T>* Y, cplx<T>* A, cplx<T>* B, int l) {
  const int n = 1 << l, h = n >> 1;
  for (int m = threadIdx.x; m <= h; m += blockDim.x) {
    const cplx<T> y = Y[sw2(pos_of(m, l))], yc = conj(Y[sw2(pos_of((n - m) & (n - 1), l))]);
    const cplx<T> s = y + yc, d = mul_mi(y - yc);
    A[m] = mk(half(s.x), half(s.y));
    B[m] = mk(half(d.x), half(d.y));
  }
}

}  // namespace d2
}  // namespace sgn
