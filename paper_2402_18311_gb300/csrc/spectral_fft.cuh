// Power-of-two FFTs in registers and shared memory for the fast-transform
// Poisson solve (spectral_fft.cu).
#pragma once

#include <cuda_runtime.h>

namespace hp {
namespace fft {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// a times -i (forward) or +i (inverse)
template <bool INV>
__device__ __forceinline__ float2 cturn(float2 a) {
  return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

template <bool INV>
__device__ __forceinline__ void dft4(float2 &a0, float2 &a1, float2 &a2, float2 &a3) {
  const float2 b0 = cadd(a0, a2), b1 = csub(a0, a2), b2 = cadd(a1, a3), b3 = cturn<INV>(csub(a1, a3));
  a0 = cadd(b0, b2);
  a1 = cadd(b1, b3);
  a2 = csub(b0, b2);
  a3 = csub(b1, b3);
}

template <bool INV>
__device__ __forceinline__ void dft8(float2 (&a)[8]) {
  dft4<INV>(a[0], a[2], a[4], a[6]);
  dft4<INV>(a[1], a[3], a[5], a[7]);
  const float h = 0.70710678118654752f;  // exp(-+ i pi / 4) = h (1 -+ i)
  const float2 o1 = INV ? make_float2(h * (a[3].x - a[3].y), h * (a[3].x + a[3].y))
                        : make_float2(h * (a[3].x + a[3].y), h * (a[3].y - a[3].x));
  const float2 o2 = cturn<INV>(a[5]);
  const float2 o3 = INV ? make_float2(-h * (a[7].x + a[7].y), h * (a[7].x - a[7].y))
                        : make_float2(h * (a[7].y - a[7].x), -h * (a[7].x + a[7].y));
  const float2 e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6], o0 = a[1];
  a[0] = cadd(e0, o0); a[4] = csub(e0, o0);
  a[1] = cadd(e1, o1); a[5] = csub(e1, o1);
  a[2] = cadd(e2, o2); a[6] = csub(e2, o2);
  a[3] = cadd(e3, o3); a[7] = csub(e3, o3);
}

// Shared-memory position of element i: one float2 of padding after every
// eight keeps the strided writes between the stages free of bank conflicts.
__device__ __forceinline__ int pad(int i) { return i + (i >> 3); }
constexpr int padded(int n) { return n + n / 8; }

template <bool INV>
__device__ __forceinline__ float2 twiddle(const float2 *tw, int k) {
  const float2 w = __ldg(tw + k);
  return INV ? make_float2(w.x, -w.y) : w;
}

// The stages from block length NS on of an N-point FFT (N = 2^LOGN) by N / 8
// threads, self-sorting (Stockham): before every stage thread t holds the
// elements t + m N / 8 in v[m], and at the end the transform's.  tw[k] =
// exp(-2 pi i k / N).  s: padded(N) entries that nobody reads any more; every
// thread of the block calls it.
template <int LOGN, bool INV, int LOGNS>
__device__ __forceinline__ void stages(float2 (&v)[8], int t, float2 *s, const float2 *tw) {
  constexpr int N = 1 << LOGN, T = N / 8, REM = LOGN - LOGNS, NS = 1 << LOGNS;
  if constexpr (REM > 0) {
    constexpr int LR = (REM == 3 || REM >= 5) ? 3 : 2;  // radix 8, then 4
    constexpr int R = 1 << LR, NB = 8 / R;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int j = t + b * T, k = j & (NS - 1);
      if constexpr (NS > 1) {
        const int step = k << (REM - LR);  // k N / (NS R)
        // each power from the table: products of powers would add their own
        // rounding errors (field error 2.4e-7 with products, 1.9e-7 without, at 1024 x 1024)
#pragma unroll
        for (int r = 1; r < R; ++r) v[b + r * NB] = cmul(v[b + r * NB], twiddle<INV>(tw, r * step));
      }
      if constexpr (R == 8)
        dft8<INV>(v);
      else
        dft4<INV>(v[b], v[b + NB], v[b + 2 * NB], v[b + 3 * NB]);
    }
    if constexpr (REM > LR) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const int j = t + b * T, k = j & (NS - 1);
        const int o = ((j >> LOGNS) << (LOGNS + LR)) + k;
#pragma unroll
        for (int r = 0; r < R; ++r) s[pad(o + r * NS)] = v[b + r * NB];
      }
      __syncthreads();
#pragma unroll
      for (int m = 0; m < 8; ++m) v[m] = s[pad(t + m * T)];
      __syncthreads();
      stages<LOGN, INV, LOGNS + LR>(v, t, s, tw);
    }
  }
}

// Thread t's elements (t + m N / 8 in v[m]) after, and s free for writing.
template <int LOGN, bool INV>
__device__ __forceinline__ void transform(float2 (&v)[8], int t, float2 *s, const float2 *tw) {
  stages<LOGN, INV, 0>(v, t, s, tw);
}

// Position of sample i in the order that turns a length-N DCT-II into an FFT:
// the even samples upwards, then the odd ones downwards.
template <int N>
__device__ __forceinline__ int dct_order(int i) {
  return (i & 1) ? N - 1 - (i >> 1) : i >> 1;
}
// and the sample at position n
template <int N>
__device__ __forceinline__ int dct_sample(int n) {
  return n < N / 2 ? 2 * n : 2 * (N - 1 - n) + 1;
}

}  // namespace fft
}  // namespace hp
