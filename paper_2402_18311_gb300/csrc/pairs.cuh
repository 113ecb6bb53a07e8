// Exact pin coordinates as pairs of FP32 numbers (wirelength.cu has the
// reasons): the sum of a cell's position and a pin's offset as s, the sum rounded,
// and e, what the rounding dropped.  Both summands are multiplied by d.pin_scale
// first: 1, or 1/2 on a design whose largest sums might overflow FP32 (there a
// subnormal number loses its last bit).
#pragma once

#include <cfloat>

#include "common.cuh"

namespace hp {

struct Pair {
  float s, e;
};
__device__ __forceinline__ Pair pin_coord(float v, float o, float scale) {
  Pair p;
  two_sum(scale * v, scale * o, p.s, p.e);
  return p;
}
__device__ __forceinline__ void pair_max(Pair &m, Pair p) {
  const bool up = p.s > m.s || (p.s == m.s && p.e > m.e);
  m.s = up ? p.s : m.s;
  m.e = up ? p.e : m.e;
}
__device__ __forceinline__ void pair_min(Pair &m, Pair p) {
  const bool dn = p.s < m.s || (p.s == m.s && p.e < m.e);
  m.s = dn ? p.s : m.s;
  m.e = dn ? p.e : m.e;
}
struct PairBox {
  Pair mx, nx, my, ny;  // maximum and minimum per axis
};
__device__ __forceinline__ PairBox empty_box() {
  const Pair lo{-FLT_MAX, 0.f}, hi{FLT_MAX, 0.f};
  return PairBox{lo, hi, lo, hi};
}
__device__ __forceinline__ void box_add(PairBox &b, float2 v, float2 o, float scale) {
  const Pair x = pin_coord(v.x, o.x, scale), y = pin_coord(v.y, o.y, scale);
  pair_max(b.mx, x); pair_min(b.nx, x);
  pair_max(b.my, y); pair_min(b.ny, y);
}
__device__ __forceinline__ Pair pair_xor(Pair p, int o) {
  return Pair{__shfl_xor_sync(0xffffffffu, p.s, o), __shfl_xor_sync(0xffffffffu, p.e, o)};
}
template <int G>
__device__ __forceinline__ void box_reduce(PairBox &b) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) {
    pair_max(b.mx, pair_xor(b.mx, o)); pair_min(b.nx, pair_xor(b.nx, o));
    pair_max(b.my, pair_xor(b.my, o)); pair_min(b.ny, pair_xor(b.ny, o));
  }
}
// An FP32 number as FP64 by moving its bits (normal numbers and zero; the
// conversion instruction is on the FP64 pipe too).
__device__ __forceinline__ double widen(float f) {
  const unsigned int u = __float_as_uint(f), x = u & 0x7f800000u;
  if (x == 0u || x == 0x7f800000u) return (u & 0x7fffffffu) ? (double)f : 0.0;
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)),
                          (int)(u << 29));
}
// What the rounding of a pair dropped: nothing of an infinite sum (whose e is not
// a number).
__device__ __forceinline__ double pair_rest(Pair p) { return widen(p.e == p.e ? p.e : 0.f); }
// A pair's number, not scaled any more (unscale: 1 / d.pin_scale): the exact sum
// rounded once to FP64.
__device__ __forceinline__ double pair_value(Pair p, double unscale) {
  return unscale * (widen(p.s) + pair_rest(p));
}

}  // namespace hp
