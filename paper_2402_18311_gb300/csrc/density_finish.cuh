// The end of a density pass, shared by the kernels that read the map: per bin
// the exact overflow excess and the bin density, and the reduction of the
// overflow (density.cu has the definitions).
#pragma once

#include "common.cuh"
#include "internal.cuh"

namespace hp {

// A nonnegative 64-bit integer as FP32 from its two 32-bit halves (two fast
// conversions and one FMA instead of the multi-instruction 64-bit one; the
// result may differ from the correctly rounded one in the last bit).
__device__ __forceinline__ float u64_to_float(unsigned long long v) {
  return fmaf((float)(unsigned int)(v >> 32), 4294967296.0f, (float)(unsigned int)v);
}

// A thread's sums over its bins.  Bins without fixed cells: their excess times
// 2^s is m 2^s - t_mant A, positive exactly when m > floor(t_mant A / 2^s); the
// sum over those bins is 2^s (sum of m) - count * t_mant A, formed once after
// the bins (the sum of m stays below the movable area, below 2^62).
struct BinSums {
  u128 acc = 0;                      // excess 2^s of bins with fixed cells
  unsigned long long m_over = 0ull;  // the others above the target: their sum
  unsigned int n_over = 0u;          // and their number
  float q2 = 0.f;                    // sum of (M / A_bin)^2
};

// What a copy's bins are read with.
struct FinishArgs {
  const ulonglong2 *M2, *Mf2, *Ms2;  // map, fillers' map (or null), stretched map (or null)
  const longlong2 *F2;
  u128 tA;  // t_mant * A_bin
  float inv_a, tf;
};
__device__ __forceinline__ FinishArgs finish_args(const Dev &d, int c) {
  FinishArgs a;
  a.M2 = reinterpret_cast<const ulonglong2 *>(d.M + (size_t)c * d.Gm);
  // with fillers their map (following M) joins rho and the concentration
  a.Mf2 = d.n_fill ? a.M2 + (d.G >> 1) : nullptr;
  a.Ms2 = d.Ms ? reinterpret_cast<const ulonglong2 *>(d.Ms + (size_t)c * d.G) : nullptr;
  a.F2 = reinterpret_cast<const longlong2 *>(d.Fmap);
  a.tA = ((u128)d.tA_hi << 64) | d.tA_lo;
  a.inv_a = (float)(1.0 / d.abin_q);
  a.tf = (float)d.t;
  return a;
}

// Excess contribution of one bin: bins without fixed cells are counted into
// (m_over, n_over) and closed after the loop; the others are summed exactly
// in 128 bits.
__device__ __forceinline__ void bin_excess(const Dev &d, unsigned long long m, long long f, u128 tA,
                                           BinSums &s) {
  if (f == 0) {
    if (m > d.tA_floor) {
      s.m_over += m;
      ++s.n_over;
    }
  } else {
    // excess * 2^s = m 2^s + t_mant F - t_mant A: exact in signed 128 bits
    // (below 2^124; F > A where fixed cells overlap, F < 0 only in a map that a
    // caller of place_overflow_noalloc brings)
    const __int128 e = (__int128)((u128)m << d.t_shift) + (__int128)d.t_mant * (__int128)f - (__int128)tA;
    if (e > 0) s.acc += (u128)e;
  }
}

// One pair of bins (2 b2, 2 b2 + 1): their excess into the sums and rho.
template <bool STRETCH>
__device__ __forceinline__ float2 finish_pair(const Dev &d, const FinishArgs &a, int b2, BinSums &s) {
  const ulonglong2 m = a.M2[b2];
  const longlong2 f = a.F2[b2];
  float mq0 = u64_to_float(m.x) * a.inv_a, mq1 = u64_to_float(m.y) * a.inv_a;
  if (a.Mf2) {
    const ulonglong2 mf = a.Mf2[b2];
    mq0 = u64_to_float(m.x + mf.x) * a.inv_a;
    mq1 = u64_to_float(m.y + mf.y) * a.inv_a;
  }
  s.q2 = fmaf(mq0, mq0, s.q2);
  s.q2 = fmaf(mq1, mq1, s.q2);
  bin_excess(d, m.x, f.x, a.tA, s);
  bin_excess(d, m.y, f.y, a.tA, s);
  float mf0 = mq0, mf1 = mq1;
  if constexpr (STRETCH) {
    const ulonglong2 ms = a.Ms2[b2];
    mf0 = u64_to_float(ms.x) * a.inv_a;
    mf1 = u64_to_float(ms.y) * a.inv_a;
  }
  return make_float2(fmaf(a.tf, u64_to_float((unsigned long long)f.x) * a.inv_a, mf0),
                     fmaf(a.tf, u64_to_float((unsigned long long)f.y) * a.inv_a, mf1));
}

// The copy's overflow from its bins' excess v (times 2^s) and its concentration
// from q2, recorded by mode: the iteration's tau (with the stop test), an
// evaluation's result, or the reset value tau_{-1} that sets the first gamma.
// Called by a warp whose lane 0 has v and q2: its FP64 division, a microsecond
// here, is shared with lane 1's (n_eff).
__device__ __forceinline__ void finish_commit(const Dev &d, int c, int mode, u128 v, float q2) {
  CopyState *cs = d.cs + c;
  q2 = __shfl_sync(0xffffffffu, q2, 0);
  const bool first = threadIdx.x == 0;
  const double r = (first ? ldexp(u128_to_double(v), -d.t_shift) : d.area2_bins) / (first ? d.mov_area_q : (double)q2);
  if (threadIdx.x == 1 && mode != FIN_EVAL) cs->n_eff = q2 > 0.f ? r : 0.0;
  if (!first) return;
  if (mode == FIN_ITER) {
    cs->tau = r;
    if (r <= (double)d.prm.tau_stop) cs->converged = cs->stopped = 1;
  } else if (mode == FIN_RESET) {
    cs->tau = cs->tau_prev = r;
    cs->gamma = gamma_of(d, r);
    if (d.prm.max_iters <= 0) cs->stopped = 1;
  } else {
    d.scal[(size_t)c * S_COUNT + S_TAU] = r;
  }
}

// The map (and the fillers') zero again at bins 2 b2 and 2 b2 + 1.
__device__ __forceinline__ void clear_pair(const Dev &d, int c, int b2) {
  ulonglong2 *M = reinterpret_cast<ulonglong2 *>(d.M + (size_t)c * d.Gm);
  M[b2] = make_ulonglong2(0ull, 0ull);
  if (d.n_fill) M[(d.G >> 1) + b2] = make_ulonglong2(0ull, 0ull);
}

struct FinishShared {
  u128 sm[32];
  float smf[32];
  int flag;
};

// The block's sums to its partial slot.
template <int NT>
__device__ __forceinline__ void finish_partial(const Dev &d, int c, const BinSums &s, FinishShared *sh) {
  const u128 tA = ((u128)d.tA_hi << 64) | d.tA_lo;
  const u128 acc = s.acc + ((u128)s.m_over << d.t_shift) - (u128)s.n_over * tA;
  const float q2 = block_sum_f<NT>(s.q2, sh->smf);
  const u128 r = block_sum_u128<NT>(acc, sh->sm);
  if (threadIdx.x == 0) {
    unsigned long long *p = d.tau_part + ((size_t)c * d.nb_red + blockIdx.x) * 2;
    p[0] = (unsigned long long)r;
    p[1] = (unsigned long long)(r >> 64);
    d.conc_part[(size_t)c * d.nb_red + blockIdx.x] = q2;
  }
}

// The copy's overflow from n partials, by one warp (an earlier kernel's
// partials, or, behind a cluster barrier, this one's).
__device__ __forceinline__ void finish_total(const Dev &d, int c, int mode, int n) {
  u128 v = 0;
  float q2 = 0.f;
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += 32) {
    const unsigned long long *p = d.tau_part + ((size_t)c * d.nb_red + i) * 2;
    v += ((u128)__ldcg(p + 1) << 64) | __ldcg(p);
    q2 += __ldcg(d.conc_part + (size_t)c * d.nb_red + i);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v += shfl_xor_u128(v, o);
    q2 += __shfl_xor_sync(0xffffffffu, q2, o);
  }
  finish_commit(d, c, mode, v, q2);
}

// The block's sums to its partial slot; the last block of each copy reduces
// them and records the overflow.
template <int NT>
__device__ __forceinline__ void finish_reduce(const Dev &d, int c, int mode, const BinSums &s,
                                              FinishShared *sh) {
  finish_partial<NT>(d, c, s, sh);
  if (!arrive_last_t0(d.ctr + (size_t)c * C_COUNT + C_FINISH, &sh->flag)) return;
  u128 v = 0;
  float q2 = 0.f;
#pragma unroll 4
  for (int i = threadIdx.x; i < (int)gridDim.x; i += NT) {
    const unsigned long long *p = d.tau_part + ((size_t)c * d.nb_red + i) * 2;
    v += ((u128)__ldcg(p + 1) << 64) | __ldcg(p);
    q2 += __ldcg(d.conc_part + (size_t)c * d.nb_red + i);
  }
  v = block_sum_u128<NT>(v, sh->sm);
  q2 = block_sum_f<NT>(q2, sh->smf);
  if (threadIdx.x < 32) finish_commit(d, c, mode, v, q2);
  if (threadIdx.x == 0) d.ctr[(size_t)c * C_COUNT + C_FINISH] = 0u;
}

}  // namespace hp
