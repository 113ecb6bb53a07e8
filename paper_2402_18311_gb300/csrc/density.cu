// Electrostatic density: exact overlap-area bin map in 64-bit fixed point and
// its conversion to bin density and overflow.
//
// The density D of Eq. 1/2 is the ePlace electrostatic density the paper
// cites.  Reading: coordinates quantised to multiples of 2^-F (x * 2^F is
// exact in FP32, rounded to the nearest integer with ties to even), movable
// map M_b = sum_i overlap(cell_i, bin_b) as int64 in units of 2^-2F,
// overflow tau = sum_b max(0, M_b - t (A_b - F_b)) / A_mov and bin density
// rho_b = (M_b + t F_b) / A_b.  Integer addition is associative, so the map
// is bit-exact and independent of the order in which cells are added.  The
// overflow sum is exact too: with t = m 2^-s (m < 2^24), every bin's excess
// times 2^s is an integer below 2^100, summed in 128-bit integers.
#include "common.cuh"
#include "density_finish.cuh"
#include "internal.cuh"

namespace hp {

constexpr int kHash = 2048;  // shared-memory aggregation table entries

// Adds one (bin, area) contribution to the block's shared-memory table, or to
// the global map when its slot is taken (bounded linear probing).  lim: the
// map's length (checked in the bounds-checking build only).  A 64-bit addition
// in shared memory is a compare-and-swap loop, which lanes on the same bin
// repeat for one another; 32-bit additions are one instruction.  So an entry
// holds two 32-bit sums, of the areas' low `limb` bits and of the rest, with
// limb chosen at create such that a block's cells cannot overflow either
// (d.limb; 0 where there is no such split: one 64-bit sum).  Density stage of
// the 2.1M-cell design, the table way: 407 -> 107 us at the dense start; the
// merged way there, where warps of many bins come here too: 93 -> 83 us.
__device__ __forceinline__ void hash_add(int *keys, unsigned long long *vals,
                                         unsigned long long *M, int b,
                                         unsigned long long a, int limb, int *err, int lim) {
  if (!HP_IN(err, b, lim, BS_MAP_BIN)) return;
  unsigned int hsh = ((unsigned int)b * 2654435761u) >> (32 - 11);
#pragma unroll 1
  for (int probe = 0; probe < 2; ++probe) {
    int k = keys[hsh];  // plain read first: no atomic when the bin is already there
    if (k == -1) k = atomicCAS(&keys[hsh], -1, b);
    if (k == -1 || k == b) {
      if (limb) {
        unsigned int *v = reinterpret_cast<unsigned int *>(vals + hsh);
        atomicAdd(v, (unsigned int)a & ((1u << limb) - 1u));
        atomicAdd(v + 1, (unsigned int)(a >> limb));
      } else {
        atomicAdd(&vals[hsh], a);
      }
      return;
    }
    hsh = (hsh + 1) & (kHash - 1);
  }
  atomicAdd(&M[b], a);
}

// Exact sum of 64-bit values over the lanes in `mask` (all of which call
// this with the same mask): three 21-bit limbs are summed with the 32-bit
// warp reduction, which cannot overflow for 32 lanes.  The scatter calls it
// with the full mask only.
__device__ __forceinline__ unsigned long long group_sum_u64(unsigned int mask,
                                                            unsigned long long a) {
  const unsigned int l0 = (unsigned int)(a & 0x1FFFFF);
  const unsigned int l1 = (unsigned int)((a >> 21) & 0x1FFFFF);
  const unsigned int l2 = (unsigned int)(a >> 42);
  const unsigned long long s0 = __reduce_add_sync(mask, l0);
  const unsigned long long s1 = __reduce_add_sync(mask, l1);
  const unsigned long long s2 = __reduce_add_sync(mask, l2);
  return s0 + (s1 << 21) + (s2 << 42);
}

// Exact warp sum of values below 2^42: two 21-bit limbs (the second below
// 2^21, so each limb's sum over 32 lanes stays below 2^26).
__device__ __forceinline__ unsigned long long warp_sum_u42(unsigned long long a) {
  const unsigned long long s0 = __reduce_add_sync(0xffffffffu, (unsigned int)(a & 0x1FFFFF));
  const unsigned long long s1 = __reduce_add_sync(0xffffffffu, (unsigned int)(a >> 21));
  return s0 + (s1 << 21);
}

// The scatter's three ways (ScatterMode) are chosen per copy from the
// effective number of occupied bins of the previous density pass, n_eff =
// (sum M)^2 / sum M^2, against the handle's thresholds d.scat_t1 < d.scat_t2
// (set at create, by the autotuner when it runs).

// In the merged path, a warp slot whose lanes form more shared-bin groups
// than this adds every term to the block table instead.  Density stage of the
// 2.1M-cell design at iterations 10 / 170 with at most four groups merged:
// 0.113 / 0.165 ms, with one: 0.086 / 0.132; every term to the table:
// 0.111 / 0.107.
constexpr int kMaxMergeGroups = 1;

// A copy without a density pass behind it (a reset: n_eff = 0) has no such
// measure.  Its blocks then look at their first 256 cells: how many of them
// share the bin of their lower-left corner with a lower lane of their warp.
// With N equally full bins that is 3968 / N on average, so 3 or fewer stand
// for a spread copy, up to 86 (N = 32) for a concentrated one.  The
// reset pass of a spread 2.1M-cell copy: 141 -> 112 us; of the 20k-cell design
// with stretching (whose map merges 3 x 3 slots the same way): 105 -> 60.
constexpr int kSampleDirect = 3, kSampleTable = 86;

// Cells with more bins than this are left to the whole warp, a bin per lane.
constexpr int kWarpBins = 32;

// What the scatter adds for a cell: its rectangle, and with STRETCH (density
// stretching, ePlace's local smoothing: the map that drives the field when it
// is on) the stretched rectangle (create-time offsets and sizes in d.st) and
// each term scaled to floor(ov R / 2^31), R = d.sR[i] <= 2^31: ov = q 2^31 + r
// gives q R + floor(r R / 2^31), exact in 64 bits.
template <bool STRETCH>
struct ScatterCell {
  QRect32 r;
  unsigned int R;
  __device__ __forceinline__ void load(const Dev &d, const float2 *xy, int i) {
    const float2 v = xy[i];
    if constexpr (STRETCH) {
      const int4 st = d.st[i];  // {x shift, y shift, stretched W, stretched H}
      R = d.sR[i];
      r = qrect32(v.x, v.y, st.z, st.w, d.scale, d.XL + st.x, d.YL + st.y, d.BW32, d.BH32, d.nx,
                  d.ny, d.ibw_q, d.ibh_q);
    } else {
      r = qrect32(v.x, v.y, d.Wq[i], d.Hq[i], d.scale, d.XL, d.YL, d.BW32, d.BH32, d.nx, d.ny,
                  d.ibw_q, d.ibh_q);
    }
  }
  __device__ __forceinline__ void none() {
    r.x0 = r.x1 = r.y0 = r.y1 = 0;
    r.ix0 = r.iy0 = 0;
    r.ix1 = r.iy1 = -1;
    R = 0u;
  }
  __device__ __forceinline__ int bins() const {
    return r.ix0 <= r.ix1 && r.iy0 <= r.iy1 ? (r.ix1 - r.ix0 + 1) * (r.iy1 - r.iy0 + 1) : 0;
  }
  __device__ __forceinline__ unsigned long long term(const Dev &d, int ix, int iy) const {
    const long long ov =
        (long long)overlap32(r.x0, r.x1, ix, d.BW32) * overlap32(r.y0, r.y1, iy, d.BH32);
    if constexpr (STRETCH) {
      const unsigned long long o = (unsigned long long)ov;
      return (o >> 31) * R + (((o & 0x7fffffffull) * R) >> 31);
    } else {
      return (unsigned long long)ov;
    }
  }
};

// The cells of a warp that cover more than kWarpBins bins (movable macros), one
// after another by the whole warp: every lane takes every 32nd bin, straight
// to the map (a cell's bins are distinct, so nothing contends).  Left to its
// one lane, a macro of 17 x 17 bins held a pass of the 210k-cell mixed-size
// design for 250 us instead of BIGMEASURE.
template <bool STRETCH>
__device__ __forceinline__ void scatter_big(const Dev &d, const ScatterCell<STRETCH> &cell, int mo,
                                            unsigned long long *M, int lim) {
  unsigned int big = __ballot_sync(0xffffffffu, cell.bins() > kWarpBins);
  while (big) {
    const int l = __ffs(big) - 1;
    big &= big - 1;
    ScatterCell<STRETCH> c;
    c.r.x0 = __shfl_sync(0xffffffffu, cell.r.x0, l);
    c.r.x1 = __shfl_sync(0xffffffffu, cell.r.x1, l);
    c.r.y0 = __shfl_sync(0xffffffffu, cell.r.y0, l);
    c.r.y1 = __shfl_sync(0xffffffffu, cell.r.y1, l);
    c.r.ix0 = __shfl_sync(0xffffffffu, cell.r.ix0, l);
    c.r.ix1 = __shfl_sync(0xffffffffu, cell.r.ix1, l);
    c.r.iy0 = __shfl_sync(0xffffffffu, cell.r.iy0, l);
    c.r.iy1 = __shfl_sync(0xffffffffu, cell.r.iy1, l);
    c.R = __shfl_sync(0xffffffffu, cell.R, l);
    const int m = __shfl_sync(0xffffffffu, mo, l);
    const int h = c.r.iy1 - c.r.iy0 + 1, n = c.bins();
    for (int k = threadIdx.x & 31; k < n; k += 32) {
      const int ix = c.r.ix0 + k / h, iy = c.r.iy0 + k % h;
      const unsigned long long t = c.term(d, ix, iy);
      const int b = m + ix * d.ny + iy;
      if (t && HP_IN(d.err, b, lim, BS_MAP_BIN)) atomicAdd(&M[b], t);
    }
  }
}

// Cells are processed grid-stride, a warp at a time, in one of three ways,
// chosen per copy from how concentrated the previous density pass was:
//  * SCAT_MERGED, very dense (the centred start of a placement, where
//    millions of cells share a few bins): each cell touches at most 2 x 2
//    bins when it is no larger than a bin (3 x 3 stretched); the warp visits
//    those slots in lock-step, lanes that hit the same bin are merged with a
//    match/reduce (exact integer sums), and one lane per distinct bin adds the
//    total to a shared-memory hash table that is flushed with one 64-bit
//    atomic per distinct bin;
//  * SCAT_TABLE, concentrated (the middle of a placement, tens to a few
//    thousand effective bins): every lane adds each term to the block's
//    shared-memory table without the match, which costs more than the
//    shared-memory conflicts it would remove once the lanes of a warp rarely
//    share a bin;
//  * SCAT_DIRECT, spread: each lane adds its overlaps straight to the map.
// Larger cells add their remaining bins through the table in the first two
// ways, and from kWarpBins bins on go to the whole warp in all three.  Every
// way adds the same integers, so the map is the same.
// BIG: the design has cells of more bins.
template <bool STRETCH, bool BIG>
__global__ void __launch_bounds__(kThreads, 6) k_scatter(Dev d, int copy0, int eval) {
  __shared__ int keys[kHash];
  __shared__ unsigned long long vals[kHash];
  constexpr int SIDE = STRETCH ? 3 : 2;  // merged slots per axis
  pdl_wait();
  const int c = copy0 + blockIdx.y;
  if (!eval && d.cs[c].stopped) return;
  const float2 *xy = d.xy + (size_t)c * d.n_cells;
  // with fillers their map follows the movable one (bin b at G + b); the
  // stretched map holds both
  unsigned long long *M = STRETCH ? d.Ms + (size_t)c * d.G : d.M + (size_t)c * d.Gm;
  const int lim = STRETCH ? d.G : d.Gm;
  const int stride = gridDim.x * blockDim.x, lane = threadIdx.x & 31;
  const double n_eff = d.cs[c].n_eff;
  int mode = d.scat_force >= 0 ? d.scat_force
                               : (n_eff < d.scat_t1 ? SCAT_MERGED
                                                    : (n_eff < d.scat_t2 ? SCAT_TABLE : SCAT_DIRECT));
  if (d.scat_force < 0 && n_eff == 0.0) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int b = -1 - lane;  // distinct where there is no cell
    if (i < d.n_mov) {
      ScatterCell<STRETCH> cell;
      cell.load(d, xy, i);
      if (cell.bins()) b = cell.r.ix0 * d.ny + cell.r.iy0;
    }
    const int shared = __syncthreads_count(lane != __ffs(__match_any_sync(0xffffffffu, b)) - 1);
    mode = shared <= kSampleDirect ? SCAT_DIRECT : (shared <= kSampleTable ? SCAT_TABLE : SCAT_MERGED);
  }
  if (mode == SCAT_DIRECT) {
    // (warp-uniform trip count here and below)
    for (int i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < d.n_mov; i0 += stride) {
      const int i = i0 + lane;
      const int mo = (STRETCH || i < d.n_real) ? 0 : d.G;
      ScatterCell<STRETCH> cell;
      if (i < d.n_mov) cell.load(d, xy, i);
      else cell.none();
      if (!BIG || cell.bins() <= kWarpBins) {
        for (int ix = cell.r.ix0; ix <= cell.r.ix1; ++ix) {
          for (int iy = cell.r.iy0; iy <= cell.r.iy1; ++iy) {
            const unsigned long long t = cell.term(d, ix, iy);
            const int b = mo + ix * d.ny + iy;
            if (t && HP_IN(d.err, b, lim, BS_MAP_BIN)) atomicAdd(&M[b], t);
          }
        }
      }
      if constexpr (BIG) scatter_big(d, cell, mo, M, lim);
    }
    return;
  }
  for (int i = threadIdx.x; i < kHash; i += blockDim.x) {
    keys[i] = -1;
    vals[i] = 0ull;
  }
  __syncthreads();
  // one cell's overlap with one bin is at most the bin area
  const bool two_limbs = (double)d.BW * (double)d.BH < 4398046511104.0;  // 2^42
  for (int i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < d.n_mov; i0 += stride) {
    const int i = i0 + lane;
    const int mo = (STRETCH || i < d.n_real) ? 0 : d.G;
    ScatterCell<STRETCH> cell;
    if (i < d.n_mov) cell.load(d, xy, i);
    else cell.none();
    const bool lone = !BIG || cell.bins() <= kWarpBins;  // added by its own lane
    int done = 0;  // slots per axis that the merge has added
    if (mode == SCAT_MERGED) {
      done = SIDE;
#pragma unroll STRETCH ? 1 : 4
      for (int sl = 0; sl < SIDE * SIDE; ++sl) {
        const int ix = cell.r.ix0 + sl % SIDE, iy = cell.r.iy0 + sl / SIDE;
        int b = -1;
        unsigned long long a = 0ull;
        if (lone && ix <= cell.r.ix1 && iy <= cell.r.iy1) {
          a = cell.term(d, ix, iy);
          if (a != 0ull) b = mo + ix * d.ny + iy;
        }
        // one full-warp reduction per bin shared by several lanes (a per-group
        // mask would serialise the groups inside every reduction); each
        // group's lowest lane keeps the total, then all of them add at once:
        // alone on its bin straight to the map, shared through the block table
        const unsigned int mask = __match_any_sync(0xffffffffu, b);
        const bool lead = b >= 0 && lane == __ffs(mask) - 1;
        const bool shared = __popc(mask) > 1;
        unsigned int groups = __ballot_sync(0xffffffffu, lead && shared);
        if (__popc(groups) > kMaxMergeGroups) {
          // many small groups: one reduction per group would cost more than
          // the few same-address conflicts of adding every term to the table
          if (b >= 0) hash_add(keys, vals, M, b, a, d.limb, d.err, lim);
          continue;
        }
        unsigned long long tot = a;
        while (groups) {
          const int l = __ffs(groups) - 1;
          groups &= groups - 1;
          const int key = __shfl_sync(0xffffffffu, b, l);
          const unsigned long long mine = b == key ? a : 0ull;
          const unsigned long long t =
              two_limbs ? warp_sum_u42(mine) : group_sum_u64(0xffffffffu, mine);
          if (lane == l) tot = t;
        }
        if (lead) {
          if (shared)
            hash_add(keys, vals, M, b, tot, d.limb, d.err, lim);
          else if (HP_IN(d.err, b, lim, BS_MAP_BIN))
            atomicAdd(&M[b], tot);
        }
      }
    }
    // all bins through the table, or those beyond the merged slots
    if (lone && (cell.r.ix1 - cell.r.ix0 >= done || cell.r.iy1 - cell.r.iy0 >= done)) {
      for (int ix = cell.r.ix0; ix <= cell.r.ix1; ++ix) {
        for (int iy = cell.r.iy0; iy <= cell.r.iy1; ++iy) {
          if (ix - cell.r.ix0 < done && iy - cell.r.iy0 < done) continue;  // done above
          const unsigned long long t = cell.term(d, ix, iy);
          if (t) hash_add(keys, vals, M, mo + ix * d.ny + iy, t, d.limb, d.err, lim);
        }
      }
    }
    if constexpr (BIG) {
      __syncwarp();
      scatter_big(d, cell, mo, M, lim);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kHash; i += blockDim.x) {
    int k = keys[i];
    if (k >= 0) {
      const unsigned long long v = vals[i];
      atomicAdd(&M[k], d.limb ? (v & 0xffffffffull) + ((v >> 32) << d.limb) : v);
    }
  }
}

// Same map for an arbitrary cell range (the fixed cells, once at create).
__global__ void __launch_bounds__(kThreads)
    k_scatter_range(Dev d, const float2 *xy, int n0, int n1, unsigned long long *out) {
  for (int i = n0 + blockIdx.x * blockDim.x + threadIdx.x; i < n1; i += gridDim.x * blockDim.x) {
    const float2 v = xy[i];
    const QRect32 r = qrect32(v.x, v.y, d.Wq[i], d.Hq[i], d.scale, d.XL, d.YL, d.BW32, d.BH32,
                              d.nx, d.ny, d.ibw_q, d.ibh_q);
    for (int ix = r.ix0; ix <= r.ix1; ++ix) {
      const int ox = overlap32(r.x0, r.x1, ix, d.BW32);
      if (ox == 0) continue;
      for (int iy = r.iy0; iy <= r.iy1; ++iy) {
        const int oy = overlap32(r.y0, r.y1, iy, d.BH32);
        if (oy == 0) continue;
        const int b = ix * d.ny + iy;
        if (HP_IN(d.err, b, d.G, BS_MAP_BIN))
          atomicAdd(&out[b], (unsigned long long)((long long)ox * oy));
      }
    }
  }
}

__device__ __forceinline__ void store_bf16_pair(__nv_bfloat16 *hp, __nv_bfloat16 *lp, size_t b2,
                                                float v0, float v1) {
  const __nv_bfloat162 hi = __floats2bfloat162_rn(v0, v1);
  const __nv_bfloat162 lo = __floats2bfloat162_rn(v0 - __low2float(hi), v1 - __high2float(hi));
  reinterpret_cast<__nv_bfloat162 *>(hp)[b2] = hi;
  reinterpret_cast<__nv_bfloat162 *>(lp)[b2] = lo;
}

// Per bin: exact overflow excess and rho in FP32 (density_finish.cuh has both
// and what the last block does with the overflow).  STRETCH: rho comes from
// the stretched map (density stretching on); the overflow always from M.  Two
// bins per thread and step (G is even): 16-byte loads and paired bf16
// conversions and stores.  FOLD (the even/odd split of the tensor-core
// solve): four bins per step, (x, y), (x, y+1) and their mirrors
// (x, ny-1-y), (x, ny-2-y), and rho leaves as the sums rho_y + rho_{ny-1-y}
// at y and the differences at ny/2 + y (y < ny/2).  Handles with a fused
// solve form rho there and come here for the overflow alone;
// clear: they leave the map zero.
template <bool STRETCH, bool FOLD>
__global__ void __launch_bounds__(kThreads) k_density_finish(Dev d, int copy0, int mode, int clear) {
  __shared__ FinishShared fs;
  pdl_wait();
  const int c = copy0 + blockIdx.y;
  if (mode == FIN_ITER && d.cs[c].stopped) return;
  const FinishArgs fa = finish_args(d, c);
  BinSums sums;
  if constexpr (FOLD) {
    __nv_bfloat16 *rh = d.rho_h + (size_t)c * d.G, *rl = d.rho_l + (size_t)c * d.G;
    const int q4 = d.ny >> 2, nq = d.G >> 2, hy = d.ny >> 1;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nq; t += gridDim.x * blockDim.x) {
      const int x = t / q4, y = 2 * (t - x * q4);  // y even, below ny/2
      const int row = x * d.ny;
      const float2 a = finish_pair<STRETCH>(d, fa, (row + y) >> 1, sums);
      // bins ny-2-y and ny-1-y
      const float2 b = finish_pair<STRETCH>(d, fa, (row + d.ny - 2 - y) >> 1, sums);
      store_bf16_pair(rh, rl, (size_t)(row + y) >> 1, __fadd_rn(a.x, b.y), __fadd_rn(a.y, b.x));
      store_bf16_pair(rh, rl, (size_t)(row + hy + y) >> 1, __fsub_rn(a.x, b.y),
                      __fsub_rn(a.y, b.x));
    }
  } else {
    const int G2 = d.G >> 1;
    for (int b2 = blockIdx.x * blockDim.x + threadIdx.x; b2 < G2; b2 += gridDim.x * blockDim.x) {
      const float2 rv = finish_pair<STRETCH>(d, fa, b2, sums);
      if (d.solve != SOLVE_GEMM) {
        if (clear) clear_pair(d, c, b2);
        continue;
      }
      if (d.tc)
        store_bf16_pair(d.rho_h + (size_t)c * d.G, d.rho_l + (size_t)c * d.G, b2, rv.x, rv.y);
      else
        reinterpret_cast<float2 *>(d.rho + (size_t)c * d.G)[b2] = rv;
    }
  }
  finish_reduce<kThreads>(d, c, mode, sums, &fs);
}

// Floor of the scatter's memory work at the current positions: per movable
// cell the same loads (position and quantised size) and one 64-bit reduction
// into each bin the cell covers (the bins from an FP32 estimate of its
// corners), none of the exact rectangle arithmetic.  It adds into the map,
// which the caller clears.
__global__ void __launch_bounds__(kThreads) k_scatter_floor(Dev d, int copy0) {
  const int c = copy0 + blockIdx.y;
  const float2 *xy = d.xy + (size_t)c * d.n_cells;
  unsigned long long *M = d.M + (size_t)c * d.Gm;
  const float is = 1.f / d.scale;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d.n_mov; i += gridDim.x * blockDim.x) {
    const int mo = i < d.n_real ? 0 : d.G;
    const float2 v = xy[i];
    const float w = (float)d.Wq[i] * is, h = (float)d.Hq[i] * is;
    const int ix0 = min(max((int)floorf((v.x - d.fxl) * d.fibw), 0), d.nx - 1);
    const int ix1 = min(max((int)floorf((v.x + w - d.fxl) * d.fibw), 0), d.nx - 1);
    const int iy0 = min(max((int)floorf((v.y - d.fyl) * d.fibh), 0), d.ny - 1);
    const int iy1 = min(max((int)floorf((v.y + h - d.fyl) * d.fibh), 0), d.ny - 1);
    for (int ix = ix0; ix <= ix1; ++ix)
      for (int iy = iy0; iy <= iy1; ++iy) {
        const int b = mo + ix * d.ny + iy;
        if (HP_IN(d.err, b, d.Gm, BS_MAP_BIN)) atomicAdd(&M[b], 1ull);
      }
  }
}

void launch_scatter_floor(const Dev &d, int copy0, int ncopy, cudaStream_t st) {
  k_scatter_floor<<<dim3(d.cell_blocks, ncopy), kThreads, 0, st>>>(d, copy0);
}

template <bool STRETCH>
static void scatter(const Dev &d, int copy0, int ncopy, int eval, cudaStream_t st) {
  const dim3 grid(d.cell_blocks, ncopy);
  if (d.has_big)
    k_scatter<STRETCH, true><<<grid, kThreads, 0, st>>>(d, copy0, eval);
  else
    k_scatter<STRETCH, false><<<grid, kThreads, 0, st>>>(d, copy0, eval);
}

void launch_scatter_main(const Dev &d, int copy0, int ncopy, int eval, cudaStream_t st) {
  scatter<false>(d, copy0, ncopy, eval, st);
}

void launch_scatter(const Dev &d, int copy0, int ncopy, int eval, cudaStream_t st) {
  scatter<false>(d, copy0, ncopy, eval, st);
  if (d.Ms) {
    cudaMemsetAsync(d.Ms + (size_t)copy0 * d.G, 0, sizeof(unsigned long long) * d.G * ncopy, st);
    scatter<true>(d, copy0, ncopy, eval, st);
  }
}

void launch_scatter_fixed(const Dev &d, const float2 *xy, int n0, int n1,
                          unsigned long long *out, cudaStream_t st) {
  if (n1 <= n0) return;
  int blocks = (n1 - n0 + kThreads - 1) / kThreads;
  if (blocks > 4096) blocks = 4096;
  k_scatter_range<<<blocks, kThreads, 0, st>>>(d, xy, n0, n1, out);
}

void launch_density_finish(const Dev &d, int copy0, int ncopy, int mode, int clear, cudaStream_t st) {
  dim3 grid(d.bin_blocks, ncopy);
  const bool fold = d.bfly && d.solve == SOLVE_GEMM;
  auto *k = d.Ms ? (fold ? k_density_finish<true, true> : k_density_finish<true, false>)
                 : (fold ? k_density_finish<false, true> : k_density_finish<false, false>);
  launch_pdl(k, grid, dim3(kThreads), 0, st, d, copy0, mode, clear);
}

}  // namespace hp
