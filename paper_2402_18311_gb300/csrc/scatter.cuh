// The density scatter's device code, shared by the handles' kernels (density.cu)
// and the allocation-free overflow (noalloc.cu): exact overlap areas added to
// a 64-bit map.
#pragma once

#include "common.cuh"
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
// design for 250 us; the whole scatter and finish there now take 26.
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
// One block's part of a scatter of n cells into the map M of lim entries:
// load(cell, i) reads cell i (each once), offset(i) is added to its bins.  keys,
// vals: the block's table (kHash entries).  BIG: there may be cells of more
// than kWarpBins bins.
template <bool STRETCH, bool BIG, typename Load, typename Offset>
__device__ __forceinline__ void scatter_block(const Dev &d, int n, double n_eff, unsigned long long *M,
                                              int lim, int *keys, unsigned long long *vals, Load load,
                                              Offset offset) {
  constexpr int SIDE = STRETCH ? 3 : 2;  // merged slots per axis
  const int stride = gridDim.x * kThreads, lane = threadIdx.x & 31;
  int mode = d.scat_force >= 0 ? d.scat_force
                               : (n_eff < d.scat_t1 ? SCAT_MERGED
                                                    : (n_eff < d.scat_t2 ? SCAT_TABLE : SCAT_DIRECT));
  // (a warp's lanes stay together: i0 is its first cell)
  int i0 = blockIdx.x * kThreads + (threadIdx.x & ~31);
  ScatterCell<STRETCH> cell;
  auto fetch = [&]() {
    if (i0 + lane < n) load(cell, i0 + lane);
    else cell.none();
  };
  fetch();
  if (d.scat_force < 0 && n_eff == 0.0) {
    // (distinct where there is no cell)
    const int b = cell.bins() ? cell.r.ix0 * d.ny + cell.r.iy0 : -1 - lane;
    const int shared = __syncthreads_count(lane != __ffs(__match_any_sync(0xffffffffu, b)) - 1);
    mode = shared <= kSampleDirect ? SCAT_DIRECT : (shared <= kSampleTable ? SCAT_TABLE : SCAT_MERGED);
  }
  if (mode == SCAT_DIRECT) {
    while (i0 < n) {
      const int mo = offset(i0 + lane);
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
      i0 += stride;
      fetch();
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
  while (i0 < n) {
    const int mo = offset(i0 + lane);
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
    i0 += stride;
    fetch();
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

}  // namespace hp
