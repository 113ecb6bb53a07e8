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
#include "scatter.cuh"

namespace hp {

// BIG: the design has cells of more than kWarpBins bins.
template <bool STRETCH, bool BIG>
__global__ void __launch_bounds__(kThreads, 6) k_scatter(Dev d, int copy0, int eval) {
  __shared__ int keys[kHash];
  __shared__ unsigned long long vals[kHash];
  pdl_wait();
  const int c = copy0 + blockIdx.y;
  if (!eval && d.cs[c].stopped) return;
  const float2 *xy = d.xy + (size_t)c * d.n_cells;
  // with fillers their map follows the movable one (bin b at G + b); the
  // stretched map holds both
  unsigned long long *M = STRETCH ? d.Ms + (size_t)c * d.G : d.M + (size_t)c * d.Gm;
  scatter_block<STRETCH, BIG>(
      d, d.n_mov, d.cs[c].n_eff, M, STRETCH ? d.G : d.Gm, keys, vals,
      [&](ScatterCell<STRETCH> &cell, int i) { cell.load(d, xy, i); },
      [&](int i) { return (STRETCH || i < d.n_real) ? 0 : d.G; });
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
