// Per-cell gradient assembly, preconditioning, the Nesterov/Lipschitz update
// and the per-copy scalar schedule (Eq. 2 minimised by Nesterov's method, as
// in the ePlace/DREAMPlace placers that the paper runs as the
// global-placement step of Algorithm 1).
//
// Iteration k at reference point v_k (this library's reading; the paper
// cites the method without restating it):
//   gamma_k = gamma_base w_bin 10^((20/9) tau_{k-1} - 11/9)
//   g_k = (gWL + lambda gD) / max(1, pins_i + lambda area_i)
//   alpha_k = alpha0 w_bin / rms(g_0) at k = 0, else |v_k - v_{k-1}| / |g_k - g_{k-1}|
//   u_{k+1} = clamp(v_k - alpha_k g_k)
//   a_{k+1} = (1 + sqrt(4 a_k^2 + 1)) / 2
//   v_{k+1} = clamp(u_{k+1} + (a_k - 1)/a_{k+1} (u_{k+1} - u_k))
//   lambda_0 = eta |gWL|_1 / |gD|_1;  lambda_{k+1} = lambda_k clamp(mu^(1 - dHPWL/dref))
// Per-cell work is FP32 (GB300's FP64 rate is tiny); each thread sums its
// few cells in FP32, each block sums its threads with a compensated FP32
// tree and publishes one FP64 partial; the last block of each copy reduces the partials in a fixed order
// and advances the copy's scalars, so every run of the same input gives the
// same bits and no separate scalar kernels are launched.
#include <math.h>

#include "common.cuh"
#include "internal.cuh"

namespace hp {

__device__ __forceinline__ double *part_ptr(const Dev &d, int c, int slot) {
  return d.part + ((size_t)c * S_COUNT + slot) * d.nb_red;
}

// Fixed-order sums of NS slots' partials by a whole block; valid in thread
// 0.  Four independent accumulators per slot keep 4 * NS loads in flight
// (a single running sum would wait a full L2 round trip per partial).
template <int NT, int NS>
__device__ void sum_slots(const Dev &d, int c, const int (&slots)[NS], int n, double (&out)[NS],
                          double *sm) {
  const double *p[NS];
  double v[NS][4];
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    p[s] = part_ptr(d, c, slots[s]);
    v[s][0] = v[s][1] = v[s][2] = v[s][3] = 0.0;
  }
  int i = threadIdx.x;
  for (; i + 3 * NT < n; i += 4 * NT) {
#pragma unroll
    for (int s = 0; s < NS; ++s) {
#pragma unroll
      for (int u = 0; u < 4; ++u) v[s][u] += p[s][i + u * NT];
    }
  }
  for (; i < n; i += NT) {
#pragma unroll
    for (int s = 0; s < NS; ++s) v[s][0] += p[s][i];
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) out[s] = block_sum<NT>((v[s][0] + v[s][1]) + (v[s][2] + v[s][3]), sm);
}

template <int NT>
__device__ double sum_slot(const Dev &d, int c, int slot, int n, double *sm) {
  const int slots[1] = {slot};
  double out[1];
  sum_slots<NT, 1>(d, c, slots, n, out, sm);
  return out[0];
}

// Sums of NS slots' partials (n[s] of them) by a whole block, all slots in
// one pass: their loads, their trees' FP64 steps and their barriers overlap.
// Fixed order; out[s] valid in every thread.  sm: NS * NT / 32 + NS entries.
template <int NT, int NS>
__device__ __forceinline__ void sum_slots_all(const Dev &d, int c, const int (&slots)[NS],
                                              const int (&n)[NS], double (&out)[NS], double *sm) {
  const double *p[NS];
  int nmax = 0;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    p[s] = part_ptr(d, c, slots[s]);
    out[s] = 0.0;
    nmax = max(nmax, n[s]);
  }
#pragma unroll 2
  for (int i = threadIdx.x; i < nmax; i += NT) {
#pragma unroll
    for (int s = 0; s < NS; ++s)
      if (i < n[s]) out[s] += __ldcg(p[s] + i);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int s = 0; s < NS; ++s) out[s] += __shfl_xor_sync(0xffffffffu, out[s], o);
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int s = 0; s < NS; ++s) sm[s * (NT / 32) + (threadIdx.x >> 5)] = out[s];
  }
  __syncthreads();
  if (threadIdx.x < NS) {
    double v[NT / 32];
#pragma unroll
    for (int i = 0; i < NT / 32; ++i) v[i] = sm[threadIdx.x * (NT / 32) + i];
#pragma unroll
    for (int o = NT / 64; o > 0; o >>= 1) {
#pragma unroll
      for (int i = 0; i < o; ++i) v[i] += v[i + o];
    }
    sm[NS * (NT / 32) + threadIdx.x] = v[0];
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < NS; ++s) out[s] = sm[NS * (NT / 32) + s];
}

// The schedule's scalars that do not depend on one another, each by a thread
// of its own warp so that their FP64 chains run side by side: momentum, gamma
// and (k >= 1) lambda's factor.  Every thread of the block calls it.
struct NextScalars {
  double a_next, coef, gamma, mu;
};
__device__ __forceinline__ void next_scalars(const Dev &d, const CopyState *cs, bool first,
                                             double hpwl, NextScalars *s) {
  const place_params &P = d.prm;
  if (threadIdx.x == 32) {
    const double a = cs->a;
    s->a_next = (1.0 + sqrt(4.0 * a * a + 1.0)) / 2.0;
    s->coef = (a - 1.0) / s->a_next;
  } else if (threadIdx.x == 64) {
    s->gamma = gamma_of(d, cs->tau);
  } else if (threadIdx.x == 96 && !first) {
    const double y = 1.0 - (hpwl - cs->hpwl_prev) / d.dref;
    const double mu = d.lg_mu != 0.0 && fabs(y * d.lg_mu) < 900.0 ? pow_log2(y, d.lg_mu, d.lg_mu_lo)
                                                                  : pow((double)P.mu_base, y);
    s->mu = fmin(fmax(mu, (double)P.mu_lo), (double)P.mu_hi);
  }
}

// Momentum, lambda schedule and gamma after iteration k, whose step length is
// alpha (thread 0, after a barrier behind next_scalars).
__device__ __forceinline__ void advance_scalars(CopyState *cs, bool first, double alpha,
                                                const NextScalars &s) {
  cs->alpha = alpha;
  cs->a_next = s.a_next;
  cs->coef = s.coef;
  if (!first) cs->lam *= s.mu;
  cs->hpwl_prev = cs->hpwl;
  cs->tau_prev = cs->tau;
  cs->gamma = s.gamma;
}

// Gradient of the wirelength (the cell's packed fixed-point pin-gradient sum,
// read and cleared for the next pass) and of the density (field gather -sum_b a_ib E_b) for every movable cell.
// For k >= 1 (lambda known) the preconditioned gradient and the step-size
// norms are formed here too, and the last block advances the scalars.
// STRETCH (density stretching on): the field is gathered over the cell's
// stretched rectangle and scaled by its density scale R / 2^31.
// Cells of more bins than kWarpGather (movable macros) are gathered by the
// whole warp: left to one lane, a macro of 17 x 17 bins held the
// stage for 110 us instead of 28 on the 210k-cell mixed-size design.
constexpr float kWarpGather = 32.f;

// PAIR: the field as (Ex, Ey) pairs (fused solves), one 8-byte load
// per bin instead of two of 4 bytes from two planes.
// BIG: the design has such cells (the other designs' kernel is 15% faster
// without the warp-wide step).
template <bool STRETCH, bool PAIR, bool BIG>
__global__ void __launch_bounds__(kThreads, 3) k_cell_grad(Dev d, int copy0, int eval) {
  __shared__ double smd[6 * (kThreads / 32) + 6];
  __shared__ float2 smc[3 * (kThreads / 32)];
  __shared__ double s_pre[3];
  __shared__ NextScalars s_next;
  __shared__ int flag;
  pdl_wait();
  const int c = copy0 + blockIdx.y;
  CopyState *cs = d.cs + c;
  if (!eval && cs->stopped) return;
  const int k = cs->k;
  const bool full = !eval && k >= 1;
  const float lam = (float)cs->lam;
  const int par = cs->parity;
  const size_t cn = (size_t)c * d.n_cells, cm = (size_t)c * d.n_mov;
  const float2 *xy = d.xy + cn;
  unsigned long long *ga = d.gacc + cm;
  const float *ex = d.E + (size_t)c * 3 * d.G, *ey = ex + d.G;
  const float2 *exy = reinterpret_cast<const float2 *>(ex);
  auto field = [&](size_t b) { return PAIR ? exy[b] : make_float2(ex[b], ey[b]); };
  float n1 = 0.f, d1 = 0.f, dg2 = 0.f;
  const float2 *wh = d.wh, *pa = d.pa, *go = d.g[par ^ 1] + cm;
  // every load of the next cell is issued while this cell's field gather is
  // in flight (the gather depends on the position): two cells' loads per
  // thread in flight, at 80 registers and three blocks per SM (measured on
  // the 2.1M-cell design: the stage 0.062 -> 0.059 ms at iteration 500, the
  // iteration 0.310 -> 0.306 ms; four blocks of 64 registers with only the
  // position prefetched, or of 40 registers, were slower)
  const int stride = gridDim.x * blockDim.x;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  const float2 zero2 = make_float2(0.f, 0.f);
  float2 vnext = i < d.n_mov ? xy[i] : zero2, whn = i < d.n_mov ? wh[i] : zero2;
  unsigned long long gsn = i < d.n_mov ? ga[i] : 0ull;
  float2 pan = zero2, gon = zero2;
  if (full && i < d.n_mov) {
    pan = pa[i]; gon = go[i];
  }
  // A large design has thousands of WA partials: each block adds up its share
  // (a warp, while the loads above are in flight), and the last block sums one
  // value per block.  Left to the last block alone they are 3.5 us of one SM's
  // FP64 pipe at 2.1M cells (5163 partials, two values each); at 210k cells
  // (1925) the blocks' extra FP64 work costs a batched handle what it saves, so
  // the line lies between.  It does not depend on the number of copies, so that
  // a copy sums in the same order in every batch.
  const bool pre = !eval && d.wa_blocks_total > 2048 && gridDim.x >= 64;
  if (pre && threadIdx.x >= kThreads - 32) {
    double h = 0.0, w = 0.0, v = 0.0;
    const int step = gridDim.x * 32, j0 = blockIdx.x + gridDim.x * (threadIdx.x & 31);
    for (int j = j0; j < d.wa_blocks_total; j += step) {
      h += part_ptr(d, c, S_HPWL)[j];
      w += part_ptr(d, c, S_WL)[j];
    }
    if (k > 0)
      for (int j = j0; j < d.cell_blocks; j += step) v += part_ptr(d, c, S_DV2)[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      h += __shfl_xor_sync(0xffffffffu, h, o);
      w += __shfl_xor_sync(0xffffffffu, w, o);
      v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    if (threadIdx.x == kThreads - 1) {
      s_pre[0] = h; s_pre[1] = w; s_pre[2] = v;
    }
  }
  // (BIG: a warp's lanes stay together to the last cell)
  for (; i - (BIG ? (int)(threadIdx.x & 31) : 0) < d.n_mov; i += stride) {
    const bool valid = BIG ? i < d.n_mov : true;
    const unsigned long long gs = gsn;
    const float2 vi = vnext;
    const float wi = whn.x, hi = whn.y;
    const float np = pan.x, ar = pan.y, gxp = gon.x, gyp = gon.y;
    const int in = i + stride;
    if (in < d.n_mov) {
      vnext = xy[in];
      whn = wh[in];
      gsn = ga[in];
      if (full) {
        pan = pa[in]; gon = go[in];
      }
    }
    if (valid) ga[i] = 0ull;
    const float2 sw = unpack_grad(d, gs);
    const float sx = sw.x, sy = sw.y;
    // density gradient: -sum_b |cell ∩ b| E_b over the bins the cell covers,
    // in FP32 with coordinates relative to the first bin's corner (exact
    // subtractions, so each overlap keeps FP32 relative precision)
    const float xi = vi.x, yi = vi.y;
    float xg = xi, yg = yi, wg = wi, hg = hi, scale_g = 1.f;
    if (STRETCH && valid) {
      const int4 st = d.st[i];
      xg = xi - (float)st.x * d.inv_scale;
      yg = yi - (float)st.y * d.inv_scale;
      wg = (float)st.z * d.inv_scale;
      hg = (float)st.w * d.inv_scale;
      scale_g = (float)d.sR[i] * 4.656612873077393e-10f;  // 2^-31
    }
    const int ix0 = min(max((int)floorf((xg - d.fxl) * d.fibw), 0), d.nx - 1);
    const int iy0 = min(max((int)floorf((yg - d.fyl) * d.fibh), 0), d.ny - 1);
    const float rx = xg - (d.fxl + (float)ix0 * d.fbw), ry = yg - (d.fyl + (float)iy0 * d.fbh);
    const float rx1 = rx + wg, ry1 = ry + hg;
    float dx = 0.f, dy = 0.f;
    const bool wide = valid && !(wg <= d.fbw && hg <= d.fbh);
    // bins per axis, rounded up or one more (0 for a cell that is not on the grid)
    float nbx = 0.f, nby = 0.f;
    if constexpr (BIG) {
      nbx = rx1 > 0.f ? fminf(rx1 * d.fibw, 8192.f) + 1.f : 0.f;
      nby = ry1 > 0.f ? fminf(ry1 * d.fibh, 8192.f) + 1.f : 0.f;
    }
    const bool big = BIG && wide && nbx * nby > kWarpGather;
    if (valid && !wide) {
      // no larger than a bin: at most the 2 x 2 bins from (ix0, iy0), the
      // far ones loaded only where the cell reaches them
      const float ox0 = fmaxf(fminf(rx1, d.fbw) - fmaxf(rx, 0.f), 0.f);
      const float oy0 = fmaxf(fminf(ry1, d.fbh) - fmaxf(ry, 0.f), 0.f);
      const float ox1 = ix0 + 1 < d.nx ? fmaxf(rx1 - d.fbw, 0.f) : 0.f;
      const float oy1 = iy0 + 1 < d.ny ? fmaxf(ry1 - d.fbh, 0.f) : 0.f;
      const size_t b0 = (size_t)ix0 * d.ny + iy0;
      if (HP_IN(d.err, (long long)b0 + (ox1 > 0.f ? d.ny : 0) + (oy1 > 0.f ? 1 : 0), d.G,
                BS_FIELD_BIN)) {
        const bool far = ox1 > 0.f && oy1 > 0.f;
        const float2 e00 = field(b0), e01 = oy1 > 0.f ? field(b0 + 1) : zero2;
        const float2 e10 = ox1 > 0.f ? field(b0 + d.ny) : zero2, e11 = far ? field(b0 + d.ny + 1) : zero2;
        dx = -(ox0 * fmaf(oy0, e00.x, oy1 * e01.x) + ox1 * fmaf(oy0, e10.x, oy1 * e11.x));
        dy = -(ox0 * fmaf(oy0, e00.y, oy1 * e01.y) + ox1 * fmaf(oy0, e10.y, oy1 * e11.y));
      }
    } else if (wide && !big) {
      for (int kx = 0, ix = ix0; ix < d.nx && (float)kx * d.fbw < rx1; ++kx, ++ix) {
        const float ox = fminf(rx1, (float)(kx + 1) * d.fbw) - fmaxf(rx, (float)kx * d.fbw);
        if (!(ox > 0.f)) continue;
        for (int ky = 0, iy = iy0; iy < d.ny && (float)ky * d.fbh < ry1; ++ky, ++iy) {
          const float oy = fminf(ry1, (float)(ky + 1) * d.fbh) - fmaxf(ry, (float)ky * d.fbh);
          if (!(oy > 0.f)) continue;
          const float a = ox * oy;
          if (!HP_IN(d.err, (long long)ix * d.ny + iy, d.G, BS_FIELD_BIN)) continue;
          const float2 e = field((size_t)ix * d.ny + iy);
          dx = fmaf(-a, e.x, dx);
          dy = fmaf(-a, e.y, dy);
        }
      }
    }
    if constexpr (BIG) {
      // cells of more bins (movable macros) one after another by the whole warp,
      // a bin per lane, in a fixed order
      unsigned int bigs = __ballot_sync(0xffffffffu, big);
      while (bigs) {
        const int l = __ffs(bigs) - 1;
        bigs &= bigs - 1;
        const float bx = __shfl_sync(0xffffffffu, rx, l), by = __shfl_sync(0xffffffffu, ry, l);
        const float bx1 = __shfl_sync(0xffffffffu, rx1, l), by1 = __shfl_sync(0xffffffffu, ry1, l);
        const int jx = __shfl_sync(0xffffffffu, ix0, l), jy = __shfl_sync(0xffffffffu, iy0, l);
        const int mx = min((int)__shfl_sync(0xffffffffu, nbx, l) + 1, d.nx - jx);
        const int my = min((int)__shfl_sync(0xffffffffu, nby, l) + 1, d.ny - jy);
        float sx = 0.f, sy = 0.f;
        for (int q = threadIdx.x & 31; q < mx * my; q += 32) {
          const int kx = q / my, ky = q - kx * my;
          const float ox = fminf(bx1, (float)(kx + 1) * d.fbw) - fmaxf(bx, (float)kx * d.fbw);
          const float oy = fminf(by1, (float)(ky + 1) * d.fbh) - fmaxf(by, (float)ky * d.fbh);
          const size_t bin = (size_t)(jx + kx) * d.ny + jy + ky;
          if (!(ox > 0.f) || !(oy > 0.f) || !HP_IN(d.err, bin, d.G, BS_FIELD_BIN)) continue;
          const float2 e = field(bin);
          sx = fmaf(-ox * oy, e.x, sx);
          sy = fmaf(-ox * oy, e.y, sy);
        }
  #pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          sx += __shfl_xor_sync(0xffffffffu, sx, o);
          sy += __shfl_xor_sync(0xffffffffu, sy, o);
        }
        if ((threadIdx.x & 31) == l) {
          dx = sx;
          dy = sy;
        }
      }
      if (!valid) break;  // the warp's last step
    }
    if constexpr (STRETCH) {
      dx *= scale_g;
      dy *= scale_g;
    }
    if (!full) {  // raw gradients are read only by k = 0 (lambda_0) and evaluations
      d.gwx[cm + i] = sx; d.gwy[cm + i] = sy;
      d.gdx[cm + i] = dx; d.gdy[cm + i] = dy;
    }
    n1 += fabsf(sx) + fabsf(sy);
    d1 += fabsf(dx) + fabsf(dy);
    if (full) {
      const float rP = 1.f / fmaxf(1.f, np + lam * ar);
      const float gx = (sx + lam * dx) * rP, gy = (sy + lam * dy) * rP;
      d.g[par][cm + i] = make_float2(gx, gy);
      const float ax = gx - gxp, ay = gy - gyp;
      dg2 += ax * ax + ay * ay;
    }
  }
  // per-thread sums in FP32 (a few cells each), compensated block sums:
  // these norms set lambda_0 and every step length
  float nv[3] = {n1, d1, dg2};
  double nr[3];
  block_sums_fc<kThreads, 3>(nv, smc, nr);
  if (threadIdx.x == 0) {
    part_ptr(d, c, S_GW1)[blockIdx.x] = nr[0];
    part_ptr(d, c, S_GD1)[blockIdx.x] = nr[1];
    part_ptr(d, c, S_DG2)[blockIdx.x] = nr[2];
    if (pre) {
      part_ptr(d, c, S_PH)[blockIdx.x] = s_pre[0];
      part_ptr(d, c, S_PW)[blockIdx.x] = s_pre[1];
      part_ptr(d, c, S_PV)[blockIdx.x] = s_pre[2];
    }
  }
  if (eval) return;
  if (!arrive_last_t0(d.ctr + (size_t)c * C_COUNT + C_CELL, &flag)) return;
  // The serial end of the iteration: k_update waits for it.  Its FP64 work is
  // spread over the block (all sums in one pass, the scalars on four warps, no
  // pow): with one sum after another and all scalars on thread 0 an iteration
  // took 74.6 us at 1k cells, 113 at 210k and 337 at 2.1M; so, 64.0, 100 and
  // 321.
  // |v_k - v_{k-1}|^2 (S_DV2): the partials of the step that led here
  // (k_update or k_redo_step, one per block of their grid)
  const int ng = gridDim.x;
  const int slots[6] = {pre ? S_PH : S_HPWL, pre ? S_PW : S_WL, S_GW1, S_GD1, S_DG2, pre ? S_PV : S_DV2};
  const int cnt[6] = {pre ? ng : d.wa_blocks_total, pre ? ng : d.wa_blocks_total, ng, ng, ng,
                      k > 0 ? (pre ? ng : d.cell_blocks) : 0};
  double sum[6];
  sum_slots_all<kThreads, 6>(d, c, slots, cnt, sum, smd);
  next_scalars(d, cs, k == 0, sum[0], &s_next);
  const double s1 = sum[2], s2 = sum[3], s3 = sum[4], s4 = sum[5];
  double lam0 = 0.0, est = 0.0;
  if (threadIdx.x == 0) {
    if (k == 0)
      lam0 = s2 > 0 ? (double)d.prm.lambda_eta * s1 / s2 : (double)d.prm.lambda_eta;
    else
      est = s3 > 0 ? sqrt(s4) / sqrt(s3) : cs->alpha;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    cs->hpwl = sum[0];
    cs->wl = sum[1];
    if (k == 0) {
      cs->lam = lam0;
    } else {
      // backtracking: a step-length estimate below 0.95 times the step that
      // led here sends k_update back to redo that step with the estimate
      if (d.prm.max_backtracks > 0 && cs->n_back < d.prm.max_backtracks && est < 0.95 * cs->alpha) {
        cs->alpha = est;
        cs->n_back += 1;
        cs->n_back_total += 1;
        cs->reject = 1;
      } else {
        cs->n_back = 0;
        advance_scalars(cs, false, est, s_next);
      }
    }
    d.ctr[(size_t)c * C_COUNT + C_CELL] = 0u;
  }
}

// k == 0 only: preconditioned gradient once lambda_0 is known, |g|^2, and the
// first step length.
__global__ void __launch_bounds__(kThreads) k_precond0(Dev d, int copy0) {
  __shared__ double smd[kThreads / 32 + 1];
  __shared__ float2 smc[32];
  __shared__ NextScalars s_next;
  __shared__ int flag;
  pdl_wait();
  const int c = copy0 + blockIdx.y;
  CopyState *cs = d.cs + c;
  if (cs->stopped || cs->k != 0) return;
  const float lam = (float)cs->lam;
  const int par = cs->parity;
  const size_t cm = (size_t)c * d.n_mov;
  float g2 = 0.f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d.n_mov; i += gridDim.x * blockDim.x) {
    const float2 q = d.pa[i];
    float P = fmaxf(1.f, q.x + lam * q.y);
    float gx = (d.gwx[cm + i] + lam * d.gdx[cm + i]) / P;
    float gy = (d.gwy[cm + i] + lam * d.gdy[cm + i]) / P;
    d.g[par][cm + i] = make_float2(gx, gy);
    g2 += gx * gx + gy * gy;
  }
  const double r = block_sum_fc<kThreads>(g2, smc);
  if (threadIdx.x == 0) part_ptr(d, c, S_G2)[blockIdx.x] = r;
  if (!arrive_last_t0(d.ctr + (size_t)c * C_COUNT + C_PRE0, &flag)) return;
  const int slots[1] = {S_G2}, cnt[1] = {(int)gridDim.x};
  double s[1];
  sum_slots_all<kThreads, 1>(d, c, slots, cnt, s, smd);
  next_scalars(d, cs, true, 0.0, &s_next);
  double alpha = 0.0;
  if (threadIdx.x == 0) {
    const double rms = sqrt(s[0] / (2.0 * d.n_mov));
    alpha = rms > 0 ? (double)d.prm.alpha0 * d.w_bin / rms : 0.0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    advance_scalars(cs, true, alpha, s_next);
    d.ctr[(size_t)c * C_COUNT + C_PRE0] = 0u;
  }
}

// Nesterov step with clamping into the die; the last block closes the
// iteration (k, a_k, buffer parity, max_iters stop).  KEEP_U (backtracking
// on) also saves u_k, and a step that the cell-gradient pass rejected is
// left to k_redo_step.
template <bool KEEP_U>
__global__ void __launch_bounds__(kThreads) k_update(Dev d, int copy0) {
  __shared__ int flag;
  __shared__ float2 smc[32];
  pdl_wait();
  const int c = copy0 + blockIdx.y;
  CopyState *cs = d.cs + c;
  if (cs->stopped) return;
  if constexpr (KEEP_U) {
    if (cs->reject) return;
  }
  const float alpha = (float)cs->alpha, coef = (float)cs->coef;
  const int par = cs->parity;
  const size_t cn = (size_t)c * d.n_cells, cm = (size_t)c * d.n_mov;
  float dv2 = 0.f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d.n_mov; i += gridDim.x * blockDim.x) {
    const float2 s = d.wh[i];
    const float xh = d.fxh - s.x, yh = d.fyh - s.y;
    const float2 v = d.xy[cn + i];
    const float vx = v.x, vy = v.y;
    const float2 u = d.u[cm + i], g = d.g[par][cm + i];
    const float ux = u.x, uy = u.y;
    float nux = fmaxf(d.fxl, fminf(vx - alpha * g.x, xh));
    float nuy = fmaxf(d.fyl, fminf(vy - alpha * g.y, yh));
    float nvx = fmaxf(d.fxl, fminf(nux + coef * (nux - ux), xh));
    float nvy = fmaxf(d.fyl, fminf(nuy + coef * (nuy - uy), yh));
    if constexpr (KEEP_U) {  // a rejected next step restarts from v_k and u_k
      d.vp[cm + i] = v;
      d.up[cm + i] = u;
    }
    d.u[cm + i] = make_float2(nux, nuy);
    d.xy[cn + i] = make_float2(nvx, nvy);
    const float bx = nvx - vx, by = nvy - vy;
    dv2 += bx * bx + by * by;
  }
  // |v_{k+1} - v_k|^2 per block, for the next iteration's step length: the
  // update knows both points, so v_k need not be stored and read back
  const double r = block_sum_fc<kThreads>(dv2, smc);
  if (threadIdx.x == 0) part_ptr(d, c, S_DV2)[blockIdx.x] = r;
  if (!arrive_last_t0(d.ctr + (size_t)c * C_COUNT + C_UPDATE, &flag)) return;
  if (threadIdx.x == 0) {
    // the iteration's record: its HPWL (WA pass) and overflow at v_k, the
    // step length taken, and the lambda and gamma the next iteration uses
    place_iter_record r;
    r.iter = cs->k;
    r.backtracks = cs->n_back_total;
    r.hpwl_wa = cs->hpwl;
    r.overflow = cs->tau;
    r.lambda = cs->lam;
    r.gamma = cs->gamma;
    r.alpha = cs->alpha;
    d.hist[(size_t)c * d.hist_cap + (cs->n_hist % d.hist_cap)] = r;
    cs->n_hist += 1;
    cs->k += 1;
    cs->a = cs->a_next;
    cs->parity ^= 1;
    if (cs->k >= d.prm.max_iters) cs->stopped = 1;
    d.ctr[(size_t)c * C_COUNT + C_UPDATE] = 0u;
  }
}

// Backtracking: redo the rejected step from v_{k-1}, u_{k-1} and g_{k-1}
// with the shorter length the cell-gradient pass stored; k, a_k and the
// buffer parity stay.  Launched after k_update on handles with backtracking.
__global__ void __launch_bounds__(kThreads) k_redo_step(Dev d, int copy0) {
  __shared__ int flag;
  __shared__ float2 smc[32];
  pdl_wait();
  const int c = copy0 + blockIdx.y;
  CopyState *cs = d.cs + c;
  if (cs->stopped || !cs->reject) return;
  const float alpha = (float)cs->alpha, coef = (float)cs->coef;
  const int par = cs->parity;
  const size_t cn = (size_t)c * d.n_cells, cm = (size_t)c * d.n_mov;
  const float2 *go = d.g[par ^ 1] + cm;
  float dv2 = 0.f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d.n_mov; i += gridDim.x * blockDim.x) {
    const float2 s = d.wh[i];
    const float xh = d.fxh - s.x, yh = d.fyh - s.y;
    const float2 v = d.vp[cm + i], u = d.up[cm + i], g = go[i];
    const float vx = v.x, vy = v.y, ux = u.x, uy = u.y;
    const float nux = fmaxf(d.fxl, fminf(vx - alpha * g.x, xh));
    const float nuy = fmaxf(d.fyl, fminf(vy - alpha * g.y, yh));
    d.u[cm + i] = make_float2(nux, nuy);
    const float nvx = fmaxf(d.fxl, fminf(nux + coef * (nux - ux), xh));
    const float nvy = fmaxf(d.fyl, fminf(nuy + coef * (nuy - uy), yh));
    d.xy[cn + i] = make_float2(nvx, nvy);
    const float bx = nvx - vx, by = nvy - vy;
    dv2 += bx * bx + by * by;
  }
  const double r = block_sum_fc<kThreads>(dv2, smc);  // the redone step's |v_k - v_{k-1}|^2
  if (threadIdx.x == 0) part_ptr(d, c, S_DV2)[blockIdx.x] = r;
  if (!arrive_last_t0(d.ctr + (size_t)c * C_COUNT + C_UPDATE, &flag)) return;
  if (threadIdx.x == 0) {
    cs->reject = 0;
    d.ctr[(size_t)c * C_COUNT + C_UPDATE] = 0u;
  }
}

// Optimiser reset: new positions where there are any, the movable ones clamped
// into the die, u = v, and initial scalars (tau_{-1} and gamma_0 follow from
// the density pass).
__global__ void __launch_bounds__(kThreads) k_reset(Dev d, int copy0, NewXy src) {
  const int c = copy0 + blockIdx.y;
  const size_t cn = (size_t)c * d.n_cells, cm = (size_t)c * d.n_mov;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d.n_mov; i += gridDim.x * blockDim.x) {
    const float2 v = i >= src.lo && i < src.hi ? make_float2(src.x[i - src.lo], src.y[i - src.lo])
                                               : d.xy[cn + i];
    const float2 s = d.wh[i];
    float vx = fmaxf(d.fxl, fminf(v.x, d.fxh - s.x));
    float vy = fmaxf(d.fyl, fminf(v.y, d.fyh - s.y));
    d.xy[cn + i] = make_float2(vx, vy);
    d.u[cm + i] = make_float2(vx, vy);
    d.gacc[cm + i] = 0ull;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    CopyState s = {};
    s.a = 1.0;
    d.cs[c] = s;
  }
}

// Reduce one slot for evaluation calls: d.scal[c * S_COUNT + slot].
__global__ void __launch_bounds__(kRedThreads) k_reduce_slot(Dev d, int slot, int nvals,
                                                             int copy0) {
  __shared__ double sm[32];
  const int c = copy0 + blockIdx.x;
  double s = sum_slot<kRedThreads>(d, c, slot, nvals, sm);
  if (threadIdx.x == 0) d.scal[(size_t)c * S_COUNT + slot] = s;
}

// Cells [0, n0) and, past `skip` others, the rest of n cells: x and y (either
// may be null) from interleaved positions.
__global__ void k_unpack_xy(float *x, float *y, const float2 *src, int n0, int n, int skip) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float2 v = src[i < n0 ? i : i + skip];
    if (x) x[i] = v.x;
    if (y) y[i] = v.y;
  }
}

void launch_unpack_xy(float *x, float *y, const float2 *src, int n0, int n, int skip, cudaStream_t st) {
  if (n <= 0) return;
  int b = (n + kThreads - 1) / kThreads;
  k_unpack_xy<<<b < 4096 ? b : 4096, kThreads, 0, st>>>(x, y, src, n0, n, skip);
}

// A copy's WA gradient sums as floats (the design's movable cells), and cleared
// for the next pass: place_eval_wirelength, which needs nothing else of the
// cell-gradient pass.
__global__ void __launch_bounds__(kThreads) k_wa_unpack(Dev d, int copy, float *gx, float *gy) {
  unsigned long long *ga = d.gacc + (size_t)copy * d.n_mov;
  for (int i = blockIdx.x * kThreads + threadIdx.x; i < d.n_mov; i += gridDim.x * kThreads) {
    const float2 g = unpack_grad(d, ga[i]);
    ga[i] = 0ull;
    if (i < d.n_real) {
      gx[i] = g.x;
      gy[i] = g.y;
    }
  }
}
void launch_wa_unpack(const Dev &d, int copy, float *gx, float *gy, cudaStream_t st) {
  k_wa_unpack<<<d.cell_blocks, kThreads, 0, st>>>(d, copy, gx, gy);
}

namespace {
using CellGrad = void (*)(Dev, int, int);
CellGrad cell_grad_kernel(bool stretch, bool pair, bool big) {
  static const CellGrad k[2][2][2] = {
      {{k_cell_grad<false, false, false>, k_cell_grad<false, false, true>},
       {k_cell_grad<false, true, false>, k_cell_grad<false, true, true>}},
      {{k_cell_grad<true, false, false>, k_cell_grad<true, false, true>},
       {k_cell_grad<true, true, false>, k_cell_grad<true, true, true>}}};
  return k[stretch][pair][big];
}
}  // namespace

void launch_cell_grad(const Dev &d, int copy0, int ncopy, int eval, cudaStream_t st) {
  launch_pdl(cell_grad_kernel(d.Ms != nullptr, d.solve != SOLVE_GEMM, d.has_big != 0),
             dim3(d.cg_blocks, ncopy), dim3(kThreads), 0, st, d, copy0, eval);
}
// One failing index check and no access (place_test_bounds_check).
__global__ void k_test_bounds(Dev d) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    const long long i = d.n_cells;  // one past the last cell
    if (HP_IN(d.err, i, d.n_cells, BS_WA_CELL)) d.err[1] = 0;  // (reached only when it passes)
  }
}
void launch_test_bounds(const Dev &d, cudaStream_t st) { k_test_bounds<<<1, 32, 0, st>>>(d); }

int cell_grad_blocks_per_sm(const Dev &d) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &n, cell_grad_kernel(d.prm.stretch != 0, d.solve != SOLVE_GEMM, d.has_big != 0), kThreads,
          0) != cudaSuccess || n < 1)
    n = 1;
  return n;
}
void launch_precond0(const Dev &d, int copy0, int ncopy, cudaStream_t st) {
  launch_pdl(k_precond0, dim3(d.cell_blocks, ncopy), dim3(kThreads), 0, st, d, copy0);
}
void launch_update(const Dev &d, int copy0, int ncopy, cudaStream_t st) {
  const dim3 grid(d.cell_blocks, ncopy);
  if (d.up) {
    launch_pdl(k_update<true>, grid, dim3(kThreads), 0, st, d, copy0);
    launch_pdl(k_redo_step, grid, dim3(kThreads), 0, st, d, copy0);
  } else {
    launch_pdl(k_update<false>, grid, dim3(kThreads), 0, st, d, copy0);
  }
}
void launch_reset(const Dev &d, int copy0, int ncopy, const NewXy &src, cudaStream_t st) {
  k_reset<<<dim3(d.cell_blocks, ncopy), kThreads, 0, st>>>(d, copy0, src);
}
void launch_reduce_slot(const Dev &d, int slot, int nvals, int copy0, int ncopy,
                        cudaStream_t st) {
  k_reduce_slot<<<ncopy, kRedThreads, 0, st>>>(d, slot, nvals, copy0);
}

}  // namespace hp
