// WireMask perturbation (the perturbation step of Algorithm 1; Section 4.2):
// every movable macro, one after another, moves to the grid position where
// the HPWL grows least.  Reading used by this library:
//   - macros: the movable cells flagged is_macro, by decreasing area (ties
//     by index);
//   - candidates: the macro's lower-left corner on a bin corner,
//     X_i = fl32(xl + i (xh - xl)/nx), inside the die (X_i + w <= xh);
//   - wire mask: the weighted HPWL (Eq. 1) of the macro's nets with the
//     macro at the candidate and every other pin where it is (macros moved
//     earlier in the pass at their new places).  For one net, with the
//     other pins' extent [o-, o+] and the macro's pin offsets [d-, d+], the
//     x part is max(o+, X + d+) - min(o-, X + d-).  The mask is separable,
//     Fx(X_i) + Fy(Y_j), each axis summed over the macro's nets in netlist
//     order;
//   - obstacles: every fixed cell and the macros moved before this one;
//     overlap of positive area blocks a candidate (touching is allowed);
//   - choice: the smallest (Fx + Fy, |X - x| + |Y - y|, j, i) among the
//     free candidates, (x, y) the macro's position before it moves; with
//     none free the macro stays.
// Every value that decides a comparison is FP64 from a fixed sequence of
// correctly rounded operations (explicit _rn intrinsics, so no contraction
// into fused multiply-adds), so the result is bit-exact and
// independent of the launch shape.
//
// What bounds it: the chain over the macros, so everything that does not
// depend on the macros moved before is done once, in parallel, and a macro
// costs two launches:
//   - k_wm_static, once per pass, a block per net with macros on it: the extent
//     of the net's pins on other cells than movable macros (exact FP32 pairs,
//     pairs.cuh, as FP64 minima and maxima are GB300's slowest instructions),
//     and from it, adding the net's macros from the last one to move back to
//     the first, for each of them the extent of those pins and of the
//     macros that still stand where they were;
//   - k_wm_mask per macro: each net's extent with that of the macros that have
//     moved (kept per net, one step of minimum and maximum a macro), the two
//     mask axes with the distances of their corners, and every obstacle as the
//     exact range of candidate columns and rows that it blocks (stepping from a
//     guess);
//   - k_wm_select per macro: a block per row of candidates turns the
//     obstacles that cover the row into a bit mask, so that a candidate costs
//     one bit test, one FP64 addition and one comparison; the last block
//     reduces the rows' winners, moves the macro and adds it to its nets'
//     moved extents.
// So the tables hold one entry per macro and net, and a macro's cost depends on
// the number of its nets, not on how many macros share them.
// Copies run side by side (blockIdx.y; w.group of them).  One pass over 32 macros of
// a 210k-cell design on 512 x 512 bins, restored before and read back: 3.7 -> 0.54 ms against one warp per net in FP64
// and four launches a macro.  (Launching each kernel early, by
// griddepcontrol.launch_dependents at its start or before its last step, took
// 28 us a macro instead of 15: measured, not taken.)
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "internal.cuh"
#include "pairs.cuh"

namespace hp {

namespace {

constexpr int kWmThreads = 128;   // select: threads per row of candidates
constexpr int kWmLines = 64;      // mask: grid lines (and nets in shared memory) per block
constexpr int kWmNetThreads = 256;

__device__ __forceinline__ double wm_step(double lo, double hi, int n) {
  return __ddiv_rn(__dsub_rn(hi, lo), (double)n);
}
// Candidate corner i: fl32(lo + i b) with b = (hi - lo) / n.
__device__ __forceinline__ double wm_corner_b(double lo, double b, int i) {
  return (double)__double2float_rn(__dadd_rn(lo, __dmul_rn((double)i, b)));
}
__device__ __forceinline__ double wm_corner(double lo, double hi, int n, int i) {
  return wm_corner_b(lo, wm_step(lo, hi, n), i);
}

// First k in [0, n] at which a predicate that is false and then true over
// [0, n) holds (n when it never does), stepping from a guess.
template <typename P>
__device__ __forceinline__ int first_true(int n, int guess, P pred) {
  int k = min(max(guess, 0), n);
  while (k > 0 && pred(k - 1)) --k;
  while (k < n && !pred(k)) ++k;
  return k;
}

// The corners i whose macro rectangle [X_i, X_i + w) overlaps [o0, o1) with
// positive length: X_i < o1 and o0 < X_i + w.  The corners are
// nondecreasing in i (rounding is monotone), so the first test holds for i
// below some bound and the second from some bound on.  Two searches over the
// same FP64 expressions, each from an estimate that is at most a corner or two
// off, give the range [i0, i1] exactly.
__device__ __forceinline__ int2 blocked_range(double lo, double b, int n, double w, double o0,
                                              double o1) {
  const float ib = 1.f / (float)b;
  const int g0 = (int)floorf(fminf(fmaxf((float)(o0 - w - lo) * ib, -2.f), 16384.f));
  const int g1 = (int)floorf(fminf(fmaxf((float)(o1 - lo) * ib, -2.f), 16384.f));
  const int i0 = first_true(n, g0 + 1, [&](int i) { return o0 < __dadd_rn(wm_corner_b(lo, b, i), w); });
  const int i1 = first_true(n, g1 + 1, [&](int i) { return !(wm_corner_b(lo, b, i) < o1); }) - 1;
  return make_int2(i0, i1);
}

// A candidate's key, compared as integers: the FP64 objective and distance in
// an order-preserving form (neither is ever -0), then the candidate's index.
// no_best() is after every candidate.
struct Best {
  unsigned long long obj, dist;
  int idx;  // flat candidate index j * nx + i
};
constexpr int kNoIdx = 0x7fffffff;
__device__ __forceinline__ Best no_best() { return Best{~0ull, ~0ull, kNoIdx}; }

__device__ __forceinline__ unsigned long long ordered(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  return u ^ ((u >> 63) ? ~0ull : 0x8000000000000000ull);
}

__device__ __forceinline__ bool better(const Best &a, const Best &b) {
  if (a.obj != b.obj) return a.obj < b.obj;
  if (a.dist != b.dist) return a.dist < b.dist;
  return a.idx < b.idx;
}

// Block-wide minimum (every thread of the block calls it); result in thread 0.
__device__ Best block_best(Best v) {
  __shared__ Best sb[kWmThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const Best w{__shfl_xor_sync(0xffffffffu, v.obj, o), __shfl_xor_sync(0xffffffffu, v.dist, o),
                 __shfl_xor_sync(0xffffffffu, v.idx, o)};
    if (better(w, v)) v = w;
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sb[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 1; k < kWmThreads / 32; ++k)
      if (better(sb[k], v)) v = sb[k];
  }
  return v;
}

// An extent {x-, x+, y-, y+}; empty: +-inf.
struct Extent {
  double v[4];
};
__device__ __forceinline__ Extent no_extent() { return Extent{{INFINITY, -INFINITY, INFINITY, -INFINITY}}; }
__device__ __forceinline__ void extent_add(Extent &a, const Extent &b) {
  a.v[0] = fmin(a.v[0], b.v[0]); a.v[1] = fmax(a.v[1], b.v[1]);
  a.v[2] = fmin(a.v[2], b.v[2]); a.v[3] = fmax(a.v[3], b.v[3]);
}
// A macro's pins on one net, with its corner at p and their offsets' extent o.
// (Rounding is monotone: the extent of the rounded sums is the rounded sum of
// the extent.)
__device__ __forceinline__ Extent extent_at(float2 p, float4 o) {
  return Extent{{__dadd_rn((double)p.x, (double)o.x), __dadd_rn((double)p.x, (double)o.y),
                 __dadd_rn((double)p.y, (double)o.z), __dadd_rn((double)p.y, (double)o.w)}};
}
__device__ __forceinline__ Extent load_extent(const double *p, size_t k) {
  Extent e;
#pragma unroll
  for (int i = 0; i < 4; ++i) e.v[i] = p[4 * k + i];
  return e;
}
__device__ __forceinline__ void store_extent(double *p, size_t k, const Extent &e) {
#pragma unroll
  for (int i = 0; i < 4; ++i) p[4 * k + i] = e.v[i];
}

// Net blockIdx.x of those with macros on them, its entries (a macro and the net)
// in the macros' order: the extent of its pins on other cells than movable
// macros, and for each entry that extent with the macros after it added, at
// their places before the pass.
__global__ void __launch_bounds__(kWmNetThreads) k_wm_static(Dev d, WmDev w, int copy0) {
  constexpr int kWarps = kWmNetThreads / 32;
  __shared__ PairBox sb[kWarps];
  __shared__ Extent se[kWarps], carry;
  const int c = copy0 + blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float2 *xy = d.xy + (size_t)c * d.n_cells;
  const int q0 = w.dptr[blockIdx.x], q1 = w.dptr[blockIdx.x + 1];
  int e = w.mnet[w.dent[q0]];
  HP_FIX(d.err, e, d.n_nets, BS_WM_NET);
  PairBox b = empty_box();
  bool any = false;
  for (int j = d.net_ptr[e] + threadIdx.x; j < d.net_ptr[e + 1]; j += kWmNetThreads) {
    if (!HP_IN(d.err, j, d.n_pins, BS_WM_NET)) break;
    int cj = d.pin_cell[j];
    HP_FIX(d.err, cj, d.n_cells, BS_WM_CELL);
    if (cj < d.n_real && d.is_macro[cj]) continue;
    box_add(b, xy[cj], d.pin_off[j], d.pin_scale);
    any = true;
  }
  box_reduce<32>(b);
  if (lane == 0) sb[warp] = b;
  any = __syncthreads_or(any);
  double *sbox = w.sbox + (size_t)blockIdx.y * w.n_entries * 4;
  if (threadIdx.x < 32) {
    b = sb[threadIdx.x % kWarps];
    box_reduce<kWarps>(b);
    if (threadIdx.x == 0) {
      const double un = d.pin_unscale;
      const Extent s = any ? Extent{{pair_value(b.nx, un), pair_value(b.mx, un), pair_value(b.ny, un),
                                     pair_value(b.my, un)}}
                           : no_extent();
      if (q1 - q0 == 1) {
        store_extent(sbox, w.dent[q0], s);
      } else {
        carry = s;
        store_extent(w.moved, (size_t)blockIdx.y * w.n_shared + w.slot[w.dent[q0]], no_extent());
      }
    }
  }
  if (q1 - q0 == 1) return;
  // a net of several macros: a scan from its last entry, in steps of a block
  for (int end = q1; end > q0; end -= kWmNetThreads) {
    const int q = end - 1 - (int)threadIdx.x;  // thread 0 has the last one
    int s = 0;
    Extent v = no_extent();
    if (q >= q0) {
      s = w.dent[q];
      int m = w.mcell[s];
      HP_FIX(d.err, m, d.n_cells, BS_WM_CELL);
      v = extent_at(xy[m], w.own[s]);
    }
    // inclusive over the warp, then the warps before and the steps before
    Extent in = v;
    for (int o = 1; o < 32; o <<= 1) {
      Extent x;
#pragma unroll
      for (int i = 0; i < 4; ++i) x.v[i] = __shfl_up_sync(0xffffffffu, in.v[i], o);
      if (lane >= o) extent_add(in, x);
    }
    Extent out;  // exclusive
#pragma unroll
    for (int i = 0; i < 4; ++i) out.v[i] = __shfl_up_sync(0xffffffffu, in.v[i], 1);
    if (lane == 0) out = no_extent();
    if (lane == 31) se[warp] = in;
    __syncthreads();
    for (int k = 0; k < warp; ++k) extent_add(out, se[k]);
    extent_add(out, carry);
    if (q >= q0) store_extent(sbox, s, out);
    __syncthreads();  // (carry and se have been read)
    if (threadIdx.x == kWmNetThreads - 1) {
      extent_add(out, v);
      carry = out;
    }
  }
}

// Macro t.  Blocks [0, lines): kWmLines grid lines each, line q < nx the
// column Fx(X_q), then the rows Fy(Y_q), summed over the macro's nets in
// order, and the distance of the corner from the macro's old one (-1: the
// macro would leave the die).  The other blocks: the obstacles' ranges.
__global__ void __launch_bounds__(kWmLines) k_wm_mask(Dev d, WmDev w, int t, int copy0, int lines) {
  __shared__ double box[8][kWmLines];
  __shared__ double sw[kWmLines];
  // the tables are the handle's constants: read before the wait
  const int c = copy0 + blockIdx.y;
  const float2 *xy = d.xy + (size_t)c * d.n_cells;
  int m = w.order[t];
  HP_FIX(d.err, m, d.n_cells, BS_WM_CELL);
  const double mw = (double)d.w[m], mh = (double)d.h[m];
  const double bx = wm_step(d.die_xl, d.die_xh, d.nx), by = wm_step(d.die_yl, d.die_yh, d.ny);
  if ((int)blockIdx.x >= lines) {
    const int o = (blockIdx.x - lines) * kWmLines + threadIdx.x;
    if (o >= w.n_fixed + t) return;
    int oc = w.obst[o];
    HP_FIX(d.err, oc, d.n_cells, BS_WM_CELL);
    const double ow = (double)d.w[oc], oh = (double)d.h[oc];
    pdl_wait();
    const float2 p = xy[oc];
    const int2 rx = blocked_range(d.die_xl, bx, d.nx, mw, (double)p.x, __dadd_rn((double)p.x, ow));
    const int2 ry = blocked_range(d.die_yl, by, d.ny, mh, (double)p.y, __dadd_rn((double)p.y, oh));
    w.range[(size_t)blockIdx.y * (w.n_fixed + w.n_macros) + o] = make_int4(rx.x, rx.y, ry.x, ry.y);
    return;
  }
  const int q = blockIdx.x * kWmLines + threadIdx.x;
  const bool isx = q < d.nx, live = q < d.nx + d.ny;
  const int i = isx ? q : q - d.nx;
  const double X = isx ? wm_corner_b(d.die_xl, bx, i) : wm_corner_b(d.die_yl, by, i);
  const int a = isx ? 0 : 2;
  const int s0 = w.mptr[t], nn = w.mptr[t + 1] - s0;
  double acc = 0.0;
  bool waited = false;
  for (int n0 = 0; n0 < nn; n0 += kWmLines) {
    __syncthreads();
    const int s = s0 + n0 + threadIdx.x;
    const bool mine = n0 + (int)threadIdx.x < nn;
    // box: other pins' extent {o-x, o+x, o-y, o+y}, then the macro's own pin
    // offsets {d-x, d+x, d-y, d+y}
    float4 own;
    int shared = -1;
    if (mine) {
      int e = w.mnet[s];
      HP_FIX(d.err, e, d.n_nets, BS_WM_NET);
      sw[threadIdx.x] = d.net_w ? (double)d.net_w[e] : 1.0;
      own = w.own[s];
      shared = w.slot[s];
    }
    if (!waited) pdl_wait();
    waited = true;
    if (mine) {
      Extent o = load_extent(w.sbox + (size_t)blockIdx.y * w.n_entries * 4, s);
      if (shared >= 0)  // the net's macros that have moved
        extent_add(o, load_extent(w.moved + (size_t)blockIdx.y * w.n_shared * 4, shared));
#pragma unroll
      for (int k = 0; k < 4; ++k) box[k][threadIdx.x] = o.v[k];
      box[4][threadIdx.x] = (double)own.x; box[5][threadIdx.x] = (double)own.y;
      box[6][threadIdx.x] = (double)own.z; box[7][threadIdx.x] = (double)own.w;
    }
    __syncthreads();
    if (live) {
      const int cnt = min(kWmLines, nn - n0);
      for (int k = 0; k < cnt; ++k) {
        const double hi = fmax(box[a + 1][k], __dadd_rn(X, box[a + 5][k]));
        const double lo = fmin(box[a][k], __dadd_rn(X, box[a + 4][k]));
        acc = __dadd_rn(acc, __dmul_rn(sw[k], __dsub_rn(hi, lo)));
      }
    }
  }
  if (!waited) pdl_wait();
  if (live) {
    const float2 pm = xy[m];
    const bool in = isx ? __dadd_rn(X, mw) <= d.die_xh : __dadd_rn(X, mh) <= d.die_yh;
    const double dist = in ? fabs(__dsub_rn(X, isx ? (double)pm.x : (double)pm.y)) : -1.0;
    const size_t o = (size_t)blockIdx.y * (d.nx + d.ny) + q;
    w.f[o] = acc;
    w.dist[o] = dist;
  }
}

// Macro t: row j = blockIdx.x of the candidates.
__global__ void __launch_bounds__(kWmThreads) k_wm_select(Dev d, WmDev w, int t, int copy0) {
  __shared__ unsigned int blocked[8192 / 32];
  __shared__ int flag;
  __shared__ float2 place;
  int m = w.order[t];
  HP_FIX(d.err, m, d.n_cells, BS_WM_CELL);
  const int s0 = w.mptr[t], s1 = w.more[t] ? w.mptr[t + 1] : s0;
  pdl_wait();
  const int c = copy0 + blockIdx.y, j = blockIdx.x, nob = w.n_fixed + t;
  const double *f = w.f + (size_t)blockIdx.y * (d.nx + d.ny);
  const double *dist = w.dist + (size_t)blockIdx.y * (d.nx + d.ny);
  const int4 *range = w.range + (size_t)blockIdx.y * (w.n_fixed + w.n_macros);
  Best best = no_best();
  const double fy = f[d.nx + j], dy = dist[d.nx + j];
  if (dy >= 0.0) {  // (the whole block)
    const int words = (d.nx + 31) / 32;
    for (int i = threadIdx.x; i < words; i += kWmThreads) blocked[i] = 0u;
    __syncthreads();
    for (int o = threadIdx.x; o < nob; o += kWmThreads) {
      const int4 r = range[o];  // columns [x, y], rows [z, w]
      if (j < r.z || j > r.w) continue;
      const int lo = max(r.x, 0), hi = min(r.y, d.nx - 1);
      for (int k = lo >> 5; k <= hi >> 5 && lo <= hi; ++k) {
        const unsigned int from = k == lo >> 5 ? 0xffffffffu << (lo & 31) : 0xffffffffu;
        const unsigned int to = k == hi >> 5 ? 0xffffffffu >> (31 - (hi & 31)) : 0xffffffffu;
        atomicOr(&blocked[k], from & to);
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < d.nx; i += kWmThreads) {
      if (blocked[i >> 5] >> (i & 31) & 1u) continue;
      const double dx = dist[i];
      if (dx < 0.0) continue;
      const unsigned long long obj = ordered(__dadd_rn(f[i], fy));
      if (obj > best.obj) continue;
      const Best v{obj, ordered(__dadd_rn(dx, dy)), j * d.nx + i};
      if (better(v, best)) best = v;
    }
  }
  best = block_best(best);
  if (threadIdx.x == 0) {
    const size_t k = (size_t)blockIdx.y * d.ny + j;
    w.bobj[k] = best.obj;
    w.bdist[k] = best.dist;
    w.bidx[k] = best.idx;
  }
  if (!arrive_last_t0(w.ctr + blockIdx.y, &flag)) return;
  best = no_best();
  for (int k = threadIdx.x; k < d.ny; k += kWmThreads) {
    const size_t s = (size_t)blockIdx.y * d.ny + k;
    const Best v{__ldcg(w.bobj + s), __ldcg(w.bdist + s), __ldcg(w.bidx + s)};
    if (better(v, best)) best = v;
  }
  best = block_best(best);
  if (threadIdx.x == 0) {
    w.ctr[blockIdx.y] = 0u;
    float2 *at = d.xy + (size_t)c * d.n_cells + m;
    float2 p = *at;
    if (best.idx != kNoIdx && HP_IN(d.err, best.idx, d.nx * d.ny, BS_WM_BIN)) {
      const int jj = best.idx / d.nx, i = best.idx - jj * d.nx;
      p = make_float2((float)wm_corner(d.die_xl, d.die_xh, d.nx, i),
                      (float)wm_corner(d.die_yl, d.die_yh, d.ny, jj));
      *at = p;
    }
    place = p;
  }
  if (s1 == s0) return;  // no later macro shares a net with this one
  __syncthreads();
  for (int s = s0 + threadIdx.x; s < s1; s += kWmThreads) {
    const int k = w.slot[s];
    if (k < 0) continue;
    const size_t at = (size_t)blockIdx.y * w.n_shared + k;
    Extent e = load_extent(w.moved, at);
    extent_add(e, extent_at(place, w.own[s]));
    store_extent(w.moved, at, e);
  }
}

}  // namespace

void launch_wiremask(const Dev &d, const WmDev &w, int copy0, int ncopy, cudaStream_t st) {
  const int lines = (d.nx + d.ny + kWmLines - 1) / kWmLines;
  for (int c = copy0; c < copy0 + ncopy; c += w.group) {
    const int k = std::min(w.group, copy0 + ncopy - c);
    if (w.n_dnets > 0) k_wm_static<<<dim3(w.n_dnets, k), kWmNetThreads, 0, st>>>(d, w, c);
    for (int t = 0; t < w.n_macros; ++t) {
      const int ranges = (w.n_fixed + t + kWmLines - 1) / kWmLines;
      launch_pdl(k_wm_mask, dim3(lines + ranges, k), dim3(kWmLines), 0, st, d, w, t, c, lines);
      launch_pdl(k_wm_select, dim3(d.ny, k), dim3(kWmThreads), 0, st, d, w, t, c);
    }
  }
}

}  // namespace hp
