// Spectral Poisson solve by fast transforms, for grids whose sides are powers
// of two from 64 to 4096: the sums of spectral.cu in FP32, O(log n) instead
// of O(n) operations per bin and direction, in three kernels:
//   rows     per row x, along y: the density finish of its bins (overflow and
//            bin density, density.cu) and T[x][v] = sum_y rho_xy c_v(y)
//   columns  per column v, along x: A = sum_x T c_u(x), the coefficients
//            B = c_u c_v A / (w_u^2 + w_v^2), and back along x:
//            P[x][v] = sum_u w_u B s_u(x), Q[x][v] = sum_u B c_u(x)
//   fields   per row x, along y: Ex = sum_v P c_v(y), Ey = sum_v w_v Q s_v(y)
//            (and psi = sum_v Q c_v(y))
// with c_k(i) = cos(pi k (i + 1/2) / N), s_k(i) = sin(pi k (i + 1/2) / N).
//
// A cosine transform of N samples is an N-point FFT of them in the order
// "even ones upwards, odd ones downwards" (Makhoul, IEEE Trans. ASSP 28,
// 1980): with V that FFT, W_k = exp(-i pi k / 2N) V_k holds X_k = Re W_k and
// X_{N-k} = -Im W_k; backwards, V_k = exp(i pi k / 2N) (C_k - i C_{N-k}) / 2.
// A sine sum is (-1)^i times the cosine sum of the reversed coefficients,
// s_k(i) = (-1)^i c_{N-k}(i).  Two real sequences share one complex FFT: two
// rows, two columns (P of both and Q of both on the way back), Ex beside Ey.
//
// What bounds it: latency.  The three kernels move about 44 bytes per bin, in
// L2, and every FFT waits on its 3 to 4 exchanges through shared memory.  So
// each thread holds 8 points (radix 8 and 4: few exchanges), the density
// finish shares the first kernel (no density map in memory, one launch less),
// both inverse transforms along x stay in the kernel that has the column, and
// the field leaves as (Ex, Ey) pairs, which is what the cell gradient
// gathers.  Against four dependent GEMMs on the tensor cores behind a density
// finish of its own (120 times the arithmetic), one iteration: 100 -> 76 us at
// 210k cells and 512^2 bins, 321 -> 269 at 2.1M and 1024^2; the field's error
// against FP64 7e-6 -> 2e-7.  Sides below 64 are the small solve's; above 4096
// one FFT no longer fits a block's threads at 8 points each.
#include "common.cuh"
#include "density_finish.cuh"
#include "internal.cuh"
#include "spectral_fft.cuh"

namespace hp {

using namespace fft;

namespace {

// FFTs per block of the row kernels (N points, N / 8 threads each): 256
// threads, fewer for the short rows of small grids (more blocks).
constexpr int row_ffts(int logn) { return logn >= 11 ? 1 : (logn >= 9 ? 256 / (1 << (logn - 3)) : (logn >= 7 ? 4 : 8)); }

// W_k of the two real sequences packed in the FFT Z: Z_k and Z_{N-k}, and
// c = exp(-i pi k / 2N).
__device__ __forceinline__ void dct_pair(float2 z, float2 zr, float2 c, float2 &wa, float2 &wb) {
  const float2 va = make_float2(0.5f * (z.x + zr.x), 0.5f * (z.y - zr.y));
  const float2 vb = make_float2(0.5f * (z.y + zr.y), 0.5f * (zr.x - z.x));
  wa = cmul(c, va);
  wb = cmul(c, vb);
}

// exp(i pi k / 2N) (a + i b) / 2 with c = exp(-i pi k / 2N)
__device__ __forceinline__ float2 half_turn(float2 c, float a, float b) {
  return make_float2(0.5f * fmaf(a, c.x, b * c.y), 0.5f * fmaf(b, c.x, -a * c.y));
}

template <int LOGN, bool STRETCH>
__global__ void __launch_bounds__(row_ffts(LOGN) * (1 << (LOGN - 3)))
    k_fft_rows(Dev d, int copy0, int mode) {  // (its overflow partials: k_fft_columns)
  constexpr int N = 1 << LOGN, T = N / 8, F = row_ffts(LOGN), NT = F * T;
  __shared__ float2 sm[F * padded(N)];
  __shared__ FinishShared fs;
  pdl_wait();
  const int c = copy0 + blockIdx.y;
  if (mode == FIN_ITER) {
    const int stopped = d.cs[c].stopped;
    // for the columns, beside whose blocks the stop test writes it
    if (blockIdx.x == 0 && threadIdx.x == 0) d.ctr[(size_t)c * C_COUNT + C_SKIP] = stopped;
    if (stopped) return;
  }
  const int f = threadIdx.x / T, t = threadIdx.x % T;
  const int xa = 2 * (blockIdx.x * F + f);  // rows xa and xa + 1
  float2 *s = sm + f * padded(N);
  BinSums sums;
  const FinishArgs fa = finish_args(d, c);
  // each thread's bin pairs of both rows, then the rows, less the mean density
  // (the solve drops the constant mode, and without it the transforms' rounding
  // errors are relative to what varies), as one complex sequence in DCT order
  {
    float2 ra[4], rb[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int q = t + m * T;  // bins 2q and 2q + 1
      ra[m] = finish_pair<STRETCH>(d, fa, xa * (N / 2) + q, sums);
      rb[m] = finish_pair<STRETCH>(d, fa, (xa + 1) * (N / 2) + q, sums);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int q = t + m * T;
      s[pad(q)] = make_float2(ra[m].x - d.rho_mean, rb[m].x - d.rho_mean);
      s[pad(N - 1 - q)] = make_float2(ra[m].y - d.rho_mean, rb[m].y - d.rho_mean);
    }
  }
  // the map is zero again for the next pass
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int q = t + m * T;
    clear_pair(d, c, xa * (N / 2) + q);
    clear_pair(d, c, (xa + 1) * (N / 2) + q);
  }
  __syncthreads();
  float2 v[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) v[m] = s[pad(t + m * T)];
  __syncthreads();
  transform<LOGN, false>(v, t, s, d.fft_wy);
#pragma unroll
  for (int m = 0; m < 8; ++m) s[pad(t + m * T)] = v[m];
  __syncthreads();
  float *Ta = d.T + (size_t)c * 3 * d.G + (size_t)xa * N, *Tb = Ta + N;
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int k = t + m * T;
    float2 wa, wb;
    dct_pair(v[m], s[pad((N - k) & (N - 1))], __ldg(d.fft_cy + k), wa, wb);
    Ta[k] = wa.x;
    Tb[k] = wb.x;
  }
  finish_partial<NT>(d, c, sums, &fs);
}

// CP column pairs per block, M / 8 threads each.  One more block per copy
// reduces the overflow of the row kernel's partials: beside the transforms
// instead of at the end of that kernel, whose last block held the next one up
// for 4 us.  The stop test there may end the copy, so the other blocks do not read
// its flag but what the row kernel found.
template <int LOGM, int CP>
__global__ void __launch_bounds__(CP * (1 << (LOGM - 3)))
    k_fft_columns(Dev d, int copy0, int mode, int partials) {
  constexpr int M = 1 << LOGM, T = M / 8, NT = CP * T;
  __shared__ float2 sm[CP * padded(M)];
  pdl_wait();
  const int c = copy0 + blockIdx.y;
  if (mode == FIN_ITER && d.ctr[(size_t)c * C_COUNT + C_SKIP]) return;
  if (blockIdx.x == gridDim.x - 1) {
    if (threadIdx.x < 32) finish_total(d, c, mode, partials);
    return;
  }
  const int ny = d.ny, v0 = blockIdx.x * 2 * CP;
  const float *Tc = d.T + (size_t)c * 3 * d.G + v0;
  {
    float2 r[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int i = threadIdx.x + m * NT, p = i % CP, x = i / CP;
      r[m] = *reinterpret_cast<const float2 *>(Tc + (size_t)x * ny + 2 * p);
    }
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int i = threadIdx.x + m * NT, p = i % CP, x = i / CP;
      sm[p * padded(M) + pad(dct_order<M>(x))] = r[m];
    }
  }
  __syncthreads();
  const int p = threadIdx.x / T, t = threadIdx.x % T;
  float2 *s = sm + p * padded(M);
  float2 z[8], w[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) z[m] = s[pad(t + m * T)];
  __syncthreads();
  transform<LOGM, false>(z, t, s, d.fft_wx);
#pragma unroll
  for (int m = 0; m < 8; ++m) s[pad(t + m * T)] = z[m];
  __syncthreads();
  // per frequency k of both columns: the coefficients at k and M - k, and the
  // spectra for the way back, P of both columns in one FFT and Q of both in the
  // other (a rounding error of an FFT is relative to the larger of its two
  // sequences: P and Q = P / w_u differ by the grid's side, neighbouring
  // columns hardly)
  const int va = v0 + 2 * p;
  const float wva = d.wv[va], wvb = d.wv[va + 1], cva = d.cv[va], cvb = d.cv[va + 1];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int k = t + m * T, kr = (M - k) & (M - 1);
    const float2 e = __ldg(d.fft_cx + k);
    float2 xa, xb;
    dct_pair(z[m], s[pad(kr)], e, xa, xb);
    const float wu = d.wu[k], wr = d.wu[kr], cu = d.cu[k], cr = d.cu[kr];
    const float wu2 = wu * wu, wr2 = wr * wr;
    const float da = fmaf(wva, wva, wu2), ra = fmaf(wva, wva, wr2);
    const float db = fmaf(wvb, wvb, wu2), rb = fmaf(wvb, wvb, wr2);
    // B at k and at M - k; the constant mode (0, 0) is dropped, and there is
    // no frequency M (k = 0)
    const float ba = (k == 0 && va == 0) ? 0.f : xa.x * cu * cva / da;
    const float bb = xb.x * cu * cvb / db;
    const float bar = k == 0 ? 0.f : -xa.y * cr * cva / ra;
    const float bbr = k == 0 ? 0.f : -xb.y * cr * cvb / rb;
    // P: reversed coefficients of w_u B (s_u = +- c_{M-u}); Q: B
    const float pa = wu * ba, par = wr * bar, pb = wu * bb, pbr = wr * bbr;
    if (k == 0) {
      z[m] = make_float2(0.f, 0.f);
      w[m] = make_float2(ba, bb);
    } else {
      // P: (Pa_{M-k} - i Pa_k) + i (Pb_{M-k} - i Pb_k); Q: (Ba_k - i Ba_{M-k}) + i (Bb_k - i Bb_{M-k})
      z[m] = half_turn(e, par + pb, pbr - pa);
      w[m] = half_turn(e, ba + bbr, bb - bar);
    }
  }
  __syncthreads();
  transform<LOGM, true>(z, t, s, d.fft_wx);
  transform<LOGM, true>(w, t, s, d.fft_wx);
  // (16-byte stores of every second row; collected in shared memory first, so
  // that a row's columns leave together, the two kernels take 37 us instead of
  // 32 at 1024^2 bins)
  float4 *PQ = reinterpret_cast<float4 *>(d.SB + (size_t)c * 3 * d.G) + (va >> 1);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int x = dct_sample<M>(t + m * T);
    const bool odd = m >= 4;  // the second half of the order holds the odd samples
    PQ[(size_t)x * (ny >> 1)] =
        make_float4(odd ? -z[m].x : z[m].x, w[m].x, odd ? -z[m].y : z[m].y, w[m].y);
  }
}

// The field of row x.  PSI: planes Ex, Ey and psi (place_eval_field) instead
// of (Ex, Ey) pairs.
template <int LOGN, bool PSI>
__global__ void __launch_bounds__(row_ffts(LOGN) * (1 << (LOGN - 3)))
    k_fft_fields(Dev d, int copy0, int eval) {
  constexpr int N = 1 << LOGN, T = N / 8, F = row_ffts(LOGN);
  __shared__ float2 sm[F * padded(N)];
  pdl_wait();
  const int c = copy0 + blockIdx.y;
  if (!eval && d.cs[c].stopped) return;
  const int f = threadIdx.x / T, t = threadIdx.x % T;
  const int x = blockIdx.x * F + f;
  float2 *s = sm + f * padded(N);
  const float2 *PQ = reinterpret_cast<const float2 *>(d.SB + (size_t)c * 3 * d.G) + (size_t)x * N;
  float2 z[8];
  float q[8], qr[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int k = t + m * T, kr = (N - k) & (N - 1);
    const float2 a = PQ[k], b = PQ[kr];
    const float2 e = __ldg(d.fft_cy + k);
    const float r = d.wv[k] * a.y, rr = d.wv[kr] * b.y;
    // (P_k - i P_{N-k}) + i (R_{N-k} - i R_k), R = w_v Q
    z[m] = k == 0 ? make_float2(a.x, 0.f) : half_turn(e, a.x + r, rr - b.x);
    if constexpr (PSI) {
      q[m] = a.y;
      qr[m] = b.y;
    }
  }
  transform<LOGN, true>(z, t, s, d.fft_wy);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const bool odd = m >= 4;
    s[pad(dct_sample<N>(t + m * T))] = make_float2(z[m].x, odd ? -z[m].y : z[m].y);
  }
  __syncthreads();
  float *E = d.E + (size_t)c * 3 * d.G;
  if constexpr (!PSI) {
    float4 *out = reinterpret_cast<float4 *>(E) + (size_t)x * (N / 2);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int y = 2 * (t + m * T);
      const float2 a = s[pad(y)], b = s[pad(y + 1)];
      out[t + m * T] = make_float4(a.x, a.y, b.x, b.y);
    }
  } else {
    float *o = E + (size_t)x * N;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const float2 a = s[pad(t + m * T)];
      o[t + m * T] = a.x;
      o[d.G + t + m * T] = a.y;
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int k = t + m * T;
      const float2 e = __ldg(d.fft_cy + k);
      z[m] = k == 0 ? make_float2(q[m], 0.f) : half_turn(e, q[m], -qr[m]);
    }
    transform<LOGN, true>(z, t, s, d.fft_wy);
#pragma unroll
    for (int m = 0; m < 8; ++m) o[2 * (size_t)d.G + dct_sample<N>(t + m * T)] = z[m].x;
  }
}

int log2i(int n) {
  int l = 0;
  while ((1 << l) < n) ++l;
  return l;
}

template <int LOGN>
void rows(const Dev &d, int copy0, int ncopy, int mode, cudaStream_t st) {
  const dim3 grid(d.nx / 2 / row_ffts(LOGN), ncopy), block(row_ffts(LOGN) << (LOGN - 3));
  if (d.Ms)
    launch_pdl(k_fft_rows<LOGN, true>, grid, block, 0, st, d, copy0, mode);
  else
    launch_pdl(k_fft_rows<LOGN, false>, grid, block, 0, st, d, copy0, mode);
}

// Four pairs of columns per block (whole 32-byte sectors; fewer of the longest
// columns), half of that where it would leave SMs without a block.  A column's result does not depend on it.
template <int LOGM>
void columns(const Dev &d, int copy0, int ncopy, int mode, cudaStream_t st) {
  constexpr int MOST = LOGM >= 12 ? 1 : (LOGM == 11 ? 2 : 4);
  constexpr int HALF = MOST > 1 && LOGM > 6 ? MOST / 2 : MOST;  // (at least a warp)
  const int partials = d.nx / 2 / row_ffts(log2i(d.ny));
  if (d.ny / 2 / MOST * ncopy < d.sms)
    launch_pdl(k_fft_columns<LOGM, HALF>, dim3(d.ny / 2 / HALF + 1, ncopy), dim3(HALF << (LOGM - 3)), 0,
               st, d, copy0, mode, partials);
  else
    launch_pdl(k_fft_columns<LOGM, MOST>, dim3(d.ny / 2 / MOST + 1, ncopy), dim3(MOST << (LOGM - 3)), 0,
               st, d, copy0, mode, partials);
}

template <int LOGN>
void fields(const Dev &d, int copy0, int ncopy, int psi, int eval, cudaStream_t st) {
  const dim3 grid(d.nx / row_ffts(LOGN), ncopy), block(row_ffts(LOGN) << (LOGN - 3));
  if (psi)
    launch_pdl(k_fft_fields<LOGN, true>, grid, block, 0, st, d, copy0, eval);
  else
    launch_pdl(k_fft_fields<LOGN, false>, grid, block, 0, st, d, copy0, eval);
}

}  // namespace

bool fft_side(int n) { return n >= 64 && n <= 4096 && (n & (n - 1)) == 0; }

#define HP_BY_LENGTH(n, F, ...)          \
  switch (log2i(n)) {                    \
    case 6: F<6>(__VA_ARGS__); break;    \
    case 7: F<7>(__VA_ARGS__); break;    \
    case 8: F<8>(__VA_ARGS__); break;    \
    case 9: F<9>(__VA_ARGS__); break;    \
    case 10: F<10>(__VA_ARGS__); break;  \
    case 11: F<11>(__VA_ARGS__); break;  \
    default: F<12>(__VA_ARGS__); break;  \
  }

void launch_fft_rows(const Dev &d, int copy0, int ncopy, int mode, cudaStream_t st) {
  HP_BY_LENGTH(d.ny, rows, d, copy0, ncopy, mode, st)
}

void launch_fft_solve(const Dev &d, int copy0, int ncopy, int mode, int with_psi, cudaStream_t st) {
  HP_BY_LENGTH(d.nx, columns, d, copy0, ncopy, mode, st)
  HP_BY_LENGTH(d.ny, fields, d, copy0, ncopy, with_psi, mode != FIN_ITER, st)
}

}  // namespace hp
