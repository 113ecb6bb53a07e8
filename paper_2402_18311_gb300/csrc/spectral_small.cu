// Spectral Poisson solve of a small grid (at most 4096 bins, FP32 path, few
// copies: choose_solve in api.cu) in one
// kernel: the density finish and the four transforms of spectral.cu by one
// thread-block cluster per copy.
//
// What bounds it: launches and latency.  A 64 x 64 grid is 1 MFLOP per
// transform; as a chain of five kernels (finish and four GEMMs of one 64 x 64
// tile, which is one block) each step took 7 to 10 us with 8 of the chip's
// 4864 warps busy.  Here eight blocks of 512 threads hold one output element
// per thread and stage and meet at a cluster barrier (hundreds of ns) where
// the chain had a kernel boundary; every block forms the whole density for
// itself, so the first transform waits for nobody.  One iteration of the
// 1k-cell design on 64 x 64 bins: 64.0 -> 40.3 us.  The line at 4096 bins and
// sides of 128: there a stage is one element per thread and its operands fit
// in shared memory.  (The fast transforms take 37.7 us on 64 x 64 bins but no
// side that is not a power of two, and round differently; here the results of
// every small grid stay what the GEMMs gave.)
//
// Each element is the same chain of fused multiply-adds over ascending k as
// in the tiled GEMM of spectral.cu, and the weights are its expressions, so
// both give the same bits.
#include "common.cuh"
#include "density_finish.cuh"
#include "internal.cuh"

namespace hp {

namespace {

constexpr int kSmallBlocks = 8;  // blocks of the cluster
constexpr int kSmallNT = 512;
constexpr int kSmallBins = kSmallBlocks * kSmallNT;
constexpr int kSmallSide = 128;
// a B operand: `rows` rows of `K` floats, 4 floats of padding each
constexpr int kSmallB = kSmallBins + 4 * kSmallSide;

// Shared memory: two B operands, then the block's rows of the four stages'
// transform matrices (six with both fields): side^2 / 8 floats each.
inline int small_smem(int nx, int ny) {
  return (int)sizeof(float) * (2 * kSmallB + 3 * (nx * nx + ny * ny) / kSmallBlocks);
}

__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// B operand written by the cluster (hence from L2) into shared memory.
__device__ __forceinline__ void load_b(float *sb, const float *src, int rows, int K) {
  const int q = K >> 2;
  for (int i = threadIdx.x; i < rows * q; i += kSmallNT) {
    const int r = i / q, k = i - r * q;
    *reinterpret_cast<float4 *>(sb + r * (K + 4) + 4 * k) =
        __ldcg(reinterpret_cast<const float4 *>(src) + i);
  }
}

// n floats of a transform matrix into shared memory (n a multiple of 4).
__device__ __forceinline__ void load_a(float *sa, const float *src, int n) {
  for (int i = threadIdx.x; i < (n >> 2); i += kSmallNT)
    reinterpret_cast<float4 *>(sa)[i] = __ldg(reinterpret_cast<const float4 *>(src) + i);
}

// sum_k A[k] B[k], ascending k
__device__ __forceinline__ float dot(const float *A, const float *sb, int K) {
  float acc = 0.f;
#pragma unroll 4
  for (int k = 0; k < K; k += 4) {
    const float4 a = *reinterpret_cast<const float4 *>(A + k);
    const float4 b = *reinterpret_cast<const float4 *>(sb + k);
    acc = fmaf(a.x, b.x, acc);
    acc = fmaf(a.y, b.y, acc);
    acc = fmaf(a.z, b.z, acc);
    acc = fmaf(a.w, b.w, acc);
  }
  return acc;
}

// PSI: planes Ex, Ey and psi (place_eval_field) instead of (Ex, Ey) pairs.
template <bool STRETCH, bool PSI>
__global__ void __cluster_dims__(kSmallBlocks, 1, 1) __launch_bounds__(kSmallNT)
    k_solve_small(Dev d, int copy0, int mode) {
  extern __shared__ __align__(16) float dyn_small[];
  __shared__ FinishShared fs;
  float *const sb[2] = {dyn_small, dyn_small + kSmallB};
  // a stage's outputs run along its B operand's rows, so this block has side /
  // 8 rows of each transform matrix; they are constants of the handle, loaded
  // before the wait for the scatter
  const int na = d.ny * d.ny / kSmallBlocks, nb = d.nx * d.nx / kSmallBlocks;
  float *const a1 = sb[1] + kSmallB, *const a2 = a1 + na, *const a3 = a2 + nb, *const a3s = a3 + na,
        *const a4s = a3s + na, *const a4 = a4s + nb;
  load_a(a1, d.Cn + blockIdx.x * na, na);
  load_a(a2, d.Cm + blockIdx.x * nb, nb);
  load_a(a3, d.CTn + blockIdx.x * na, na);
  load_a(a3s, d.STn + blockIdx.x * na, na);
  load_a(a4s, d.STm + blockIdx.x * nb, nb);
  load_a(a4, d.CTm + blockIdx.x * nb, nb);
  pdl_wait();
  const int c = copy0 + blockIdx.y;
  if (mode == FIN_ITER && d.cs[c].stopped) return;  // the whole cluster
  const int nx = d.nx, ny = d.ny, G = d.G, per = G / kSmallBlocks;  // G: a multiple of 256
  float *T = d.T + (size_t)c * 3 * G, *SB = d.SB + (size_t)c * 3 * G, *E = d.E + (size_t)c * 3 * G;
  // the density of every bin as the first B operand (rows x, K = ny), the
  // sums over this block's share of the bins
  BinSums sums;
  const FinishArgs fa = finish_args(d, c);
  const int share = per >> 1, s0 = blockIdx.x * share;  // bin pairs
  for (int b2 = threadIdx.x; b2 < (G >> 1); b2 += kSmallNT) {
    BinSums one;
    const float2 r = finish_pair<STRETCH>(d, fa, b2, one);
    if (b2 >= s0 && b2 < s0 + share) {
      sums.acc += one.acc;
      sums.m_over += one.m_over;
      sums.n_over += one.n_over;
      sums.q2 += one.q2;
    }
    const int x = 2 * b2 / ny, y = 2 * b2 - x * ny;
    *reinterpret_cast<float2 *>(&sb[0][x * (ny + 4) + y]) = r;
  }
  __syncthreads();
  const int i = blockIdx.x * per + threadIdx.x;  // this thread's output element
  const int ry = blockIdx.x * (ny / kSmallBlocks), rx = blockIdx.x * (nx / kSmallBlocks);
  const bool own = threadIdx.x < per;
  // 1: T[v][x] = sum_y Cn[v][y] rho[x][y]
  if (own) {
    const int v = i / nx, x = i - v * nx;
    T[i] = dot(a1 + (v - ry) * ny, &sb[0][x * (ny + 4)], ny);
  }
  finish_partial<kSmallNT>(d, c, sums, &fs);
  cluster_arrive();
  cluster_wait();
  // every block has read the map: zero it for the next pass
  if (own) {
    unsigned long long *M = d.M + (size_t)c * d.Gm;
    M[i] = 0ull;
    if (d.n_fill) M[G + i] = 0ull;
  }
  // 2: a[u][v] = c_u c_v sum_x Cm[u][x] T[v][x], and the fields' coefficients
  load_b(sb[0], T, ny, nx);
  __syncthreads();
  if (own) {
    const int u = i / ny, v = i - u * ny;
    const float a = dot(a2 + (u - rx) * nx, &sb[0][v * (nx + 4)], nx) * d.cu[u] * d.cv[v];
    const float wu = d.wu[u], wv = d.wv[v];
    const float den = wu * wu + wv * wv;
    const float inv = i == 0 ? 0.f : 1.f / den;
    SB[i] = a * wu * inv;
    SB[G + i] = a * wv * inv;
    if constexpr (PSI) SB[2 * G + i] = a * inv;
  }
  cluster_arrive();
  // the copy's overflow, while the others arrive
  if (blockIdx.x == 0 && threadIdx.x < 32) {
    finish_total(d, c, mode, kSmallBlocks);
    __syncwarp();
  }
  cluster_wait();
  // 3: T_w[y][u] = sum_v A_w[y][v] B_w[u][v], A = (C_N^T, S_N, C_N^T)
  load_b(sb[0], SB, nx, ny);
  load_b(sb[1], SB + G, nx, ny);
  __syncthreads();
  if (own) {
    const int y = i / nx, u = i - y * nx;
    T[i] = dot(a3 + (y - ry) * ny, &sb[0][u * (ny + 4)], ny);
    T[G + i] = dot(a3s + (y - ry) * ny, &sb[1][u * (ny + 4)], ny);
  }
  if constexpr (PSI) {
    __syncthreads();
    load_b(sb[0], SB + 2 * G, nx, ny);
    __syncthreads();
    if (own) {
      const int y = i / nx, u = i - y * nx;
      T[2 * G + i] = dot(a3 + (y - ry) * ny, &sb[0][u * (ny + 4)], ny);
    }
  }
  cluster_arrive();
  cluster_wait();
  // 4: E_w[x][y] = sum_u A_w[x][u] T_w[y][u], A = (S_M, C_M^T, C_M^T)
  load_b(sb[0], T, ny, nx);
  load_b(sb[1], T + G, ny, nx);
  __syncthreads();
  if (own) {
    const int x = i / ny, y = i - x * ny;
    const float ex = dot(a4s + (x - rx) * nx, &sb[0][y * (nx + 4)], nx);
    const float ey = dot(a4 + (x - rx) * nx, &sb[1][y * (nx + 4)], nx);
    if constexpr (PSI) {
      E[i] = ex;
      E[G + i] = ey;
    } else {
      reinterpret_cast<float2 *>(E)[i] = make_float2(ex, ey);
    }
  }
  if constexpr (PSI) {
    __syncthreads();
    load_b(sb[0], T + 2 * G, ny, nx);
    __syncthreads();
    if (own) {
      const int x = i / ny, y = i - x * ny;
      E[2 * G + i] = dot(a4 + (x - rx) * nx, &sb[0][y * (nx + 4)], nx);
    }
  }
}

}  // namespace

bool small_grid(int nx, int ny) {
  return nx * ny <= kSmallBins && nx <= kSmallSide && ny <= kSmallSide;
}

// The kernels' dynamic shared memory, for every grid that they take.
int small_prepare() {
  const int most = small_smem(kSmallSide, kSmallBins / kSmallSide);
  cudaError_t e = cudaSuccess;
  auto set = [&](auto *k) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  };
  set(k_solve_small<false, false>);
  set(k_solve_small<false, true>);
  set(k_solve_small<true, false>);
  set(k_solve_small<true, true>);
  return e == cudaSuccess ? 0 : -1;
}

void launch_solve_small(const Dev &d, int copy0, int ncopy, int mode, int with_psi, cudaStream_t st) {
  const dim3 grid(kSmallBlocks, ncopy), block(kSmallNT);
  const size_t smem = small_smem(d.nx, d.ny);
  if (d.Ms && with_psi)
    launch_pdl(k_solve_small<true, true>, grid, block, smem, st, d, copy0, mode);
  else if (d.Ms)
    launch_pdl(k_solve_small<true, false>, grid, block, smem, st, d, copy0, mode);
  else if (with_psi)
    launch_pdl(k_solve_small<false, true>, grid, block, smem, st, d, copy0, mode);
  else
    launch_pdl(k_solve_small<false, false>, grid, block, smem, st, d, copy0, mode);
}

}  // namespace hp
