// Shuffle and Shuffle (all) perturbations (the perturbation step of
// Algorithm 1; Section 4.2: a random fraction p of the macros, or of all the
// cells, exchange their locations among themselves).  Reading used by this
// library:
//   - every cell i draws r_i, the (i+1)-th output of SplitMix64 started from
//     `seed` (Steele, Lea and Flood, OOPSLA 2014), evaluated directly from
//     its counter: state = seed + (i+1) * 0x9E3779B97F4A7C15, then the mix;
//   - the k = floor(p n + 1/2) candidates with the smallest (r_i, i) are
//     selected; candidates are the movable macros (Shuffle) or all movable
//     cells (Shuffle (all));
//   - taking the selected cells in key order t_0, t_1, ... and in index order
//     s_0 < s_1 < ..., cell t_j receives the centre of cell s_j, clamped into
//     the die.  New corners are computed in FP64 and rounded once.
// Selection and permutation are integer work and bit-exact.
//
// The keys are the outputs of a bijective 64-bit mix, so they are distinct and
// spread evenly.  That makes a full sort unnecessary: the cells go to buckets
// by their key's leading bits (48 to 96 a bucket), only the buckets that start
// below rank k are kept, and a warp ranks each bucket in shared memory by
// counting the smaller keys.  The selected cells in index order are a bit mask
// and its prefix counts.  All copies of a batched handle go through the same
// launches (blockIdx.y).  What bounds it: the two passes of one L2 atomic per
// cell.  Against a bitonic sort of (key, index) pairs, one copy after another
// (324 passes at 210k cells), eight copies of 210k cells restored, shuffled at
// p = 0.5 and read back: 11.3 -> 0.46 ms (0.65 before the copies' positions were
// set in place).
#include "common.cuh"
#include "internal.cuh"

namespace hp {

__device__ __forceinline__ unsigned long long splitmix64_at(unsigned long long seed,
                                                            unsigned long long i) {
  unsigned long long z = seed + (i + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

namespace {

constexpr int kShufBucket = 96;   // most cells a bucket holds on average (at least half of it)
constexpr int kShufCap = 256;     // keys of a bucket kept in shared memory
constexpr int kShufTile = 256;    // mask words (of 32 cells) per tile of the prefix counts

// One copy's scratch.  Keys, indices and both orders live in the copy's
// gradient arrays, whose contents the reset behind the perturbation drops;
// the counters in d.sh.
struct Shuf {
  unsigned long long *key;  // [n_real] bucket by bucket
  unsigned int *id;         // [n_real]
  unsigned int *recv;       // [k] receivers in key order
  unsigned int *donor;      // [k] donors in index order
  float2 *moved;            // [k] the receivers' new corners
  unsigned int *start;      // [nb + 1] first rank of each bucket
  unsigned int *cursor;     // [nb] counts, then the next free slot
  unsigned int *mask;       // [words] selected cells
  unsigned int *tile;       // [tiles] selected cells per tile
};
__device__ __forceinline__ Shuf shuf(const Dev &d, int c) {
  const size_t cm = (size_t)c * d.n_mov;
  unsigned int *w = d.sh + (size_t)c * d.sh_stride;
  Shuf s;
  s.key = reinterpret_cast<unsigned long long *>(d.g[0] + cm);
  s.moved = d.g[1] + cm;
  s.id = reinterpret_cast<unsigned int *>(d.gwx + cm);
  s.recv = reinterpret_cast<unsigned int *>(d.gwy + cm);
  s.donor = reinterpret_cast<unsigned int *>(d.gdx + cm);
  s.cursor = w;
  s.mask = w + d.sh_nb;
  s.tile = s.mask + d.sh_words;
  s.start = s.tile + d.sh_tiles;
  return s;
}

__device__ __forceinline__ unsigned int bucket_of(const Dev &d, unsigned long long key) {
  return d.sh_lg ? (unsigned int)(key >> (64 - d.sh_lg)) : 0u;
}
__device__ __forceinline__ bool candidate(const Dev &d, int op, int i) {
  return op == PLACE_SHUFFLE_ALL || d.is_macro[i];
}

__global__ void __launch_bounds__(kThreads) k_shuf_count(Dev d, int copy0, int op, unsigned long long seed) {
  const Shuf s = shuf(d, copy0 + blockIdx.y);
  for (int i = blockIdx.x * kThreads + threadIdx.x; i < d.n_real; i += gridDim.x * kThreads)
    if (candidate(d, op, i)) atomicAdd(&s.cursor[bucket_of(d, splitmix64_at(seed + blockIdx.y, i))], 1u);
}

// Exclusive scan of one value per thread over a block of NT threads.
template <int NT>
__device__ __forceinline__ unsigned int block_scan(unsigned int v, unsigned int *sm) {
  unsigned int x = v;
  const int l = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int y = __shfl_up_sync(0xffffffffu, x, o);
    if (l >= o) x += y;
  }
  __syncthreads();
  if (l == 31) sm[w] = x;
  __syncthreads();
  if (w == 0) {
    unsigned int t = l < NT / 32 ? sm[l] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int y = __shfl_up_sync(0xffffffffu, t, o);
      if (l >= o) t += y;
    }
    if (l < NT / 32) sm[l] = t;
  }
  __syncthreads();
  return x - v + (w ? sm[w - 1] : 0u);
}

// Counts -> first ranks, one block per copy.
__global__ void __launch_bounds__(1024) k_shuf_scan(Dev d, int copy0) {
  __shared__ unsigned int sm[32];
  const Shuf s = shuf(d, copy0 + blockIdx.x);
  const int per = (d.sh_nb + 1023) / 1024, b0 = threadIdx.x * per;
  unsigned int sum = 0u;
  for (int b = b0; b < min(b0 + per, d.sh_nb); ++b) sum += s.cursor[b];
  unsigned int at = block_scan<1024>(sum, sm);
  for (int b = b0; b < min(b0 + per, d.sh_nb); ++b) {
    const unsigned int n = s.cursor[b];
    s.start[b] = at;
    s.cursor[b] = at;
    at += n;
  }
}

// The candidates of every bucket that starts below rank k (the buckets end
// below n_real, the number of cells).
__global__ void __launch_bounds__(kThreads)
    k_shuf_scatter(Dev d, int copy0, int op, unsigned long long seed, unsigned int k) {
  const Shuf s = shuf(d, copy0 + blockIdx.y);
  for (int i = blockIdx.x * kThreads + threadIdx.x; i < d.n_real; i += gridDim.x * kThreads) {
    if (!candidate(d, op, i)) continue;
    const unsigned long long key = splitmix64_at(seed + blockIdx.y, i);
    const unsigned int b = bucket_of(d, key);
    if (s.start[b] >= k) continue;
    unsigned int at = atomicAdd(&s.cursor[b], 1u);
    HP_FIX(d.err, at, d.n_real, BS_PERM);
    s.key[at] = key;
    s.id[at] = (unsigned int)i;
  }
}

// One warp per bucket: every cell's rank is its bucket's first rank plus the
// number of smaller (key, index) pairs in the bucket.
__global__ void __launch_bounds__(kThreads) k_shuf_rank(Dev d, int copy0, unsigned int k) {
  __shared__ unsigned long long sk[kThreads / 32][kShufCap];
  const Shuf s = shuf(d, copy0 + blockIdx.y);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  for (int b = blockIdx.x * (kThreads / 32) + w; b < d.sh_nb; b += gridDim.x * (kThreads / 32)) {
    const unsigned int at = s.start[b];
    if (at >= k) break;  // the starts ascend
    const int n = (int)(s.cursor[b] - at);
    const unsigned long long *keys = s.key + at;
    const unsigned int *ids = s.id + at;
    const bool staged = n <= kShufCap;
    if (staged) {
      for (int e = l; e < n; e += 32) sk[w][e] = keys[e];
      __syncwarp();
    }
    for (int e = l; e < n; e += 32) {
      const unsigned long long key = keys[e];
      const unsigned int id = ids[e];
      unsigned int r = 0u;
      if (staged) {
#pragma unroll 8
        for (int f = 0; f < n; ++f) r += sk[w][f] < key ? 1u : 0u;
      } else {  // (a bucket far above the mean: the same count from memory)
        for (int f = 0; f < n; ++f) r += keys[f] < key ? 1u : 0u;
      }
      r += at;
      if (r < k) {
        s.recv[r] = id;
        atomicOr(&s.mask[id >> 5], 1u << (id & 31));
      }
    }
    __syncwarp();
  }
}

__global__ void __launch_bounds__(kShufTile) k_shuf_tiles(Dev d, int copy0) {
  __shared__ unsigned int sm[32];
  const Shuf s = shuf(d, copy0 + blockIdx.y);
  const int word = blockIdx.x * kShufTile + threadIdx.x;
  const unsigned int v = word < d.sh_words ? __popc(s.mask[word]) : 0u;
  const unsigned int before = block_scan<kShufTile>(v, sm);
  if (threadIdx.x == kShufTile - 1) s.tile[blockIdx.x] = before + v;
}

// The selected cells in index order: a tile's first position is the sum of
// the tiles before it.
__global__ void __launch_bounds__(kShufTile) k_shuf_donors(Dev d, int copy0, unsigned int k) {
  __shared__ unsigned int sm[32];
  const Shuf s = shuf(d, copy0 + blockIdx.y);
  unsigned int sum = 0u;
  for (int t = threadIdx.x; t < (int)blockIdx.x; t += kShufTile) sum += s.tile[t];
  const unsigned int part = block_scan<kShufTile>(sum, sm);
  __shared__ unsigned int base;
  if (threadIdx.x == kShufTile - 1) base = part + sum;
  const int word = blockIdx.x * kShufTile + threadIdx.x;
  unsigned int m = word < d.sh_words ? s.mask[word] : 0u;
  unsigned int at = block_scan<kShufTile>(__popc(m), sm) + base;  // (its barriers publish base)
  while (m) {
    const int bit = __ffs(m) - 1;
    m &= m - 1;
    if (at < k) s.donor[at] = (unsigned int)(word * 32 + bit);
    ++at;
  }
}

__global__ void __launch_bounds__(kThreads) k_shuf_move(Dev d, int copy0, int k) {
  const int c = copy0 + blockIdx.y;
  const Shuf sh = shuf(d, c);
  const float2 *xy = d.xy + (size_t)c * d.n_cells;
  for (int j = blockIdx.x * kThreads + threadIdx.x; j < k; j += gridDim.x * kThreads) {
    int r = (int)sh.recv[j];   // receiver (key order)
    int s = (int)sh.donor[j];  // donor (index order)
    HP_FIX(d.err, r, d.n_real, BS_PERM);
    HP_FIX(d.err, s, d.n_real, BS_PERM);
    const float2 ps = xy[s];
    double cx = (double)ps.x + 0.5 * (double)d.w[s];
    double cy = (double)ps.y + 0.5 * (double)d.h[s];
    double nx = cx - 0.5 * (double)d.w[r];
    double ny = cy - 0.5 * (double)d.h[r];
    nx = fmax(d.die_xl, fmin(nx, d.die_xh - (double)d.w[r]));
    ny = fmax(d.die_yl, fmin(ny, d.die_yh - (double)d.h[r]));
    sh.moved[j] = make_float2((float)nx, (float)ny);
  }
}

__global__ void __launch_bounds__(kThreads) k_shuf_apply(Dev d, int copy0, int k) {
  const int c = copy0 + blockIdx.y;
  const Shuf sh = shuf(d, c);
  float2 *xy = d.xy + (size_t)c * d.n_cells;
  for (int j = blockIdx.x * kThreads + threadIdx.x; j < k; j += gridDim.x * kThreads) {
    const int r = (int)sh.recv[j];
    if (!HP_IN(d.err, r, d.n_real, BS_PERM)) continue;
    xy[r] = sh.moved[j];
  }
}

int grid_for(int n) {
  const int b = (n + kThreads - 1) / kThreads;
  return b < 1 ? 1 : (b > 4096 ? 4096 : b);
}

}  // namespace

// Buckets, mask words, tiles and 32-bit words of scratch per copy.
void shuffle_plan(Dev &d) {
  d.sh_lg = 0;
  while (((long long)kShufBucket << d.sh_lg) < d.n_real) ++d.sh_lg;
  d.sh_nb = 1 << d.sh_lg;
  d.sh_words = (d.n_real + 31) / 32;
  d.sh_tiles = (d.sh_words + kShufTile - 1) / kShufTile;
  d.sh_stride = 2 * d.sh_nb + 1 + d.sh_words + d.sh_tiles;
}

// Shuffle of copies [copy0, copy0 + ncopy): copy copy0 + y draws from seed + y;
// k (at least 1) of the candidates exchange places.
void launch_shuffle(const Dev &d, int copy0, int ncopy, int op, int k, uint64_t seed, cudaStream_t st) {
  const dim3 cells(grid_for(d.n_real), ncopy), sel(grid_for(k), ncopy);
  const unsigned long long sd = seed;
  // counts and mask
  cudaMemsetAsync(d.sh + (size_t)copy0 * d.sh_stride, 0, sizeof(unsigned int) * (size_t)d.sh_stride * ncopy, st);
  k_shuf_count<<<cells, kThreads, 0, st>>>(d, copy0, op, sd);
  k_shuf_scan<<<ncopy, 1024, 0, st>>>(d, copy0);
  k_shuf_scatter<<<cells, kThreads, 0, st>>>(d, copy0, op, sd, (unsigned int)k);
  k_shuf_rank<<<dim3(grid_for(d.sh_nb * 32), ncopy), kThreads, 0, st>>>(d, copy0, (unsigned int)k);
  k_shuf_tiles<<<dim3(d.sh_tiles, ncopy), kShufTile, 0, st>>>(d, copy0);
  k_shuf_donors<<<dim3(d.sh_tiles, ncopy), kShufTile, 0, st>>>(d, copy0, (unsigned int)k);
  k_shuf_move<<<sel, kThreads, 0, st>>>(d, copy0, k);
  k_shuf_apply<<<sel, kThreads, 0, st>>>(d, copy0, k);
}

}  // namespace hp
