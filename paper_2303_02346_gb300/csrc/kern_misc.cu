// Support kernels: counting sort of particles into grid cells, permutations
// between the library's particle order and the caller's, tool kinematics and
// its adjoint, losses and loss seeds.
#include <climits>

#include "common.cuh"
#include "kernels.h"
#include "perm.h"
#include "share.h"
#include "sum3.cuh"

namespace mpm {

constexpr int fX = 0, fV = 3, fC = 6, fF = 15;
static inline int blocks_for(long long n, int t) { return int((n + t - 1) / t); }

// ---------------------------------------------------------------------------
// counting sort by (scene, Morton order of the cell of the stencil origin).
// The Morton order keeps every 4^3 grid block contiguous (its cells are the
// code's lowest 6 bits) and orders the particles of a block by cell, so that
// a warp's consecutive particles occupy few, densely filled cells: the scatter
// then makes few reductions per particle.
// ---------------------------------------------------------------------------
// with_class: water particles before every other material (their keys offset
// by S x MB), so that the non-water particles occupy the index range [Nl, N).
//
// The bins are dense (one per cell, class and scene), the particles are not: a
// pass over all of them (clear, scan, add the tile sums) moved 5 x 134 MB for a
// 256^3 grid. Cells are therefore counted per 4^3 block as well (64
// consecutive codes), the scan over the bins runs over the block counts, and
// only the cells of blocks that hold particles are scanned, read and cleared
// again; every bin and block count is zero between sorts. A re-sort of 2M
// particles on 256^3: 366 -> 185 us so, 117 with sort_gather_kernel (mean of the 20
// sorts of a trajectory, kernel by kernel).
constexpr int kBlockBits = 6;  // cells of a 4^3 block: the lowest 6 bits of a code

// One atomic per warp and cell (and per warp and block): the lanes of equal
// cell take consecutive ranks.
__global__ void __launch_bounds__(256)
sort_key_kernel(Params P, const float* __restrict__ st, const uint32_t* __restrict__ tag,
                uint32_t* __restrict__ key, uint32_t* __restrict__ rank,
                uint32_t* __restrict__ bins, uint32_t* __restrict__ blk_cnt, int with_class) {
  constexpr unsigned kAll = 0xffffffffu;
  const int N = P.N;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool valid = p < N;
  uint32_t k = 0;
  if (valid) {
    int b[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float bf = base_floor(grid_coord(st[(fX + d) * N + p], P));
      bf = fminf(fmaxf(bf, 0.0f), float(P.n - 3));  // NaN -> 0
      b[d] = int(bf);
    }
    const uint32_t tg = tag[p];
    k = uint32_t(tag_scene(tg)) * uint32_t(P.MB) + morton3(uint32_t(b[0]), uint32_t(b[1]), uint32_t(b[2]));
    if (with_class && P.mat[tag_mat(tg)].kind != kLiquid) k += uint32_t(P.S) * uint32_t(P.MB);
    key[p] = k;
  }
  const unsigned vmask = __ballot_sync(kAll, valid);
  if (!valid) return;
  const unsigned same = __match_any_sync(vmask, k);
  const unsigned below = (1u << lane) - 1u;
  const int first = __ffs(same) - 1;
  uint32_t base = 0;
  if (lane == first) base = atomicAdd(&bins[k], uint32_t(__popc(same)));
  base = __shfl_sync(same, base, first);
  rank[p] = base + uint32_t(__popc(same & below));
  const unsigned blk = __match_any_sync(vmask, k >> kBlockBits);
  if ((blk & below) == 0u) atomicAdd(&blk_cnt[k >> kBlockBits], uint32_t(__popc(blk)));
}

constexpr int kScanThreads = 1024;
constexpr int kScanPer = 4;
constexpr int kScanTile = kScanThreads * kScanPer;

__device__ inline uint32_t block_exclusive_scan(uint32_t v, uint32_t* warp_sums, uint32_t& total) {
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[wid] = x;
  __syncthreads();
  if (wid == 0) {
    uint32_t s = warp_sums[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    warp_sums[lane] = s;
  }
  __syncthreads();
  uint32_t pre = (wid > 0 ? warp_sums[wid - 1] : 0u) + x - v;
  total = warp_sums[31];
  __syncthreads();
  return pre;
}

// exclusive scan of each tile of a into out; tile totals to sums
__global__ void __launch_bounds__(kScanThreads) scan_tiles_kernel(const uint32_t* __restrict__ a,
                                                                  uint32_t* __restrict__ out, long long n,
                                                                  uint32_t* __restrict__ sums) {
  __shared__ uint32_t ws[32];
  long long base = (long long)blockIdx.x * kScanTile + threadIdx.x * kScanPer;
  uint32_t v[kScanPer], s = 0;
#pragma unroll
  for (int i = 0; i < kScanPer; ++i) {
    v[i] = (base + i < n) ? a[base + i] : 0u;
    s += v[i];
  }
  uint32_t total;
  uint32_t pre = block_exclusive_scan(s, ws, total);
#pragma unroll
  for (int i = 0; i < kScanPer; ++i) {
    if (base + i < n) out[base + i] = pre;
    pre += v[i];
  }
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// single CTA: exclusive scan of the tile totals (any count, looped)
__global__ void __launch_bounds__(kScanThreads) scan_sums_kernel(uint32_t* __restrict__ sums, int n) {
  __shared__ uint32_t ws[32];
  uint32_t carry = 0;
  for (int off = 0; off < n; off += kScanThreads) {
    int i = off + threadIdx.x;
    uint32_t v = i < n ? sums[i] : 0u;
    uint32_t total;
    uint32_t pre = block_exclusive_scan(v, ws, total);
    if (i < n) sums[i] = pre + carry;
    carry += total;
  }
}

// The cells of the occupied blocks: exclusive scan of each block's 64 counts
// from the block's first slot, in place; blk_start receives that slot (the
// scanned tile's value plus the tiles' totals before it, sums; nullptr: there is
// one tile). A warp looks at 32 blocks and
// takes the occupied ones four at a time, 2 cells a lane, so that four blocks'
// loads are in flight.
__global__ void __launch_bounds__(256)
cell_scan_kernel(uint32_t* __restrict__ bins, const uint32_t* __restrict__ blk_cnt,
                 uint32_t* __restrict__ blk_start, const uint32_t* __restrict__ sums, int n_blk) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int b0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * 32;
  const int b = b0 + lane;
  const bool occ = b < n_blk && blk_cnt[b] != 0u;
  uint32_t start = 0;
  if (occ) {
    start = blk_start[b] + (sums ? sums[b / kScanTile] : 0u);
    blk_start[b] = start;
  }
  unsigned mask = __ballot_sync(kAll, occ);
  while (mask) {
    int j[4];
    uint2 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      j[u] = mask ? __ffs(mask) - 1 : -1;
      mask &= mask - 1u;
      if (j[u] >= 0) v[u] = reinterpret_cast<const uint2*>(bins)[(size_t)(b0 + j[u]) * 32 + lane];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (j[u] < 0) continue;
      const uint32_t s = v[u].x + v[u].y;
      uint32_t x = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kAll, x, o);
        if (lane >= o) x += y;
      }
      const uint32_t pre = __shfl_sync(kAll, start, j[u]) + x - s;
      reinterpret_cast<uint2*>(bins)[(size_t)(b0 + j[u]) * 32 + lane] = make_uint2(pre, pre + v[u].x);
    }
  }
}

// Zero again the bins of the occupied blocks and their counts.
__global__ void __launch_bounds__(256)
cell_clear_kernel(uint32_t* __restrict__ bins, uint32_t* __restrict__ blk_cnt, int n_blk) {
  const int lane = threadIdx.x & 31;
  const int b0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * 32;
  const int b = b0 + lane;
  const bool occ = b < n_blk && blk_cnt[b] != 0u;
  if (occ) blk_cnt[b] = 0u;
  for (unsigned mask = __ballot_sync(0xffffffffu, occ); mask; mask &= mask - 1u)
    reinterpret_cast<uint2*>(bins)[(size_t)(b0 + __ffs(mask) - 1) * 32 + lane] = make_uint2(0u, 0u);
}

// Each sorted slot's source particle.
__global__ void __launch_bounds__(256)
sort_index_kernel(int N, const uint32_t* __restrict__ key, const uint32_t* __restrict__ rank,
                  const uint32_t* __restrict__ offs, int* __restrict__ src) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < N) src[offs[key[p]] + rank[p]] = p;
}

// The state in sorted order, read through the slots' source particles, which
// pid_out holds at entry (each thread replaces its own by the particle's id).
// Bound by memory once eight fields are in flight a thread: only one word a
// particle is written out of order, and the reads of a nearly sorted state
// share their sectors. (Every field stored to its slot by its source's thread:
// 139 us for 2M water particles, 84 here and 9 for the index.)
__global__ void __launch_bounds__(256)
sort_gather_kernel(int N, const float* __restrict__ st_in, const uint32_t* __restrict__ tag_in,
                   const int* __restrict__ pid_in, float* __restrict__ st_out, uint32_t* __restrict__ tag_out,
                   int* pid_out, Params P) {
  constexpr int kBatch = 8;
  static_assert((fF + 1) % kBatch == 0 && kStateFields % kBatch == 0, "whole batches of fields");
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= N) return;
  const int p = pid_out[q];
  const uint32_t tg = tag_in[p];
  const int id = pid_in[p];
  const bool liquid = is_liquid(P.mat[tag_mat(tg)].kind);
  const int nf = liquid ? fF + 1 : kStateFields;  // a liquid carries only J = F[0]
  for (int f = 0; f < nf; f += kBatch) {
    float v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) v[u] = st_in[(long long)(f + u) * N + p];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) st_out[(long long)(f + u) * N + q] = v[u];
  }
  tag_out[q] = tg;
  pid_out[q] = id;
}

// Returns its launches.
static int bin_particles(const Params& P, const float* st, const uint32_t* tag, SortBuffers sb, int with_class,
                          cudaStream_t s) {
  const int N = P.N;
  if (N == 0) return 0;
  const int n_blk = int(((with_class ? 2LL : 1LL) * sb.n_bins) >> kBlockBits);
  sort_key_kernel<<<blocks_for(N, 256), 256, 0, s>>>(P, st, tag, sb.key, sb.rank, sb.bins, sb.blk_cnt, with_class);
  const int tiles = blocks_for(n_blk, kScanTile);
  scan_tiles_kernel<<<tiles, kScanThreads, 0, s>>>(sb.blk_cnt, sb.blk_start, n_blk, sb.tile_sums);
  if (tiles > 1) scan_sums_kernel<<<1, kScanThreads, 0, s>>>(sb.tile_sums, tiles);
  cell_scan_kernel<<<blocks_for(n_blk, 256), 256, 0, s>>>(sb.bins, sb.blk_cnt, sb.blk_start,
                                                          tiles > 1 ? sb.tile_sums : nullptr, n_blk);
  return tiles > 1 ? 4 : 3;
}

int launch_bin(const Params& P, const float* st, const uint32_t* tag, SortBuffers sb, cudaStream_t s) {
  return bin_particles(P, st, tag, sb, 0, s);
}

void launch_bin_clear(const Params& P, SortBuffers sb, cudaStream_t s) {
  if (P.N == 0) return;
  const int n_blk = int((2LL * sb.n_bins) >> kBlockBits);
  cell_clear_kernel<<<blocks_for(n_blk, 256), 256, 0, s>>>(sb.bins, sb.blk_cnt, n_blk);
}

// count of water particles (the material of each tag) into *out
__global__ void count_water_kernel(Params P, const uint32_t* __restrict__ tag, int* __restrict__ out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  const bool w = p < P.N && P.mat[tag_mat(tag[p])].kind == kLiquid;
  const int c = __syncthreads_count(w);  // one atomic per CTA on the one word (2M particles: 31 -> 8 us)
  if (threadIdx.x == 0 && c) atomicAdd(out, c);
}

void launch_count_water(const Params& P, const uint32_t* tag, int* out, cudaStream_t s) {
  cudaMemsetAsync(out, 0, sizeof(int), s);
  if (P.N > 0) count_water_kernel<<<blocks_for(P.N, 256), 256, 0, s>>>(P, tag, out);
}

int launch_sort(const Params& P, const float* st_in, const uint32_t* tag_in, const int* pid_in,
                 float* st_out, uint32_t* tag_out, int* pid_out, SortBuffers sb, cudaStream_t s) {
  const int N = P.N;
  if (N == 0) return 0;
  const int binned = bin_particles(P, st_in, tag_in, sb, 1, s);
  sort_index_kernel<<<blocks_for(N, 256), 256, 0, s>>>(N, sb.key, sb.rank, sb.bins, pid_out);
  sort_gather_kernel<<<blocks_for(N, 256), 256, 0, s>>>(N, st_in, tag_in, pid_in, st_out, tag_out, pid_out, P);
  launch_bin_clear(P, sb, s);
  return binned + 3;
}

// ---------------------------------------------------------------------------
// caller order <-> library order
// ---------------------------------------------------------------------------
// rows of `fields` values -> SoA: dst[c * stride + p] = src[p * fields + c]
__global__ void rows_to_fields_kernel(const float* __restrict__ src, float* __restrict__ dst, int N, int fields,
                                      int stride) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  for (int c = 0; c < fields; ++c) dst[(long long)c * stride + p] = src[(long long)p * fields + c];
}

__global__ void inverse_perm_kernel(const int* __restrict__ pid, int* __restrict__ inv, int N) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < N) inv[pid[p]] = p;
}

// dst[f][p'] = src[f][inv_from[pid_to[p']]]: writes coalesced, reads gathered
// (the two orders differ by one re-sort, so the reads stay mostly local). Both
// orders have the same first n_first particles, of which only the first
// f_first fields are copied (water carries J alone of F's nine).
__global__ void permute_state_kernel(const float* __restrict__ src, float* __restrict__ dst,
                                     const int* __restrict__ inv_from, const int* __restrict__ pid_to, int N,
                                     int n_first, int f_first, int fields) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= N) return;
  const long long p = inv_from[pid_to[q]];
  const int nf = q < n_first ? f_first : fields;
#pragma unroll 8
  for (int f = 0; f < nf; ++f) dst[(long long)f * N + q] = src[(long long)f * N + p];
}

void launch_permute_state(const float* src, float* dst, const int* pid_from, const int* pid_to, int* inv, int N,
                          int n_first, int f_first, int fields, cudaStream_t s) {
  if (N == 0) return;
  inverse_perm_kernel<<<blocks_for(N, 256), 256, 0, s>>>(pid_from, inv, N);
  permute_state_kernel<<<blocks_for(N, 256), 256, 0, s>>>(src, dst, inv, pid_to, N, n_first, f_first, fields);
}

void launch_rows_to_fields(const float* src, float* dst, int N, int fields, int stride, cudaStream_t s) {
  if (N == 0) return;
  rows_to_fields_kernel<<<blocks_for(N, 256), 256, 0, s>>>(src, dst, N, fields, stride);
}

__global__ void init_state_kernel(float* __restrict__ st, int N) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  for (int k = 0; k < 9; ++k) {
    st[(long long)(6 + k) * N + p] = 0.0f;                       // C = 0
    st[(long long)(15 + k) * N + p] = (k % 4 == 0) ? 1.0f : 0.0f;  // F = I
  }
}

void launch_init_state(float* st, int N, cudaStream_t s) {
  if (N == 0) return;
  init_state_kernel<<<blocks_for(N, 256), 256, 0, s>>>(st, N);
}

// x, v, C = 0, F = I and the material of particles [lo, lo + cnt) of the initial state
__global__ void init_particles_kernel(float* __restrict__ X0, uint32_t* __restrict__ tag0,
                                      const float* __restrict__ x, const float* __restrict__ v,
                                      const uint8_t* __restrict__ mat, int lo, int cnt, int N,
                                      int n_mat, int* __restrict__ err) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= cnt) return;
  long long i = (long long)lo + p;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    X0[(long long)c * N + i] = x[(long long)3 * p + c];
    X0[(long long)(3 + c) * N + i] = v[(long long)3 * p + c];
  }
  for (int k = 0; k < 9; ++k) {
    X0[(long long)(6 + k) * N + i] = 0.0f;
    X0[(long long)(15 + k) * N + i] = (k % 4 == 0) ? 1.0f : 0.0f;
  }
  uint32_t m = mat[p];
  if (m >= (uint32_t)n_mat) {
    atomicOr(err, kErrArg);
    m = 0;
  }
  tag0[i] = (tag0[i] & 0xffffff00u) | m;
}

void launch_init_particles(float* X0, uint32_t* tag0, const float* x, const float* v, const uint8_t* mat, int lo,
                           int cnt, int N, int n_mat, int* err, cudaStream_t s) {
  if (cnt == 0) return;
  init_particles_kernel<<<blocks_for(cnt, 256), 256, 0, s>>>(X0, tag0, x, v, mat, lo, cnt, N, n_mat, err);
}

// State rows in the caller's order. Bound by memory: coalesced reads of the
// fields asked for only, and one 12- or 36-byte row per particle and output
// written at its caller's place, so that no row passes through the host
// (40 steps of 2M particles with x and v read back: 34.4 ms when all 24 fields
// went to the host and back, 11.4 ms; 10 steps of 100k: 1.36 -> 0.44 ms).
__global__ void __launch_bounds__(256)
read_state_kernel(Params P, const float* __restrict__ st, const uint32_t* __restrict__ tag0,
                  const int* __restrict__ pid, int lo, int cnt, float* __restrict__ x, float* __restrict__ v,
                  float* __restrict__ C, float* __restrict__ F) {
  const int N = P.N;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  const int q = pid ? pid[p] : p;
  if (q < lo || q - lo >= cnt) return;
  const long long r = q - lo;
  if (x) {
#pragma unroll
    for (int c = 0; c < 3; ++c) x[3 * r + c] = st[(long long)(fX + c) * N + p];
  }
  if (v) {
#pragma unroll
    for (int c = 0; c < 3; ++c) v[3 * r + c] = st[(long long)(fV + c) * N + p];
  }
  if (C) {
#pragma unroll
    for (int c = 0; c < 9; ++c) C[9 * r + c] = st[(long long)(fC + c) * N + p];
  }
  if (F) {
    const bool liquid = is_liquid(P.mat[tag_mat(tag0[q])].kind);
#pragma unroll
    for (int c = 0; c < 9; ++c)
      F[9 * r + c] = (liquid && c > 0) ? ((c % 4 == 0) ? 1.0f : 0.0f) : st[(long long)(fF + c) * N + p];
  }
}

void launch_read_state(const Params& P, const float* st, const uint32_t* tag0, const int* pid, int lo, int cnt,
                       float* x, float* v, float* C, float* F, cudaStream_t s) {
  if (P.N == 0 || cnt == 0) return;
  read_state_kernel<<<blocks_for(P.N, 256), 256, 0, s>>>(P, st, tag0, pid, lo, cnt, x, v, C, F);
}

__global__ void iota_kernel(int* __restrict__ a, int N) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < N) a[p] = p;
}

int sm_count() {
  constexpr int kMaxDev = 64;
  static int cached[kMaxDev] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
    cudaGetLastError();
    return 1;
  }
  if (cached[dev] <= 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
      cudaGetLastError();
      n = 1;
    }
    cached[dev] = n;  // a plain int store: concurrent first calls write the same value
  }
  return cached[dev];
}

// Measured (GB300, gradient runs, us per launch unless stated):
// * CTAs of 128 against 256: fused step 148 / 150 (2M particles), 24.9 / 25.5
//   (200k), 17.4 / 18.2 (100k), 11.6 / 12.1 (8k); P2G adjoint 124 / 126 and
//   G2P 82 / 98 (2M). 64 a CTA: no faster at any size down to 8k.
// * fused step and G2P adjoint at 8 resident CTAs (64 registers) against 6
//   (80): 148 / 160 and 147 / 162 (2M), 45 / 47 and 46 / 50 (500k), 19.0 / 21.9
//   and 17.7 / 22.1 (130k: one wave against two); 25.3 / 24.9 and 23.8 / 23.3
//   (200k: two waves either way), 18.1 / 17.4 (100k: one wave either way). The lean
//   step of forward-only runs has 104 registers in the wide build, 4 CTAs, and was
//   not measured apart.
// * one adjoint kernel against two, whole reverse sweep: 0.53 / 0.74 ms (8k
//   particles), 0.70 / 0.74 (100k), 1.86 / 1.90 (200k), 4.22 / 4.42 (500k), 7.85
//   / 7.86 (1M), 15.1 / 14.7 (2M), 11.8 / 11.5 (3.2M in 64 scenes): fused saves a
//   launch and the adjoint state's round trip, but its 128 registers leave half
//   the warps, which counts once the chip is full for many waves.
constexpr int kFuseBelow = 1000000;
Tuning default_tuning(int N) {
  Tuning tu;
  const long long ctas = blocks_for(N, tu.scatter_threads);
  tu.scatter_ctas = tight_build_wins(ctas, sm_count(), 768 / tu.scatter_threads, 1024 / tu.scatter_threads) ? 4 : 3;
  tu.fuse_adjoint = N < kFuseBelow ? 1 : 0;
  return tu;
}

void launch_iota(int* a, int N, cudaStream_t s) {
  if (N == 0) return;
  iota_kernel<<<blocks_for(N, 256), 256, 0, s>>>(a, N);
}

// adj_field[c * N + p] += seed[pid[p] * ncomp + c], c < ncomp, for particles of
// the caller range [lo, lo + count).
__global__ void add_seed_kernel(float* __restrict__ adj, const float* __restrict__ seed,
                                const int* __restrict__ pid, int lo, int count, int N, int ncomp) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  int q = pid[p] - lo;
  if (q < 0 || q >= count) return;
  for (int c = 0; c < ncomp; ++c) adj[(long long)c * N + p] += seed[(long long)q * ncomp + c];
}

// dst += src. Seeds seldom hold more than the position's fields: zeros are read
// and nothing else (15 fields of 2M particles, three of them set: 94 -> 50 us).
__global__ void __launch_bounds__(256)
add_fields_kernel(float* __restrict__ dst, float* __restrict__ src, long long n, int clear_src) {
  constexpr int kBatch = 4;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride * kBatch) {
    float v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) v[u] = i + u * stride < n ? src[i + u * stride] : 0.0f;
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const long long j = i + u * stride;
      if (v[u] == 0.0f) continue;  // also past the end
      dst[j] += v[u];
      if (clear_src) src[j] = 0.0f;
    }
  }
}

void launch_add_fields(float* dst, float* src, long long n, int clear_src, cudaStream_t s) {
  if (n <= 0) return;
  long long blocks = (n + 255) / 256;
  const int cap = sm_count() * 8;
  add_fields_kernel<<<int(blocks < cap ? blocks : cap), 256, 0, s>>>(dst, src, n, clear_src);
}

void launch_add_seed(float* adj_field, const float* seed, const int* pid, const uint32_t*, int,
                     int lo, int count, int N, cudaStream_t s, int ncomp) {
  if (N == 0) return;
  add_seed_kernel<<<blocks_for(N, 256), 256, 0, s>>>(adj_field, seed, pid, lo, count, N, ncomp);
}

// ---------------------------------------------------------------------------
// tool kinematics (Sec. 4.2: the action is the tool's linear and angular
// velocity; App. B.1: held for a fixed number of substeps). The pose in FP64:
//   p_{n+1} = p_n + dt pdot_n,  q_{n+1} = normalize(dq(omega_n dt) q_n),
//   dq(w) = (cos(|w|/2), sin(|w|/2) w/|w|).
// Pose record per step: p (3), q (4), pdot (3), omega (3).
// ---------------------------------------------------------------------------
__device__ inline void qmul(const double* a, const double* b, double* o) {
  o[0] = a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3];
  o[1] = a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2];
  o[2] = a[0] * b[2] - a[1] * b[3] + a[2] * b[0] + a[3] * b[1];
  o[3] = a[0] * b[3] + a[1] * b[2] - a[2] * b[1] + a[3] * b[0];
}

// dq(omega dt) and, if J != null, d dq / d omega (4x3, row-major)
__device__ inline void dq_of(const double* om, double dt, double* dq, double* J) {
  double w2 = om[0] * om[0] + om[1] * om[1] + om[2] * om[2];
  double w = sqrt(w2);
  double th = 0.5 * dt * w;  // half angle
  double h = 0.5 * dt;
  // sinc(th) = sin(th)/th and (th cos th - sin th)/th^3, via series near 0
  double sinc, g;
  if (th < 1e-4) {
    double t2 = th * th;
    sinc = 1.0 - t2 / 6.0 + t2 * t2 / 120.0;
    g = -1.0 / 3.0 + t2 / 30.0;
  } else {
    sinc = sin(th) / th;
    g = (th * cos(th) - sin(th)) / (th * th * th);
  }
  dq[0] = cos(th);
  for (int i = 0; i < 3; ++i) dq[1 + i] = h * sinc * om[i];
  if (J) {
    // d cos(th)/d om = -sin(th) h om / w = -h^2 sinc om
    for (int k = 0; k < 3; ++k) J[k] = -h * h * sinc * om[k];
    // d (h sinc om_i)/d om_k = h (sinc delta_ik + om_i dsinc/dth h om_k / w)
    //                        = h sinc delta_ik + h^3 g om_i om_k
    for (int i = 0; i < 3; ++i)
      for (int k = 0; k < 3; ++k) J[3 * (1 + i) + k] = h * sinc * (i == k ? 1.0 : 0.0) + h * h * h * g * om[i] * om[k];
  }
}

__device__ inline void qnormalize(double* q) {
  const double r = 1.0 / sqrt(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
  for (int i = 0; i < 4; ++i) q[i] *= r;
}

// One CTA per scene. The chain over the actions is short (one rotation and one
// translation each) and the steps inside an action are closed form, so nothing
// walks the steps one by one: m steps of one action turn by dq(m omega dt) and
// move by m dt pdot. Per chunk of 32 actions, warp 0 (lane a: action a) takes
// the actions' whole rotations and translations, an inclusive scan over the
// lanes and the pose at each action's first step into shared memory; then
// every thread takes a step of the chunk. FP64 throughout; bound by the latency
// of its FP64 chain (200 steps in 20 actions: 45 us walked step by step, 25 us
// so).
constexpr int kToolThreads = 128;
__global__ void __launch_bounds__(kToolThreads)
tool_forward_kernel(int S, const float* __restrict__ pose0,
                                    const float* __restrict__ actions, int n_actions, int spa,
                                    int n_steps, int max_steps, double dt, float* __restrict__ poses) {
  __shared__ double sp[32][3], sq[32][4], carry[7];
  const int sc = blockIdx.x;
  const int lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    double q[4];
    for (int i = 0; i < 4; ++i) q[i] = pose0[sc * 7 + 3 + i];
    qnormalize(q);
    for (int i = 0; i < 3; ++i) carry[i] = pose0[sc * 7 + i];
    for (int i = 0; i < 4; ++i) carry[3 + i] = q[i];
  }
  __syncthreads();
  // first step of action a; the last action holds to the end
  auto first_step = [&](int a) { return a >= n_actions ? n_steps : (int)min((long long)a * spa, (long long)n_steps); };
  for (int a0 = 0; a0 < n_actions; a0 += 32) {
    if (threadIdx.x < 32) {
      const int a = a0 + lane;
      const int len = a < n_actions ? first_step(a + 1) - first_step(a) : 0;
      double D[4] = {1.0, 0.0, 0.0, 0.0}, tr[3] = {0.0, 0.0, 0.0};
      if (len > 0) {
        const float* act = actions + ((long long)sc * n_actions + a) * 6;
        double om[3];
        for (int i = 0; i < 3; ++i) {
          tr[i] = dt * len * act[i];
          om[i] = act[3 + i];
        }
        dq_of(om, dt * len, D, nullptr);
      }
      // inclusive scans across lanes: rotations compose with later ones on the left
      for (int off = 1; off < 32; off <<= 1) {
        double oD[4], ot[3];
        for (int i = 0; i < 4; ++i) oD[i] = __shfl_up_sync(0xffffffffu, D[i], off);
        for (int i = 0; i < 3; ++i) ot[i] = __shfl_up_sync(0xffffffffu, tr[i], off);
        if (lane >= off) {
          double t4[4];
          qmul(D, oD, t4);
          for (int i = 0; i < 4; ++i) D[i] = t4[i];
          for (int i = 0; i < 3; ++i) tr[i] += ot[i];
        }
      }
      double E[4], et[3], q[4], q2[4];
      for (int i = 0; i < 4; ++i) E[i] = __shfl_up_sync(0xffffffffu, D[i], 1);
      for (int i = 0; i < 3; ++i) et[i] = __shfl_up_sync(0xffffffffu, tr[i], 1);
      if (lane == 0) {
        E[0] = 1.0;
        E[1] = E[2] = E[3] = 0.0;
        et[0] = et[1] = et[2] = 0.0;
      }
      qmul(E, carry + 3, q);
      qnormalize(q);
      qmul(D, carry + 3, q2);
      qnormalize(q2);
      for (int i = 0; i < 3; ++i) sp[lane][i] = carry[i] + et[i];
      for (int i = 0; i < 4; ++i) sq[lane][i] = q[i];
      __syncwarp();
      if (lane == 31) {
        for (int i = 0; i < 3; ++i) carry[i] += tr[i];
        for (int i = 0; i < 4; ++i) carry[3 + i] = q2[i];
      }
    }
    __syncthreads();
    const int hi = first_step(a0 + 32 < n_actions ? a0 + 32 : n_actions);
    for (int n = first_step(a0) + threadIdx.x; n < hi; n += kToolThreads) {
      const int a = min(n / spa, n_actions - 1), m = n - first_step(a);
      const float* act = actions + ((long long)sc * n_actions + a) * 6;
      const double om[3] = {act[3], act[4], act[5]};
      double dq[4], q[4];
      dq_of(om, dt * m, dq, nullptr);
      qmul(dq, sq[a - a0], q);
      qnormalize(q);
      float* rec = poses + ((long long)sc * max_steps + n) * kToolFields;
      for (int i = 0; i < 3; ++i) rec[i] = float(sp[a - a0][i] + dt * m * act[i]);
      for (int i = 0; i < 4; ++i) rec[3 + i] = float(q[i]);
      for (int i = 0; i < 6; ++i) rec[7 + i] = act[i];
    }
    __syncthreads();
  }
}

void launch_tool_forward(const Params& P, const float* pose0, const float* actions, int n_actions,
                         int spa, int n_steps, int max_steps, float* poses, cudaStream_t s) {
  tool_forward_kernel<<<P.S, kToolThreads, 0, s>>>(P.S, pose0, actions, n_actions, spa, n_steps, max_steps,
                                                   (double)P.dt, poses);
}

__device__ inline void qmulf(const float* a, const float* b, float* o) {
  o[0] = a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3];
  o[1] = a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2];
  o[2] = a[0] * b[2] - a[1] * b[3] + a[2] * b[0] + a[3] * b[1];
  o[3] = a[0] * b[3] + a[1] * b[2] - a[2] * b[1] + a[3] * b[0];
}

// d R(q) / d q contracted with gR: returns dL/dq (4)
__device__ inline void rot_q_adjoint(const float* q, const float* gR, float* gq) {
  float w = q[0], x = q[1], y = q[2], z = q[3];
  const float* G = gR;
  // R = [[1-2(yy+zz), 2(xy-wz), 2(xz+wy)], [2(xy+wz), 1-2(xx+zz), 2(yz-wx)], [2(xz-wy), 2(yz+wx), 1-2(xx+yy)]]
  gq[0] = 2.0f * (-z * G[1] + y * G[2] + z * G[3] - x * G[5] - y * G[6] + x * G[7]);
  gq[1] = 2.0f * (y * G[1] + z * G[2] + y * G[3] - 2.0f * x * G[4] - w * G[5] + z * G[6] + w * G[7] - 2.0f * x * G[8]);
  gq[2] = 2.0f * (-2.0f * y * G[0] + x * G[1] + w * G[2] + x * G[3] + z * G[5] - w * G[6] + z * G[7] - 2.0f * y * G[8]);
  gq[3] = 2.0f * (-2.0f * z * G[0] - w * G[1] + x * G[2] + w * G[3] - 2.0f * z * G[4] + y * G[5] + x * G[6] + y * G[7]);
}

// Reverse sweep of the kinematics: per-step tool gradients (p, R, pdot, omega)
// -> action gradients (accumulated into action_grad, [S][n_actions][6]). One
// CTA per scene: every action's rotation increment and its Jacobian (FP64) and
// the pose and gradient rows of 128 steps at a time are staged in shared
// memory. Only the orientation's adjoint recurrence is serial, so thread 0
// walks nothing else (in FP32, the next step's operands loaded before this
// step's stores); what a step needs before and gives after it is a thread per
// step, and each action's sum a thread per component, last step first. Bound
// by the latency of the walk (200 steps: 95 us with everything in it, 34 us so).
constexpr int kToolChunk = 128;

size_t tool_backward_smem(int n_actions) {
  return (static_cast<size_t>(n_actions) * (16 + 6) + static_cast<size_t>(kToolChunk) * (kToolFields + kToolGradFields)) *
         sizeof(float);
}

__global__ void __launch_bounds__(kToolThreads)
tool_backward_kernel(const float* __restrict__ actions, int n_actions, int spa, int n_steps, int max_steps, float dt,
                     const float* __restrict__ poses, const float* __restrict__ tool_grad,
                     float* __restrict__ action_grad) {
  extern __shared__ float tsm[];
  float* sdq = tsm;                                  // [n_actions][16]: dq (4), d dq / d omega (12)
  float* sag = sdq + (size_t)n_actions * 16;         // [n_actions][6] action gradients
  // [kToolChunk][13]: the pose record; then 0-2 the position adjoint and 7-10
  // the orientation adjoint that reach the step, 3-6 its unit quaternion q
  float* srec = sag + (size_t)n_actions * 6;
  // [kToolChunk][18]: the tool gradient; then 3-6 the rotation's share of the
  // orientation adjoint, 7-10 qh, 11 1/|qq|, 12-17 the step's action gradient
  float* stg = srec + (size_t)kToolChunk * kToolFields;
  const int sc = blockIdx.x, tid = threadIdx.x;
  for (int a = tid; a < n_actions; a += kToolThreads) {
    const float* act = actions + ((long long)sc * n_actions + a) * 6;
    double om[3] = {act[3], act[4], act[5]}, dqd[4], Jd[12];
    dq_of(om, (double)dt, dqd, Jd);
    for (int i = 0; i < 4; ++i) sdq[a * 16 + i] = float(dqd[i]);
    for (int i = 0; i < 12; ++i) sdq[a * 16 + 4 + i] = float(Jd[i]);
    for (int i = 0; i < 6; ++i) sag[a * 6 + i] = 0.0f;
  }
  float Pb[3] = {0, 0, 0}, Qb[4] = {0, 0, 0, 0};  // thread 0
  for (int n1 = n_steps; n1 > 0; n1 -= kToolChunk) {
    const int n0 = max(0, n1 - kToolChunk);
    __syncthreads();
    for (int i = tid; i < (n1 - n0) * kToolFields; i += kToolThreads)
      srec[i] = poses[((long long)sc * max_steps + n0) * kToolFields + i];
    for (int i = tid; i < (n1 - n0) * kToolGradFields; i += kToolThreads)
      stg[i] = tool_grad[((long long)sc * max_steps + n0) * kToolGradFields + i];
    __syncthreads();
    for (int n = n0 + tid; n < n1; n += kToolThreads) {
      float* rec = srec + (n - n0) * kToolFields;
      float* tg = stg + (n - n0) * kToolGradFields;
      // the stored pose (a unit quaternion to FP32 precision) is re-normalised
      float q[4], qq[4], gq[4];
      const float qr = rsqrtf(rec[3] * rec[3] + rec[4] * rec[4] + rec[5] * rec[5] + rec[6] * rec[6]);
      for (int i = 0; i < 4; ++i) q[i] = rec[3 + i] * qr;
      // q_{n+1} = qh = qq / |qq|, qq = dq q
      qmulf(sdq + min(n / spa, n_actions - 1) * 16, q, qq);
      const float inq = rsqrtf(qq[0] * qq[0] + qq[1] * qq[1] + qq[2] * qq[2] + qq[3] * qq[3]);
      rot_q_adjoint(q, tg + 3, gq);
      for (int i = 0; i < 4; ++i) {
        rec[3 + i] = q[i];
        tg[3 + i] = gq[i];
        tg[7 + i] = qq[i] * inq;
      }
      tg[11] = inq;
    }
    __syncthreads();
    if (tid == 0) {
      float g[12], dq[4];
      auto load = [&](int n) {
        const float* tg = stg + (n - n0) * kToolGradFields;
        const float* d = sdq + min(n / spa, n_actions - 1) * 16;
#pragma unroll
        for (int i = 0; i < 12; ++i) g[i] = tg[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) dq[i] = d[i];
      };
      load(n1 - 1);
      for (int n = n1 - 1; n >= n0; --n) {
        float* rec = srec + (n - n0) * kToolFields;
        float h[12], e[4];
#pragma unroll
        for (int i = 0; i < 12; ++i) h[i] = g[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) e[i] = dq[i];
        load(n > n0 ? n - 1 : n);
        const float dotq = h[7] * Qb[0] + h[8] * Qb[1] + h[9] * Qb[2] + h[10] * Qb[3];
        float r[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) r[i] = (Qb[i] - h[7 + i] * dotq) * h[11];
        // p_{n+1} = p_n + dt pdot_n
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          rec[i] = Pb[i];
          Pb[i] += h[i];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) rec[7 + i] = Qb[i];
        // qq = L(dq) q: qb = L(dq)^T qqb
        Qb[0] = e[0] * r[0] + e[1] * r[1] + e[2] * r[2] + e[3] * r[3] + h[3];
        Qb[1] = -e[1] * r[0] + e[0] * r[1] + e[3] * r[2] - e[2] * r[3] + h[4];
        Qb[2] = -e[2] * r[0] - e[3] * r[1] + e[0] * r[2] + e[1] * r[3] + h[5];
        Qb[3] = -e[3] * r[0] + e[2] * r[1] - e[1] * r[2] + e[0] * r[3] + h[6];
      }
    }
    __syncthreads();
    for (int n = n0 + tid; n < n1; n += kToolThreads) {
      const float* rec = srec + (n - n0) * kToolFields;
      float* tg = stg + (n - n0) * kToolGradFields;
      const float* q = rec + 3;
      const float* Qn = rec + 7;
      const float* qh = tg + 7;
      const float* Jdq = sdq + min(n / spa, n_actions - 1) * 16 + 4;
      const float dotq = qh[0] * Qn[0] + qh[1] * Qn[1] + qh[2] * Qn[2] + qh[3] * Qn[3];
      float r[4], dqb[4];
      for (int i = 0; i < 4; ++i) r[i] = (Qn[i] - qh[i] * dotq) * tg[11];
      // dqb = Rm(q)^T qqb with qq = Rm(q) dq
      dqb[0] = q[0] * r[0] + q[1] * r[1] + q[2] * r[2] + q[3] * r[3];
      dqb[1] = -q[1] * r[0] + q[0] * r[1] - q[3] * r[2] + q[2] * r[3];
      dqb[2] = -q[2] * r[0] + q[3] * r[1] + q[0] * r[2] - q[1] * r[3];
      dqb[3] = -q[3] * r[0] - q[2] * r[1] + q[1] * r[2] + q[0] * r[3];
      for (int k = 0; k < 3; ++k) {
        float omb = tg[15 + k];
        for (int i = 0; i < 4; ++i) omb += Jdq[3 * i + k] * dqb[i];
        tg[12 + k] += dt * rec[k];
        tg[15 + k] = omb;
      }
    }
    __syncthreads();
    const int a0 = min(n0 / spa, n_actions - 1), a1 = min((n1 - 1) / spa, n_actions - 1);
    for (int t = tid; t < (a1 - a0 + 1) * 6; t += kToolThreads) {
      const int a = a0 + t / 6, k = t % 6;
      const long long lo = max((long long)a * spa, (long long)n0);
      const long long hi = a == n_actions - 1 ? n1 : min((long long)(a + 1) * spa, (long long)n1);
      float v = sag[a * 6 + k];
#pragma unroll 4
      for (long long n = hi - 1; n >= lo; --n) v += stg[(n - n0) * kToolGradFields + 12 + k];
      sag[a * 6 + k] = v;
    }
  }
  __syncthreads();
  for (int i = tid; i < n_actions * 6; i += kToolThreads) action_grad[(long long)sc * n_actions * 6 + i] += sag[i];
}

void launch_tool_backward(const Params& P, const float* actions, int n_actions,
                          int spa, int n_steps, int max_steps, const float* poses,
                          const float* tool_grad, float* action_grad, cudaStream_t s) {
  const size_t smem = tool_backward_smem(n_actions);
  if (smem > 48 * 1024) cudaFuncSetAttribute(tool_backward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(smem));
  tool_backward_kernel<<<P.S, kToolThreads, smem, s>>>(actions, n_actions, spa, n_steps, max_steps, P.dt, poses,
                                                       tool_grad, action_grad);
}

// ---------------------------------------------------------------------------
// losses (App. C)
// ---------------------------------------------------------------------------
__device__ inline void block_add_double(double v, double* out) {
  __shared__ double ws[32];
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) ws[wid] = v;
  __syncthreads();
  if (wid == 0) {
    double s = lane < (int)(blockDim.x >> 5) ? ws[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0 && s != 0.0) atomicAdd(out, s);
  }
}

// L_s = w sum |x - t|^2 over particles of scene `scene` (-1: all, per-scene
// totals into loss[scene]); adj_x += 2 w (x - t). The FP64 units would bound it
// (98 us at 2M particles with the sum in FP64 throughout, 17 us so), so a thread
// sums the exact squares of its kItems particles in three FP32 words, which
// loses nothing against FP64, and goes to FP64 once; particles are sorted by scene,
// so its particles seldom belong to more than one loss entry, nor do a CTA's.
template <int kItems>
__global__ void __launch_bounds__(256)
position_loss_kernel(Params P, const float* __restrict__ st, const uint32_t* __restrict__ tag,
                     int scene, float tx, float ty, float tz, float w,
                     float* __restrict__ adj, double* __restrict__ loss) {
  __shared__ double ws[8];
  __shared__ int wt[8];
  const int N = P.N;
  constexpr int kBatch = 4;
  const int base = blockIdx.x * (256 * kItems) + threadIdx.x;
  int cur = -1;
  Sum3 acc;
#pragma unroll
  for (int it = 0; it < kItems; it += kBatch) {
    uint32_t tg[kBatch];
    float d[kBatch][3], g[kBatch][3];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {  // all loads first; past the end: the last particle, not used
      const int p = min(base + (it + u) * 256, N - 1);
      tg[u] = tag[p];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        d[u][k] = st[k * N + p];
        g[u][k] = adj[k * N + p];
      }
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int p = base + (it + u) * 256, sc = tag_scene(tg[u]);
      if (p >= N || (scene >= 0 && sc != scene)) continue;
      const float d0 = d[u][0] - tx, d1 = d[u][1] - ty, d2 = d[u][2] - tz;
      adj[p] = g[u][0] + 2.0f * w * d0;
      adj[N + p] = g[u][1] + 2.0f * w * d1;
      adj[2 * N + p] = g[u][2] + 2.0f * w * d2;
      const int t = scene < 0 ? sc : 0;
      if (t != cur) {
        if (cur >= 0) atomicAdd(loss + cur, (double)w * acc.value());
        acc = Sum3();
        cur = t;
      }
      const float sq = d0 * d0 + d1 * d1 + d2 * d2;
      if (sq > 1e-25f && sq < 1e30f) {
        acc.add_square(d0);
        acc.add_square(d1);
        acc.add_square(d2);
      } else if (sq != 0.0f || d0 != 0.0f || d1 != 0.0f || d2 != 0.0f) {  // a target far outside, one met to 3e-13, or NaN
        atomicAdd(loss + t, (double)w * ((double)d0 * d0 + (double)d1 * d1 + (double)d2 * d2));
      }
    }
  }
  double l = cur >= 0 ? (double)w * acc.value() : 0.0;
  // one atomic per CTA when its particles share the loss entry
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int tmax = __reduce_max_sync(0xffffffffu, cur);
  const int tmin = __reduce_min_sync(0xffffffffu, cur >= 0 ? cur : INT_MAX);
  const bool one = tmax >= 0 && tmin == tmax;
  if (one) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  } else if (cur >= 0) {
    atomicAdd(loss + cur, l);
  }
  if (lane == 0) {
    ws[wid] = l;
    wt[wid] = one ? tmax : -1;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = -1;
    double s = 0.0;
    for (int i = 0; i < 8; ++i) {
      if (wt[i] < 0) continue;
      if (wt[i] != t && t >= 0) {
        atomicAdd(loss + t, s);
        s = 0.0;
      }
      t = wt[i];
      s += ws[i];
    }
    if (t >= 0) atomicAdd(loss + t, s);
  }
}

// Particles of a thread: with 8 the FP64 work is halved, with 4 the loads of a small
// scene wait once (the whole call, us, 8 / 4: 34.5 / 29.8 at 3k particles, 36.4 / 29.7
// at 100k, 38.1 / 38.2 at 500k, 39.5 / 50.3 at 2M).
constexpr int kLossFour = 500000;
void launch_position_loss(const Params& P, const float* st, const uint32_t* tag, int scene,
                          float tx, float ty, float tz, float w, float* adj, double* loss,
                          cudaStream_t s) {
  if (P.N == 0) return;
  const int items = P.N < kLossFour ? 4 : 8;
  auto k = items == 4 ? position_loss_kernel<4> : position_loss_kernel<8>;
  k<<<blocks_for(P.N, 256 * items), 256, 0, s>>>(P, st, tag, scene, tx, ty, tz, w, adj, loss);
}

// P2G mass of the particles of one scene into a dense float grid
__global__ void mass_scatter_kernel(Params P, const float* __restrict__ st, const uint32_t* __restrict__ tag,
                                    int scene, float* __restrict__ mg) {
  const int N = P.N;
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  uint32_t tg = tag[p];
  if (tag_scene(tg) != scene) return;
  float x[3] = {st[p], st[N + p], st[2 * N + p]};
  Stencil sc;
  make_stencil(x, P, sc);
  float m = P.mat[tag_mat(tg)].mass;
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b)
      for (int c = 0; c < 3; ++c) {
        long long idx = ((long long)(sc.base[0] + a) * P.n + sc.base[1] + b) * P.n + sc.base[2] + c;
        atomicAdd(mg + idx, m * sc.w[0][a] * sc.w[1][b] * sc.w[2][c]);
      }
}

void launch_mass_scatter(const Params& P, const float* st, const uint32_t* tag, int scene,
                         float* mgrid, cudaStream_t s) {
  if (P.N == 0) return;
  mass_scatter_kernel<<<blocks_for(P.N, 256), 256, 0, s>>>(P, st, tag, scene, mgrid);
}

// L = sum (m - m*)^2 / M^2 + sum m d* / M; dL/dm per node, in FP64. Most nodes
// hold no mass and want none: they add nothing, and their dL/dm is one rounded
// product of two FP32 numbers, the same in FP32. FP64, whose units bound the
// rest, is left to the others (128^3 nodes: 83 -> 9 us).
__global__ void mass_loss_nodes_kernel(long long n3, const float* __restrict__ mg, const float* __restrict__ tm,
                                       const float* __restrict__ td, float inv_M, float* __restrict__ dLdm,
                                       double* __restrict__ loss) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double l = 0.0;
  if (i < n3) {
    const float mf = mg[i], tf = tm[i], df = td[i], g = df * inv_M;
    if (mf == 0.0f && tf == 0.0f && isfinite(g)) {
      dLdm[i] = g;
    } else {
      double m = mf, d = m - (double)tf;
      l = d * d * (double)inv_M * inv_M + m * (double)df * inv_M;
      dLdm[i] = float(2.0 * d * inv_M * inv_M + (double)df * inv_M);
    }
  }
  if (__syncthreads_or(l != 0.0)) block_add_double(l, loss);
}

void launch_mass_loss_nodes(long long n3, const float* mgrid, const float* tm, const float* td,
                            float inv_M, float* dLdm, double* loss, cudaStream_t s) {
  mass_loss_nodes_kernel<<<blocks_for(n3, 256), 256, 0, s>>>(n3, mgrid, tm, td, inv_M, dLdm, loss);
}

// adj_x += sum_o dL/dm_i m_p grad W_o
__global__ void mass_loss_grad_kernel(Params P, const float* __restrict__ st, const uint32_t* __restrict__ tag,
                                      int scene, const float* __restrict__ g, float* __restrict__ adj) {
  const int N = P.N;
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  uint32_t tg = tag[p];
  if (tag_scene(tg) != scene) return;
  float x[3] = {st[p], st[N + p], st[2 * N + p]};
  Stencil sc;
  make_stencil(x, P, sc);
  float m = P.mat[tag_mat(tg)].mass;
  float gx = 0.f, gy = 0.f, gz = 0.f;
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b)
      for (int c = 0; c < 3; ++c) {
        long long idx = ((long long)(sc.base[0] + a) * P.n + sc.base[1] + b) * P.n + sc.base[2] + c;
        float gm = g[idx] * m * P.inv_dx;
        gx += gm * sc.dw[0][a] * sc.w[1][b] * sc.w[2][c];
        gy += gm * sc.w[0][a] * sc.dw[1][b] * sc.w[2][c];
        gz += gm * sc.w[0][a] * sc.w[1][b] * sc.dw[2][c];
      }
  adj[p] += gx;
  adj[N + p] += gy;
  adj[2 * N + p] += gz;
}

void launch_mass_loss_grad(const Params& P, const float* st, const uint32_t* tag, int scene,
                           const float* dLdm, float* adj, cudaStream_t s) {
  if (P.N == 0) return;
  mass_loss_grad_kernel<<<blocks_for(P.N, 256), 256, 0, s>>>(P, st, tag, scene, dLdm, adj);
}

}  // namespace mpm
