// Grid-based gas solver (paper Sec. 3.2 "Gas", after Stam 1999) and its
// adjoint (App. A: the projection's gradient is written by hand). The step
// and its readings are stated in include/mpm_gas.h.
//
// Every kernel is a stencil over the n^3 cells, one thread per cell, fields
// in SoA FP32 (k fastest, so a warp reads 32 consecutive cells of a row):
//   forward   advect (buoyancy folded into the back-trace and the samples),
//             divergence (+ FP64 block sums for the mean), K damped Jacobi
//             sweeps, gradient subtraction;
//   adjoint   transposed gradient, the same K sweeps, FP64 sums for the mean,
//             transposed divergence with the solid mask, transposed
//             advection (scatter of the trilinear weights by atomics plus the
//             back-trace's derivative), buoyancy.
// The per-step launch sequences are captured once per step index as CUDA
// graphs and replayed.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <string>
#include <utility>
#include <vector>

#include "graph.h"
#include "mpm_gas.h"
#include "sum3.cuh"
#include "sur_ptx.cuh"

namespace {

constexpr float kOmega = 2.0f / 3.0f;  // Jacobi weight
constexpr int kThreads = 256;
// Launch shape of the cell kernels: a CTA covers 32 cells along k (one warp)
// times 8 rows along j of one i-plane, so no thread divides its linear index.
constexpr int kBx = 32, kBy = 8;

struct Geo {
  int n;
  long long n3;
  float dx, dt_dx, beta_dt, inv2dx;
};

__device__ __forceinline__ long long cid(int n, int i, int j, int k) { return ((long long)i * n + j) * n + k; }

// this thread's cell (i, j, k) and linear index; false outside the grid
__device__ __forceinline__ bool my_cell(int n, int& i, int& j, int& k, long long& c) {
  k = blockIdx.x * kBx + threadIdx.x;
  j = blockIdx.y * kBy + threadIdx.y;
  i = blockIdx.z;
  c = ((long long)i * n + j) * n + k;
  return k < n && j < n;
}

// Neighbour bits of a cell, precomputed once from the solid mask: bit 2a is
// "the +e_a neighbour is a fluid cell", bit 2a + 1 the same for -e_a (a = x,
// y, z); kSolidBit marks a solid cell. Cells outside the grid count as solid.
enum : uint8_t { kSolidBit = 64 };

// trilinear stencil of an index-space point: base corner, fractions, and
// whether the coordinate was clamped (its derivative is then zero)
struct Tri {
  int i0[3];
  float t[3];
  bool cl[3];
};

__device__ __forceinline__ Tri tri_of(const float* X, int n) {
  Tri r;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float hi = float(n - 1);
    r.cl[a] = !(X[a] > 0.0f && X[a] < hi);
    const float x = fminf(fmaxf(X[a], 0.0f), hi);
    int b = int(floorf(x));
    b = min(b, n - 2);
    r.i0[a] = b;
    r.t[a] = x - float(b);
  }
  return r;
}

__device__ __forceinline__ float corner_w(const Tri& T, int a, int b, int c) {
  return (a ? T.t[0] : 1.0f - T.t[0]) * (b ? T.t[1] : 1.0f - T.t[1]) * (c ? T.t[2] : 1.0f - T.t[2]);
}

// d w / d t_axis of corner (a, b, c)
__device__ __forceinline__ float corner_dw(const Tri& T, int axis, int a, int b, int c) {
  const float wa = axis == 0 ? (a ? 1.0f : -1.0f) : (a ? T.t[0] : 1.0f - T.t[0]);
  const float wb = axis == 1 ? (b ? 1.0f : -1.0f) : (b ? T.t[1] : 1.0f - T.t[1]);
  const float wc = axis == 2 ? (c ? 1.0f : -1.0f) : (c ? T.t[2] : 1.0f - T.t[2]);
  return wa * wb * wc;
}

// CTA sum (thread 0's return value), every thread must call it
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double part[kThreads / 32];
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((tid & 31) == 0) part[tid >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (tid == 0)
    for (int w = 0; w < kThreads / 32; ++w) t += part[w];
  return t;
}

__global__ void __launch_bounds__(kThreads)
neighbours_kernel(int n, const uint8_t* __restrict__ solid, uint8_t* __restrict__ nbr) {
  int i, j, k;
  long long c;
  if (!my_cell(n, i, j, k, c)) return;
  auto fl = [&](int a, int b, int e) {
    return a >= 0 && b >= 0 && e >= 0 && a < n && b < n && e < n && solid[cid(n, a, b, e)] == 0;
  };
  uint8_t m = solid[c] ? kSolidBit : 0;
  if (fl(i + 1, j, k)) m |= 1;
  if (fl(i - 1, j, k)) m |= 2;
  if (fl(i, j + 1, k)) m |= 4;
  if (fl(i, j - 1, k)) m |= 8;
  if (fl(i, j, k + 1)) m |= 16;
  if (fl(i, j, k - 1)) m |= 32;
  nbr[c] = m;
}

// ---------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------
// The fields an advection samples, packed per cell: (u_x, u_y + dt beta d,
// u_z, d), i.e. the buoyancy-updated velocity and the density, so that a
// trilinear corner is one 16-byte load (and, in the adjoint, one vector
// atomic).
__global__ void __launch_bounds__(kThreads)
pack_kernel(Geo g, const float* __restrict__ u, const float* __restrict__ d, float4* __restrict__ pk) {
  int i, j, k;
  long long c;
  if (!my_cell(g.n, i, j, k, c)) return;
  const long long n3 = g.n3;
  const float dc = d[c];
  pk[c] = make_float4(u[c], u[n3 + c] + g.beta_dt * dc, u[2 * n3 + c], dc);
}

__global__ void __launch_bounds__(kThreads)
advect_kernel(Geo g, const float4* __restrict__ pk, const uint8_t* __restrict__ nbr, float* __restrict__ un,
              float* __restrict__ dn) {
  int i, j, k;
  long long c;
  if (!my_cell(g.n, i, j, k, c)) return;
  const long long n3 = g.n3;
  if (nbr[c] & kSolidBit) {
    un[c] = un[n3 + c] = un[2 * n3 + c] = dn[c] = 0.0f;
    return;
  }
  const float4 ub = pk[c];
  const float X[3] = {i - g.dt_dx * ub.x, j - g.dt_dx * ub.y, k - g.dt_dx * ub.z};
  const Tri T = tri_of(X, g.n);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float4 q = pk[cid(g.n, T.i0[0] + a, T.i0[1] + b, T.i0[2] + e)];
        const float w = corner_w(T, a, b, e);
        v.x += w * q.x;
        v.y += w * q.y;
        v.z += w * q.z;
        v.w += w * q.w;
      }
  un[c] = v.x;
  un[n3 + c] = v.y;
  un[2 * n3 + c] = v.z;
  dn[c] = v.w;
}

// FP64 adds for every cell would bound the two kernels below (GB300's FP64
// rate is a small fraction of its FP32 rate): a thread sums in three FP32 words,
// which loses nothing against FP64, and anew in FP64 where those overflow.
// Planes along i a thread walks through: fewer FP64 sums with more of them, but a
// small grid then has few threads, each waiting for its loads in turn (24^3: a pass
// of one step and its adjoint 212 us with 16 planes, 202 with 4).
__host__ __device__ inline int sum_planes(int n) { return n < 64 ? 4 : 16; }
constexpr int kSumBatch = 8;    // of them loaded at a time

// b = divergence of un on fluid cells (solid neighbours hold zero velocity);
// FP64 sum of b into *sum. 256^3: 260 -> 89 us.
__global__ void __launch_bounds__(kThreads)
divergence_kernel(Geo g, const float* __restrict__ un, const uint8_t* __restrict__ nbr, float* __restrict__ b,
                  double* __restrict__ sum) {
  const int k = blockIdx.x * kBx + threadIdx.x, j = blockIdx.y * kBy + threadIdx.y;
  const int i0 = blockIdx.z * sum_planes(g.n), i1 = min(i0 + sum_planes(g.n), g.n);
  Sum3 acc;
  if (k < g.n && j < g.n) {
    const long long n1 = g.n, n2 = (long long)g.n * g.n, n3 = g.n3;
#pragma unroll 4
    for (int i = i0; i < i1; ++i) {
      // loads issued before the bits arrive (in-grid addresses; a neighbour
      // outside the grid reads the cell itself), then chosen by the bits
      const long long c = cid(g.n, i, j, k);
      const uint8_t m = nbr[c];
      const float xp = un[i + 1 < g.n ? c + n2 : c], xm = un[i > 0 ? c - n2 : c];
      const float yp = un[n3 + (j + 1 < g.n ? c + n1 : c)], ym = un[n3 + (j > 0 ? c - n1 : c)];
      const float zp = un[2 * n3 + (k + 1 < g.n ? c + 1 : c)], zm = un[2 * n3 + (k > 0 ? c - 1 : c)];
      float s = 0.0f;
      if (m & 1) s += xp;
      if (m & 2) s -= xm;
      if (m & 4) s += yp;
      if (m & 8) s -= ym;
      if (m & 16) s += zp;
      if (m & 32) s -= zm;
      const float v = (m & kSolidBit) ? 0.0f : s * g.inv2dx;
      b[c] = v;
      acc.add(v);
    }
  }
  double own = acc.value();
  if (!isfinite(own)) {
    own = 0.0;
    for (int i = i0; i < i1; ++i) own += b[cid(g.n, i, j, k)];
  }
  const double t = block_sum(own);
  if (threadIdx.x == 0 && threadIdx.y == 0 && t != 0.0) atomicAdd(sum, t);
}

// FP64 sum over the fluid cells of x into *sum. 256^3: 258 -> 37 us.
__global__ void __launch_bounds__(kThreads)
fluid_sum_kernel(Geo g, const float* __restrict__ x, const uint8_t* __restrict__ nbr, double* __restrict__ sum) {
  const int k = blockIdx.x * kBx + threadIdx.x, j = blockIdx.y * kBy + threadIdx.y;
  const int i0 = blockIdx.z * sum_planes(g.n), i1 = min(i0 + sum_planes(g.n), g.n);
  Sum3 acc;
  if (k < g.n && j < g.n) {
    for (int i = i0; i < i1; i += kSumBatch) {
      float v[kSumBatch];
#pragma unroll
      for (int u = 0; u < kSumBatch; ++u) {  // all loads first
        const long long c = cid(g.n, min(i + u, g.n - 1), j, k);
        const float xc = x[c];
        v[u] = (i + u < i1 && !(nbr[c] & kSolidBit)) ? xc : 0.0f;
      }
#pragma unroll
      for (int u = 0; u < kSumBatch; ++u) acc.add(v[u]);
    }
  }
  double own = acc.value();
  if (!isfinite(own)) {
    own = 0.0;
    for (int i = i0; i < i1; ++i) {
      const long long c = cid(g.n, i, j, k);
      own += (nbr[c] & kSolidBit) ? 0.0f : x[c];
    }
  }
  const double t = block_sum(own);
  if (threadIdx.x == 0 && threadIdx.y == 0 && t != 0.0) atomicAdd(sum, t);
}

// mean = sum / n_fluid as one float, for the sweeps to read
__global__ void mean_kernel(const double* __restrict__ sum, double inv_nfluid, float* __restrict__ mean) {
  *mean = float(*sum * inv_nfluid);
}

// One damped Jacobi sweep on the zero-flux Laplacian of the fluid cells:
// p_out = p_in / 3 + (2/3) (sum_fluid-nbr p_in - dx^2 (rhs - mean)) / n_fluid-nbr,
// mean read from *mean when given; first: p_in = 0.
__global__ void __launch_bounds__(kThreads)
jacobi_kernel(Geo g, const float* __restrict__ p_in, float* __restrict__ p_out, const float* __restrict__ rhs,
              const uint8_t* __restrict__ nbr, const float* __restrict__ mean_p, int first) {
  int i, j, k;
  long long c;
  if (!my_cell(g.n, i, j, k, c)) return;
  const int n = g.n;
  const long long n1 = n, n2 = (long long)n * n;
  // neighbour loads issued before the neighbour bits arrive (in-grid
  // addresses; a neighbour outside the grid reads the cell itself), then
  // weighted by the bits
  float q[6], pc = 0.0f, r = 0.0f;
  if (!first) {
    q[0] = p_in[i + 1 < n ? c + n2 : c];
    q[1] = p_in[i > 0 ? c - n2 : c];
    q[2] = p_in[j + 1 < n ? c + n1 : c];
    q[3] = p_in[j > 0 ? c - n1 : c];
    q[4] = p_in[k + 1 < n ? c + 1 : c];
    q[5] = p_in[k > 0 ? c - 1 : c];
    pc = p_in[c];
  }
  r = rhs[c];
  const uint8_t m = nbr[c];
  if (m & kSolidBit) {
    p_out[c] = 0.0f;
    return;
  }
  float s = 0.0f;
  if (!first) {
#pragma unroll
    for (int t = 0; t < 6; ++t) s += (m & (1 << t)) ? q[t] : 0.0f;
  }
  const int nf = __popc(m & 63);
  const float mean = mean_p ? *mean_p : 0.0f;
  // 1 / n_fluid-nbr for n = 0..6 (no fluid neighbour: no update)
  const float inv_nf = nf == 0 ? 0.0f : nf == 1 ? 1.0f : nf == 2 ? 0.5f : nf == 3 ? (1.0f / 3.0f) : nf == 4 ? 0.25f
                     : nf == 5 ? 0.2f : (1.0f / 6.0f);
  const float upd = (s - g.dx * g.dx * (r - mean)) * inv_nf;
  p_out[c] = (1.0f - kOmega) * pc + kOmega * upd;
}

// The same sweep for n a multiple of 4: each thread updates 4 consecutive
// cells along k with 16-byte loads of p, the right-hand side and the
// neighbour bits (8 loads and one store for 4 cells instead of 9 and one per
// cell). A CTA covers 128 cells along k times 8 rows along j.
__device__ __forceinline__ float f4(const float4& v, int t) { return t == 0 ? v.x : t == 1 ? v.y : t == 2 ? v.z : v.w; }

// 1 / (number of fluid neighbours) for every set of neighbour bits (0 for
// none), in shared memory: the first 64 threads of a CTA fill it.
__device__ __forceinline__ void fill_weights(float* tab, int tid) {
  if (tid < 64) {
    const int nf = __popc(tid);
    tab[tid] = nf == 0 ? 0.0f : 1.0f / float(nf);
  }
}

// The neighbour bits of a thread's 4 cells along k when none but the grid's own
// ends along k are missing, and the weights of the first and the last cell then.
struct Ends {
  uint32_t bits;
  float w0, w3;
};
__device__ __forceinline__ Ends ends_of(bool first_in_row, bool last_in_row) {
  Ends e;
  e.bits = 0x3f3f3f3fu & ~(first_in_row ? 32u : 0u) & ~(last_in_row ? 16u << 24 : 0u);
  e.w0 = first_in_row ? 1.0f / 5.0f : 1.0f / 6.0f;
  e.w3 = last_in_row ? 1.0f / 5.0f : 1.0f / 6.0f;
  return e;
}

// Sweep of 4 cells along k: P their values, Q their neighbours at +i, -i, +j,
// -j, pl and pr the cells before and after them (zeros for cells outside the
// grid), R the right-hand side without its mean, M4 the neighbour bits (a byte a
// cell), tab from fill_weights. p is zero on solid cells before and after every
// sweep, so the sums need no tests; the bits matter only where a cell is solid
// or misses a neighbour. A row's ends are told apart from other missing
// neighbours because every warp holds one. Instructions of a pair of sweeps over
// 256^3 cells with an obstacle: 74.5 M (of warps) with each cell's bits tested
// there, 54.0 M with the weights looked up, 49.5 M with the ends set apart (55.5 M
// in a box of solid walls, where rows end in other bits).
__device__ __forceinline__ float4 sweep4(const float4& P, const float4 (&Q)[4], float pl, float pr, const float4& R,
                                         uint32_t M4, const Ends& e, const float* tab, float h2) {
  float w[4] = {e.w0, 1.0f / 6.0f, 1.0f / 6.0f, e.w3}, out[4];
  const bool plain = M4 == e.bits;
  if (!plain) {
#pragma unroll
    for (int t = 0; t < 4; ++t) w[t] = tab[(M4 >> (8 * t)) & 63u];
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const float zp = t < 3 ? f4(P, t + 1) : pr;
    const float zm = t > 0 ? f4(P, t - 1) : pl;
    const float s = f4(Q[0], t) + f4(Q[1], t) + f4(Q[2], t) + f4(Q[3], t) + zp + zm;
    // every operation spelled out: a pair rounds as two single sweeps of 4 cells do
    out[t] = fmaf(1.0f - kOmega, f4(P, t), __fmul_rn(__fmul_rn(kOmega, fmaf(-h2, f4(R, t), s)), w[t]));
  }
  if (!plain) {
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (M4 & (uint32_t(kSolidBit) << (8 * t))) out[t] = 0.0f;
  }
  return make_float4(out[0], out[1], out[2], out[3]);
}

__global__ void __launch_bounds__(kThreads)
jacobi4_kernel(Geo g, const float* __restrict__ p_in, float* __restrict__ p_out, const float* __restrict__ rhs,
               const uint8_t* __restrict__ nbr, const float* __restrict__ mean_p, int first) {
  __shared__ float tab[64];
  fill_weights(tab, threadIdx.y * kBx + threadIdx.x);
  __syncthreads();
  const int n = g.n;
  const int k0 = (blockIdx.x * kBx + threadIdx.x) * 4;
  const int j = blockIdx.y * kBy + threadIdx.y;
  const int i = blockIdx.z;
  if (k0 >= n || j >= n) return;
  const int n1 = n, n2 = n * n;
  const int c = (i * n + j) * n + k0;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 P = zero, Q[4] = {zero, zero, zero, zero};
  float pl = 0.0f, pr = 0.0f;
  if (!first) {
    P = *reinterpret_cast<const float4*>(p_in + c);
    if (i + 1 < n) Q[0] = *reinterpret_cast<const float4*>(p_in + c + n2);
    if (i > 0) Q[1] = *reinterpret_cast<const float4*>(p_in + c - n2);
    if (j + 1 < n) Q[2] = *reinterpret_cast<const float4*>(p_in + c + n1);
    if (j > 0) Q[3] = *reinterpret_cast<const float4*>(p_in + c - n1);
    pl = k0 > 0 ? p_in[c - 1] : 0.0f;
    pr = k0 + 4 < n ? p_in[c + 4] : 0.0f;
  }
  float4 R = *reinterpret_cast<const float4*>(rhs + c);
  const uint32_t M4 = *reinterpret_cast<const uint32_t*>(nbr + c);
  const float mean = mean_p ? *mean_p : 0.0f;
  R = make_float4(R.x - mean, R.y - mean, R.z - mean, R.w - mean);
  *reinterpret_cast<float4*>(p_out + c) = sweep4(P, Q, pl, pr, R, M4, ends_of(k0 == 0, k0 + 4 == n), tab, g.dx * g.dx);
}

// Two sweeps in one pass over memory. A sweep is bound by DRAM (13 bytes a
// cell: p, right-hand side and bits read, p written), so the second one is
// taken from registers and shared memory. A CTA owns a strip of R - 2 rows
// along j (all of k, 4 cells a thread, R rows of threads) and marches along i
// through `seg` planes. A strip's rows of a plane are consecutive in memory, so
// one bulk copy brings p (R + 2 rows) and one the right-hand side into a ring of
// kStages planes, up to three planes ahead (~100 KB in flight per SM; with
// plain loads one plane ahead the pair was no faster); the neighbour bits come by
// plain loads, two planes ahead. At plane i the CTA sweeps its R rows once (i +- 1
// in registers, j +- 1 from the ring), writes the result to a second ring of three
// planes, and after the step's one barrier sweeps the inner R - 2 rows of plane
// i - 1 a second time. The rows and planes of the halo are swept by both
// neighbours ((R / (R - 2)) x ((seg + 2) / seg) of the first sweep's work, none of
// the second's). Values are those of two single sweeps, bit for bit (compared at
// 160^3 to 512^3). Every wait is bounded; one that runs out sets *err. Measured per
// sweep (us, against one sweep a pass with the same arithmetic; before it 5.4 / - /
// 20.6 / 40.1): 5.6 / 4.2 at 128^3, 8.9 / 10.0 at 160^3, 13.4 / 17.0 at 192^3, 26.7 /
// 35.5 at 256^3: the pair is bound by instruction issue (0.82 of the slots), the
// single sweep by DRAM, or by L2 where everything fits there.
constexpr int kStages = 4;
struct PairShape {
  int tx, rows, strips, seg, grid_i;
  size_t smem;
};
__host__ __device__ inline size_t pair_stage_f4(int tx, int rows) { return (size_t)(2 * rows + 2) * tx; }

__global__ void __launch_bounds__(1024, 1)
jacobi2_kernel(Geo g, const float* __restrict__ p_in, float* __restrict__ p_out, const float* __restrict__ rhs,
               const uint8_t* __restrict__ nbr, const float* __restrict__ mean_p, int first, int seg,
               int* __restrict__ err) {
  extern __shared__ __align__(128) float4 sm[];
  __shared__ uint64_t bar[kStages];
  __shared__ float tab[64];
  const int n = g.n, n2 = n * n;
  const int tx = threadIdx.x, ty = threadIdx.y, TX = blockDim.x, R = blockDim.y;
  const int tid = ty * TX + tx, lane = tid & 31;
  const int plane = R * TX, per = (2 * R + 2) * TX;  // float4 of a swept plane and of a stage
  const int j0 = blockIdx.x * (R - 2);               // first inner row
  const int j = j0 + ty - 1;
  const bool row = j >= 0 && j < n;
  const bool inner = row && ty >= 1 && ty < R - 1;
  const int i0 = blockIdx.y * seg, i1 = min(i0 + seg, n);
  const int col = j * n + 4 * tx;  // only used for rows inside the grid
  // the value one cell before / after a thread's 4 comes from the neighbouring
  // lane when that holds the same row, else from shared memory (0 at the ends)
  const bool sl = tx > 0 && lane > 0, sr = tx + 1 < TX && lane < 31;
  const bool el = tx > 0 && lane == 0, er = tx + 1 < TX && lane == 31;
  const Ends ends = ends_of(tx == 0, tx + 1 == TX);
  const float mean = mean_p ? *mean_p : 0.0f, h2 = g.dx * g.dx;
  const int last = i1 - i0 + 2;  // plane i0 - 1 + o has ordinal o, 0 <= o <= last
  // sm: 3 planes of the first sweep, then kStages x (R + 2 rows of p, R rows of
  // the right-hand side); all zero, which rows outside the grid (and p in the
  // first sweep of all) stay
  for (int q = tid; q < 3 * plane + kStages * per; q += plane) sm[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  fill_weights(tab, tid);
  if (tid == 0) {
    for (int q = 0; q < kStages; ++q) sur::mbar_init(bar + q, 1);
    sur::fence_barrier_init();
  }
  sur::fence_proxy_async_smem();  // the zeros come before the copies
  __syncthreads();
  // thread 0: bring the plane of ordinal o into its slot (planes outside the
  // grid complete their phase without data)
  auto issue = [&](int o) {
    uint64_t* b = bar + o % kStages;
    const int i = i0 - 1 + o;
    if (i < 0 || i >= n) {
      sur::mbar_arrive(b);
      return;
    }
    float4* sp = sm + 3 * plane + (o % kStages) * per;
    float4* srh = sp + (R + 2) * TX;
    const int pa = max(j0 - 2, 0), pb = min(j0 + R, n);      // rows [pa, pb) of p
    const int ra = max(j0 - 1, 0), rb = min(j0 + R - 1, n);  // rows [ra, rb) of the right-hand side
    const uint32_t pbytes = first ? 0u : uint32_t(pb - pa) * n * 4u, rbytes = uint32_t(rb - ra) * n * 4u;
    sur::mbar_arrive_expect_tx(b, pbytes + rbytes);
    if (!first) sur::bulk_g2s(sp + (pa - (j0 - 2)) * TX, p_in + (size_t)i * n2 + (size_t)pa * n, pbytes, b);
    sur::bulk_g2s(srh + (ra - (j0 - 1)) * TX, rhs + (size_t)i * n2 + (size_t)ra * n, rbytes, b);
  };
  if (tid == 0)
    for (int o = 0; o < kStages && o <= last; ++o) issue(o);
  auto await = [&](int o) {
    if (!sur::mbar_wait(bar + o % kStages, (o / kStages) & 1, nullptr)) atomicOr(err, 1);
  };
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  // outside the grid the solid bits are set: the sweep gives 0
  const uint8_t* nb = nbr + col;
  auto load_m = [&](int i) -> uint32_t {
    return row && i >= 0 && i < n ? __ldg(reinterpret_cast<const uint32_t*>(nb + i * n2)) : 0x40404040u;
  };
  float4* const mine = sm + tid;                                // this thread's place in swept plane 0
  const float4* const mine_p = sm + 3 * plane + tid + TX;      // and in stage 0's p
  const float4* const mine_r = sm + 3 * plane + tid + per - plane;  // and right-hand side
  uint32_t m = load_m(i0 - 1), mn = load_m(i0), mp = 0x40404040u;
  const float4 far = (row && !first && i0 >= 2) ? __ldg(reinterpret_cast<const float4*>(p_in + (i0 - 2) * n2 + col)) : zero;
  await(0);
  await(1);
  float4 a0 = far, a1 = i0 > 0 ? mine_p[0] : zero;
  float4 s0 = zero, s1 = zero, rp = zero;  // first sweep of planes i - 2 and i - 1, right-hand side of i - 1
  int now = 0, before = 2;                 // swept plane of i and of i - 1 in the ring
  float* out = p_out + (i0 - 2) * n2 + col;  // only used for planes and rows inside the grid
  for (int o = 0; o < last; ++o) {
    const int i = i0 - 1 + o;
    const uint32_t mnn = load_m(i + 2);
    const float4 a2 = i + 1 < n ? mine_p[((o + 1) % kStages) * per] : zero;
    const float4* sp = mine_p + (o % kStages) * per;
    float4 r = mine_r[(o % kStages) * per];
    r = make_float4(r.x - mean, r.y - mean, r.z - mean, r.w - mean);
    float4 s2;
    {
      const float4 Q[4] = {a2, a0, sp[TX], sp[-TX]};
      float pl = __shfl_up_sync(0xffffffffu, a1.w, 1), pr = __shfl_down_sync(0xffffffffu, a1.x, 1);
      pl = sl ? pl : 0.0f;
      pr = sr ? pr : 0.0f;
      if (el) pl = sp[-1].w;
      if (er) pr = sp[1].x;
      s2 = sweep4(a1, Q, pl, pr, r, m, ends, tab, h2);
    }
    mine[now * plane] = s2;
    if (tid < 32 && o + 2 <= last) await(o + 2);  // read by every warp after the barrier
    __syncthreads();
    if (tid == 0 && o + kStages <= last) issue(o + kStages);  // plane i's slot is not read again
    {
      // second sweep of plane i - 1 (rows outside the strip compute it unused)
      const float4* c = mine + before * plane;
      const float4 Q[4] = {s2, s0, ty < R - 1 ? c[TX] : zero, ty > 0 ? c[-TX] : zero};
      float pl = __shfl_up_sync(0xffffffffu, s1.w, 1), pr = __shfl_down_sync(0xffffffffu, s1.x, 1);
      pl = sl ? pl : 0.0f;
      pr = sr ? pr : 0.0f;
      if (el) pl = c[-1].w;
      if (er) pr = c[1].x;
      const float4 w = sweep4(s1, Q, pl, pr, rp, mp, ends, tab, h2);
      if (inner && o >= 2) *reinterpret_cast<float4*>(out) = w;
    }
    out += n2;
    s0 = s1;
    s1 = s2;
    a0 = a1;
    a1 = a2;
    rp = r;
    mp = m;
    m = mn;
    mn = mnn;
    before = now;
    now = now == 2 ? 0 : now + 1;
  }
}

// out = un - central-difference gradient of p (p mirrored across solid faces),
// 0 on solid cells: the projected velocity, straight into the new state
__global__ void __launch_bounds__(kThreads)
gradient_kernel(Geo g, const float* __restrict__ p, const uint8_t* __restrict__ nbr, const float* __restrict__ un,
                float* __restrict__ out) {
  int i, j, k;
  long long c;
  if (!my_cell(g.n, i, j, k, c)) return;
  const uint8_t m = nbr[c];
  const long long n1 = g.n, n2 = (long long)g.n * g.n, n3 = g.n3;
  if (m & kSolidBit) {
    out[c] = out[n3 + c] = out[2 * n3 + c] = 0.0f;
    return;
  }
  const float pc = p[c];
  const long long st[3] = {n2, n1, 1};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float pp = (m & (1 << (2 * a))) ? p[c + st[a]] : pc;
    const float pm = (m & (2 << (2 * a))) ? p[c - st[a]] : pc;
    out[a * n3 + c] = un[a * n3 + c] - (pp - pm) * g.inv2dx;
  }
}

// ---------------------------------------------------------------------------
// adjoint
// ---------------------------------------------------------------------------
// t = G^T v on fluid cells (v = adjoint of the projected velocity): cell c - e
// (fluid, its + neighbour is c) contributes +v(c - e), cell c + e contributes
// -v(c + e), and c mirrors its missing neighbours onto itself.
__global__ void __launch_bounds__(kThreads)
gradient_t_kernel(Geo g, const float* __restrict__ v, const uint8_t* __restrict__ nbr, float* __restrict__ t) {
  int i, j, k;
  long long c;
  if (!my_cell(g.n, i, j, k, c)) return;
  const uint8_t m = nbr[c];
  if (m & kSolidBit) {
    t[c] = 0.0f;
    return;
  }
  const long long n1 = g.n, n2 = (long long)g.n * g.n, n3 = g.n3;
  const long long st[3] = {n2, n1, 1};
  float s = 0.0f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float* va = v + a * n3;
    const bool fh = m & (1 << (2 * a)), fl = m & (2 << (2 * a));
    if (fl) s += va[c - st[a]];
    if (fh) s -= va[c + st[a]];
    if (!fh) s += va[c];
    if (!fl) s -= va[c];
  }
  t[c] = s * g.inv2dx;
}

// ubar = v - D^T (m - mean) on fluid cells, 0 on solid cells (the advection's
// solid mask); m = the swept adjoint, *mean_p its mean over the fluid cells. The
// density's adjoint (fourth field) is not projected and only passes the mask.
__global__ void __launch_bounds__(kThreads)
divergence_t_kernel(Geo g, const float* __restrict__ v, const float* __restrict__ mm, const uint8_t* __restrict__ nbr,
                    const float* __restrict__ mean_p, float* __restrict__ ubar) {
  int i, j, k;
  long long c;
  if (!my_cell(g.n, i, j, k, c)) return;
  const long long n1 = g.n, n2 = (long long)g.n * g.n, n3 = g.n3;
  const uint8_t m = nbr[c];
  if (m & kSolidBit) {
    ubar[c] = ubar[n3 + c] = ubar[2 * n3 + c] = ubar[3 * n3 + c] = 0.0f;
    return;
  }
  ubar[3 * n3 + c] = v[3 * n3 + c];
  const float mean = *mean_p;
  const long long st[3] = {n2, n1, 1};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // b(i) = (u(i + e) - u(i - e)) / 2dx on fluid i: u(c) enters b(c - e) with +, b(c + e) with -
    float s = 0.0f;
    if (m & (2 << (2 * a))) s += mm[c - st[a]] - mean;
    if (m & (1 << (2 * a))) s -= mm[c + st[a]] - mean;
    ubar[a * n3 + c] = v[a * n3 + c] - s * g.inv2dx;
  }
}

// Transposed advection: scatter (ubar_adv, dbar_adv) of every fluid cell onto
// the trilinear corners and add the back-trace's derivative to the cell's own
// velocity adjoint. acc (float4 per cell) is zero on entry and receives the
// adjoint of the packed fields (buoyancy-updated velocity, density).
// Bound by the vector atomics: neighbouring cells along k (the lanes of a warp)
// mostly trace back to neighbouring corners, so where a lane's far corners in k
// are the next lane's near ones it hands them over and they are added together
// (5 atomics a cell instead of 9).
__global__ void __launch_bounds__(kThreads)
advect_t_kernel(Geo g, const float4* __restrict__ pk, const uint8_t* __restrict__ nbr,
                const float* __restrict__ ubar, const float* __restrict__ dbar, float4* __restrict__ acc) {
  constexpr unsigned kAll = 0xffffffffu;
  int i, j, k;
  long long c;
  bool act = my_cell(g.n, i, j, k, c);
  act = act && !(nbr[c] & kSolidBit);
  const long long n3 = g.n3;
  float4 A = make_float4(0.f, 0.f, 0.f, 0.f), ub = A;
  if (act) {
    A = make_float4(ubar[c], ubar[n3 + c], ubar[2 * n3 + c], dbar[c]);
    ub = pk[c];
  }
  act = act && (A.x != 0.0f || A.y != 0.0f || A.z != 0.0f || A.w != 0.0f);
  if (!__any_sync(kAll, act)) return;
  const float X[3] = {i - g.dt_dx * ub.x, j - g.dt_dx * ub.y, k - g.dt_dx * ub.z};
  const Tri T = tri_of(X, g.n);
  // near corner of this cell's stencil (-2: no contribution, links to nothing)
  const long long q0 = act ? cid(g.n, T.i0[0], T.i0[1], T.i0[2]) : -2;
  const long long qn = __shfl_down_sync(kAll, q0, 1);
  // the next lane's near corners are this lane's far ones: same row, next cell
  const bool give = act && (threadIdx.x & 31) < 31 && qn == q0 + 1 && T.i0[2] + 1 < g.n;
  const bool take = __shfl_up_sync(kAll, int(give), 1) && (threadIdx.x & 31) > 0;
  float gX[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const float w0 = corner_w(T, a, b, 0), w1 = corner_w(T, a, b, 1);
      float4 near = make_float4(w0 * A.x, w0 * A.y, w0 * A.z, w0 * A.w);
      const float4 far = make_float4(w1 * A.x, w1 * A.y, w1 * A.z, w1 * A.w);
      const float4 in = make_float4(__shfl_up_sync(kAll, far.x, 1), __shfl_up_sync(kAll, far.y, 1),
                                    __shfl_up_sync(kAll, far.z, 1), __shfl_up_sync(kAll, far.w, 1));
      if (!act) continue;
      if (take) near = make_float4(near.x + in.x, near.y + in.y, near.z + in.z, near.w + in.w);
      const long long q = q0 + ((long long)a * g.n + b) * g.n;
      atomicAdd(acc + q, near);
      if (!give) atomicAdd(acc + q + 1, far);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float4 v = pk[q + e];
        const float s = A.x * v.x + A.y * v.y + A.z * v.z + A.w * v.w;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) gX[ax] += corner_dw(T, ax, a, b, e) * s;
      }
    }
  if (!act) return;
  const float4 own = make_float4(T.cl[0] ? 0.0f : -g.dt_dx * gX[0], T.cl[1] ? 0.0f : -g.dt_dx * gX[1],
                                 T.cl[2] ? 0.0f : -g.dt_dx * gX[2], 0.0f);
  atomicAdd(acc + c, own);
}

// adjoint of the step's input: ubar_n = acc.xyz, dbar_n = acc.w + beta dt acc.y,
// zero on solid cells (the state there is identically zero)
__global__ void __launch_bounds__(kThreads)
finish_t_kernel(Geo g, const float4* __restrict__ acc, const uint8_t* __restrict__ nbr, float* __restrict__ ubar,
                float* __restrict__ dbar) {
  int i, j, k;
  long long c;
  if (!my_cell(g.n, i, j, k, c)) return;
  const long long n3 = g.n3;
  const bool s = nbr[c] & kSolidBit;
  const float4 a = acc[c];
  ubar[c] = s ? 0.0f : a.x;
  ubar[n3 + c] = s ? 0.0f : a.y;
  ubar[2 * n3 + c] = s ? 0.0f : a.z;
  dbar[c] = s ? 0.0f : a.w + g.beta_dt * a.y;
}

// zero a state's fields (u, d) on solid cells
__global__ void __launch_bounds__(kThreads)
mask_kernel(Geo g, const uint8_t* __restrict__ nbr, float* __restrict__ x) {
  int i, j, k;
  long long c;
  if (!my_cell(g.n, i, j, k, c) || !(nbr[c] & kSolidBit)) return;
  for (int f = 0; f < 4; ++f) x[f * g.n3 + c] = 0.0f;
}

__global__ void add_kernel(long long m, const float* __restrict__ a, float* __restrict__ b) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c < m) b[c] += a[c];
}

}  // namespace

// ---------------------------------------------------------------------------
// handle and C-ABI
// ---------------------------------------------------------------------------
struct mpm_gas {
  gas_config cfg{};
  Geo g{};
  cudaStream_t stream = nullptr, cstream = nullptr;
  int nfluid = 0;
  int sms = 1;
  uint8_t* solid = nullptr;
  uint8_t* nbr = nullptr;  // neighbour bits of every cell
  float* states = nullptr;  // (max_steps + 1) x 4 n^3: u (3), d
  float *un = nullptr, *b = nullptr, *p0 = nullptr, *p1 = nullptr;
  float *adj = nullptr, *adj2 = nullptr, *acc = nullptr;  // 4 n^3 each
  float* pack = nullptr;  // 4 n^3: packed fields (float4 per cell) of the step being advected
  double* sum = nullptr;
  float* mean = nullptr;
  int* err = nullptr;   // set by a kernel whose bounded wait ran out
  int* word = nullptr;  // pinned copy of err (grids whose sweeps go in pairs)
  int step = 0;
  bool started = false, seeds = false;
  long long launches = 0;
  std::vector<cudaGraphExec_t> fwd, bwd;
  std::vector<long long> fwd_launches, bwd_launches;
  std::string last_error;
};

namespace {

sim_status gfail(gas_h h, sim_status s, const std::string& m) {
  if (h) h->last_error = m;
  return s;
}

sim_status gcuda(gas_h h, cudaError_t e, const char* where) {
  return gfail(h, SIM_E_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

inline int nblocks(long long m) { return int((m + kThreads - 1) / kThreads); }
inline dim3 cell_grid(int n) { return dim3((n + kBx - 1) / kBx, (n + kBy - 1) / kBy, n); }
inline dim3 sum_grid(int n) {
  return dim3((n + kBx - 1) / kBx, (n + kBy - 1) / kBy, (n + sum_planes(n) - 1) / sum_planes(n));
}
const dim3 kCellBlock(kBx, kBy);

// one Jacobi sweep, 4 cells a thread when n allows 16-byte rows
void sweep(const Geo& g, const float* p_in, float* p_out, const float* rhs, const uint8_t* nbr, const float* mean,
           int first, cudaStream_t st) {
  if (g.n % 4 == 0) {
    const dim3 gr((g.n / 4 + kBx - 1) / kBx, (g.n + kBy - 1) / kBy, g.n);
    jacobi4_kernel<<<gr, kCellBlock, 0, st>>>(g, p_in, p_out, rhs, nbr, mean, first);
  } else {
    jacobi_kernel<<<cell_grid(g.n), kCellBlock, 0, st>>>(g, p_in, p_out, rhs, nbr, mean, first);
  }
}

// The projection's sweeps from p = 0, in pairs from the size on where those are
// faster (figures at jacobi2_kernel); returns the buffer that holds the result and adds the
// launches.
constexpr int kPairFrom = 160, kMaxGrid = 512;
PairShape pair_shape(int n, int sms) {
  PairShape q;
  q.tx = n / 4;
  q.rows = std::min(16, 1024 / q.tx);
  q.strips = (n + q.rows - 3) / (q.rows - 2);
  // planes per CTA: the fewest waves x (planes + halo)
  q.seg = n;
  for (int k = 1, best = 1 << 30; k <= n / 8; ++k) {
    const int planes = (n + k - 1) / k, ctas = q.strips * ((n + planes - 1) / planes);
    const int cost = (ctas + sms - 1) / sms * (planes + 3);
    if (cost < best) best = cost, q.seg = planes;
  }
  q.grid_i = (n + q.seg - 1) / q.seg;
  q.smem = sizeof(float4) * ((size_t)3 * q.rows * q.tx + kStages * pair_stage_f4(q.tx, q.rows));
  return q;
}

// The largest need of any grid size. The limit belongs to the function, not to a
// handle: one set to a handle's own need would be lowered by the next, smaller one.
int pair_smem_limit(int sms) {
  size_t most = 0;
  for (int n = kPairFrom; n <= kMaxGrid; n += 4) most = std::max(most, pair_shape(n, sms).smem);
  return int(most);
}

float* sweeps(gas_h h, const float* rhs, const float* mean, cudaStream_t st, long long* launches) {
  const Geo& g = h->g;
  float* pa = h->p0;
  float* pb = h->p1;
  int done = 0;
  const bool pairs = g.n % 4 == 0 && g.n >= kPairFrom;
  const PairShape q = pairs ? pair_shape(g.n, h->sms) : PairShape{};
  while (done < h->cfg.jacobi_iters) {
    if (pairs && h->cfg.jacobi_iters - done >= 2) {
      jacobi2_kernel<<<dim3(q.strips, q.grid_i), dim3(q.tx, q.rows), q.smem, st>>>(g, pa, pb, rhs, h->nbr, mean,
                                                                                  done == 0, q.seg, h->err);
      done += 2;
    } else {
      sweep(g, pa, pb, rhs, h->nbr, mean, done == 0, st);
      done += 1;
    }
    *launches += 1;
    std::swap(pa, pb);
  }
  return pa;
}

float* state_ptr(gas_h h, int s) { return h->states + (size_t)s * 4 * h->g.n3; }

// Launches of one forward step s -> s + 1 on stream st; returns the launch count.
long long enqueue_forward(gas_h h, int s, cudaStream_t st) {
  const Geo& g = h->g;
  const long long n3 = g.n3;
  const dim3 gr = cell_grid(g.n);
  const float* in = state_ptr(h, s);
  float* out = state_ptr(h, s + 1);
  const double inv_nf = h->nfluid > 0 ? 1.0 / h->nfluid : 0.0;
  float4* pk = reinterpret_cast<float4*>(h->pack);
  pack_kernel<<<gr, kCellBlock, 0, st>>>(g, in, in + 3 * n3, pk);
  advect_kernel<<<gr, kCellBlock, 0, st>>>(g, pk, h->nbr, h->un, out + 3 * n3);
  cudaMemsetAsync(h->sum, 0, sizeof(double), st);
  divergence_kernel<<<sum_grid(g.n), kCellBlock, 0, st>>>(g, h->un, h->nbr, h->b, h->sum);
  mean_kernel<<<1, 1, 0, st>>>(h->sum, inv_nf, h->mean);
  long long swept = 0;
  const float* pa = sweeps(h, h->b, h->mean, st, &swept);
  gradient_kernel<<<gr, kCellBlock, 0, st>>>(g, pa, h->nbr, h->un, out);
  return 5 + swept;
}

// Launches of the adjoint of step s (adj holds the adjoint of state s + 1,
// and receives the adjoint of state s).
long long enqueue_backward(gas_h h, int s, cudaStream_t st) {
  const Geo& g = h->g;
  const long long n3 = g.n3;
  const dim3 gr = cell_grid(g.n);
  const float* in = state_ptr(h, s);
  const double inv_nf = h->nfluid > 0 ? 1.0 / h->nfluid : 0.0;
  float* v = h->adj;  // u (3 n^3), d (n^3)
  // projection: ubar_pre = v - D^T M J G^T v
  gradient_t_kernel<<<gr, kCellBlock, 0, st>>>(g, v, h->nbr, h->b);
  long long swept = 0;
  const float* pa = sweeps(h, h->b, nullptr, st, &swept);
  cudaMemsetAsync(h->sum, 0, sizeof(double), st);
  fluid_sum_kernel<<<sum_grid(g.n), kCellBlock, 0, st>>>(g, pa, h->nbr, h->sum);
  mean_kernel<<<1, 1, 0, st>>>(h->sum, inv_nf, h->mean);
  divergence_t_kernel<<<gr, kCellBlock, 0, st>>>(g, v, pa, h->nbr, h->mean, h->adj2);
  // advection and buoyancy, from the packed fields of step s
  float4* pk = reinterpret_cast<float4*>(h->pack);
  pack_kernel<<<gr, kCellBlock, 0, st>>>(g, in, in + 3 * n3, pk);
  float4* acc = reinterpret_cast<float4*>(h->acc);
  cudaMemsetAsync(acc, 0, sizeof(float4) * n3, st);
  advect_t_kernel<<<gr, kCellBlock, 0, st>>>(g, pk, h->nbr, h->adj2, h->adj2 + 3 * n3, acc);
  finish_t_kernel<<<gr, kCellBlock, 0, st>>>(g, acc, h->nbr, h->adj, h->adj + 3 * n3);
  return 7 + swept;
}

sim_status run_graph(gas_h h, std::vector<cudaGraphExec_t>& cache, std::vector<long long>& counts, int s,
                     long long (*enq)(gas_h, int, cudaStream_t)) {
  if (!cache[s]) {
    const cudaError_t e =
        mpm::capture_graph(h->cstream, 0, [&](cudaStream_t cs) { counts[s] = enq(h, s, cs); }, &cache[s]);
    if (e != cudaSuccess) {
      cudaGetLastError();  // reported here
      return gcuda(h, e, "gas graph capture");
    }
  }
  cudaError_t e = cudaGraphLaunch(cache[s], h->stream);
  if (e != cudaSuccess) return gcuda(h, e, "gas graph launch");
  h->launches += counts[s];
  return SIM_OK;
}

// Wait for the stream. Where sweeps go in pairs, whose waits are bounded, the error
// word comes to pinned memory before it (to pageable memory, and for every solver, the
// five calls of a 24^3 pass took 237 us instead of 205).
sim_status sync(gas_h h, const char* where) {
  cudaError_t e = cudaSuccess;
  if (h->word) e = cudaMemcpyAsync(h->word, h->err, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
  const cudaError_t es = cudaStreamSynchronize(h->stream);
  if (e == cudaSuccess) e = es;
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return gcuda(h, e, where);
  if (h->word && *h->word) {
    cudaMemset(h->err, 0, sizeof(int));
    return gfail(h, SIM_E_TIMEOUT, std::string(where) + ": device wait timed out");
  }
  return SIM_OK;
}

cudaError_t copy_in(gas_h h, void* dst, const void* src, size_t bytes, int on_device) {
  return cudaMemcpyAsync(dst, src, bytes, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, h->stream);
}

cudaError_t copy_out(gas_h h, void* dst, const void* src, size_t bytes, int on_device) {
  return cudaMemcpyAsync(dst, src, bytes, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, h->stream);
}

}  // namespace

extern "C" {

sim_status gas_create(const gas_config* cfg, const uint8_t* solid, gas_h* out) {
  if (!cfg || !solid || !out) return SIM_E_ARG;
  *out = nullptr;
  if (cfg->n < 8 || cfg->n > kMaxGrid || !(cfg->dt > 0.0f) || cfg->jacobi_iters < 1 || cfg->max_steps < 1) return SIM_E_ARG;
  gas_h h = new mpm_gas();
  h->cfg = *cfg;
  const int n = cfg->n;
  Geo& g = h->g;
  g.n = n;
  g.n3 = (long long)n * n * n;
  g.dx = 1.0f / n;
  g.dt_dx = cfg->dt * n;
  g.beta_dt = cfg->dt * cfg->buoyancy;
  g.inv2dx = 0.5f * n;
  h->stream = static_cast<cudaStream_t>(cfg->cuda_stream);
  const size_t n3 = (size_t)g.n3;
  for (size_t c = 0; c < n3; ++c) h->nfluid += solid[c] ? 0 : 1;
  int dev = 0;
  bool ok = cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
  ok = ok && cudaStreamCreateWithFlags(&h->cstream, cudaStreamNonBlocking) == cudaSuccess;
  ok = ok && cudaMalloc(&h->solid, n3) == cudaSuccess;
  ok = ok && cudaMalloc(&h->nbr, n3) == cudaSuccess;
  ok = ok && cudaMalloc(&h->states, sizeof(float) * 4 * n3 * (size_t)(cfg->max_steps + 1)) == cudaSuccess;
  float** bufs[8] = {&h->un, &h->b, &h->p0, &h->p1, &h->adj, &h->adj2, &h->acc, &h->pack};
  const size_t sizes[8] = {3 * n3, n3, n3, n3, 4 * n3, 4 * n3, 4 * n3, 4 * n3};
  for (int q = 0; q < 8 && ok; ++q) ok = cudaMalloc(bufs[q], sizeof(float) * sizes[q]) == cudaSuccess;
  ok = ok && cudaMalloc(&h->sum, sizeof(double)) == cudaSuccess;
  ok = ok && cudaMalloc(&h->mean, sizeof(float)) == cudaSuccess;
  if (ok && n % 4 == 0 && n >= kPairFrom)
    ok = cudaMalloc(&h->err, sizeof(int)) == cudaSuccess && cudaMemset(h->err, 0, sizeof(int)) == cudaSuccess &&
         cudaMallocHost(&h->word, sizeof(int)) == cudaSuccess &&
         cudaFuncSetAttribute(jacobi2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              pair_smem_limit(h->sms)) == cudaSuccess;
  ok = ok && cudaMemcpy(h->solid, solid, n3, cudaMemcpyHostToDevice) == cudaSuccess;
  if (ok) {
    neighbours_kernel<<<cell_grid(n), kCellBlock>>>(n, h->solid, h->nbr);
    ok = cudaDeviceSynchronize() == cudaSuccess;
  }
  if (!ok) {
    cudaGetLastError();
    gas_destroy(h);
    return SIM_E_OOM;
  }
  h->fwd.assign(cfg->max_steps, nullptr);
  h->bwd.assign(cfg->max_steps, nullptr);
  h->fwd_launches.assign(cfg->max_steps, 0);
  h->bwd_launches.assign(cfg->max_steps, 0);
  *out = h;
  return SIM_OK;
}

sim_status gas_destroy(gas_h h) {
  if (!h) return SIM_OK;
  if (h->stream) cudaStreamSynchronize(h->stream);
  for (auto e : h->fwd)
    if (e) cudaGraphExecDestroy(e);
  for (auto e : h->bwd)
    if (e) cudaGraphExecDestroy(e);
  void* ptrs[14] = {h->solid, h->nbr, h->states, h->un, h->b, h->p0, h->p1, h->adj, h->adj2, h->acc, h->sum,
                    h->mean, h->pack, h->err};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (h->word) cudaFreeHost(h->word);
  if (h->cstream) cudaStreamDestroy(h->cstream);
  delete h;
  return SIM_OK;
}

sim_status gas_set_state(gas_h h, const float* u, const float* d, int on_device) {
  if (!h) return SIM_E_ARG;
  if (!u || !d) return gfail(h, SIM_E_ARG, "gas_set_state: null u or d");
  const long long n3 = h->g.n3;
  float* s0 = state_ptr(h, 0);
  cudaError_t e = copy_in(h, s0, u, sizeof(float) * 3 * n3, on_device);
  if (e == cudaSuccess) e = copy_in(h, s0 + 3 * n3, d, sizeof(float) * n3, on_device);
  if (e != cudaSuccess) return gcuda(h, e, "gas_set_state");
  mask_kernel<<<cell_grid(h->g.n), kCellBlock, 0, h->stream>>>(h->g, h->nbr, s0);
  cudaMemsetAsync(h->adj, 0, sizeof(float) * 4 * n3, h->stream);
  h->launches += 1;
  h->step = 0;
  h->started = true;
  h->seeds = false;
  return sync(h, "gas_set_state");
}

sim_status gas_step(gas_h h, int n_steps) {
  if (!h) return SIM_E_ARG;
  if (!h->started) return gfail(h, SIM_E_STATE, "gas_step: no state set");
  if (n_steps < 0 || h->step + n_steps > h->cfg.max_steps) return gfail(h, SIM_E_ARG, "gas_step: beyond max_steps");
  for (int q = 0; q < n_steps; ++q) {
    sim_status st = run_graph(h, h->fwd, h->fwd_launches, h->step, enqueue_forward);
    if (st != SIM_OK) return st;
    ++h->step;
  }
  return sync(h, "gas_step");
}

sim_status gas_get_state(gas_h h, float* u, float* d, int on_device) {
  if (!h) return SIM_E_ARG;
  if (!h->started) return gfail(h, SIM_E_STATE, "gas_get_state: no state set");
  const long long n3 = h->g.n3;
  const float* s = state_ptr(h, h->step);
  cudaError_t e = cudaSuccess;
  if (u) e = copy_out(h, u, s, sizeof(float) * 3 * n3, on_device);
  if (e == cudaSuccess && d) e = copy_out(h, d, s + 3 * n3, sizeof(float) * n3, on_device);
  if (e != cudaSuccess) return gcuda(h, e, "gas_get_state");
  return sync(h, "gas_get_state");
}

sim_status gas_add_grad(gas_h h, const float* dLdu, const float* dLdd, int on_device) {
  if (!h) return SIM_E_ARG;
  if (!h->started) return gfail(h, SIM_E_STATE, "gas_add_grad: no state set");
  const long long n3 = h->g.n3;
  const float* src[2] = {dLdu, dLdd};
  const long long cnt[2] = {3 * n3, n3};
  const long long off[2] = {0, 3 * n3};
  for (int q = 0; q < 2; ++q) {
    if (!src[q]) continue;
    cudaError_t e = copy_in(h, h->acc, src[q], sizeof(float) * cnt[q], on_device);
    if (e != cudaSuccess) return gcuda(h, e, "gas_add_grad");
    add_kernel<<<nblocks(cnt[q]), kThreads, 0, h->stream>>>(cnt[q], h->acc, h->adj + off[q]);
    h->launches += 1;
  }
  h->seeds = true;
  return sync(h, "gas_add_grad");
}

sim_status gas_backward(gas_h h, float* dLdu0, float* dLdd0, int on_device) {
  if (!h) return SIM_E_ARG;
  if (!h->started || h->step == 0) return gfail(h, SIM_E_STATE, "gas_backward: no step taken");
  for (int s = h->step - 1; s >= 0; --s) {
    sim_status st = run_graph(h, h->bwd, h->bwd_launches, s, enqueue_backward);
    if (st != SIM_OK) return st;
  }
  const long long n3 = h->g.n3;
  cudaError_t e = cudaSuccess;
  if (dLdu0) e = copy_out(h, dLdu0, h->adj, sizeof(float) * 3 * n3, on_device);
  if (e == cudaSuccess && dLdd0) e = copy_out(h, dLdd0, h->adj + 3 * n3, sizeof(float) * n3, on_device);
  if (e != cudaSuccess) return gcuda(h, e, "gas_backward");
  cudaMemsetAsync(h->adj, 0, sizeof(float) * 4 * n3, h->stream);
  h->seeds = false;
  return sync(h, "gas_backward");
}

long long gas_kernel_launches(gas_h h) { return h ? h->launches : 0; }

const char* gas_last_error(gas_h h) { return h ? h->last_error.c_str() : "null gas handle"; }

}  // extern "C"
