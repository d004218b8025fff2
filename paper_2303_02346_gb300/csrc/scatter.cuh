// Particle-to-grid scatter, one warp at a time.
//
// The particle sort keeps the particles of a cell (stencil origin) together, so
// the 32 particles of a warp lie in a few cells. A warp
//   1. writes each particle's record (fractional position f and the
//      coefficients of its per-node contribution) to its own shared memory;
//   2. finds the particles of equal cell (match_any over the stencil origin's
//      node index);
//   3. takes three cells at a time, each with 9 lanes (a, b) = column of the
//      stencil: a lane sums the contributions of the cell's particles to its
//      column's three nodes in registers, reading the records as broadcasts,
//      and adds the four values of each node with one global vector reduction.
// No step needs another warp: there is no barrier, no zeroing and no size limit,
// and the work of one warp overlaps the load latency of the others. A particle
// of a warp that spans cells of any distance (or scenes) takes the same path.
//
// What bounds it: the instruction issue and load latency of the kernels around
// it; the reductions (18 sectors per cell and warp) keep L2 below a fifth of
// its rate. It replaced a shared-memory tile per CTA (cells binned and scanned
// by the CTA, one shared FP32 atomic per cell, node and value, a flush, nine
// barriers). Per launch on the 2M-particle dam break: fused step 237 -> 148 us
// (215 at the tile's best launch shape), G2P adjoint 234 -> 147 (213), P2G
// 190 -> 113; on the 200k-particle scene 35.6 -> 24.9, 33.5 -> 23.3 and
// 30.9 -> 19.9. One cell at a time with a lane per node measured 160 and 154
// us in place of 148 and 147: each lane then repeats the column's weights.
//
// The contribution of a particle with coefficients (c, M) to node x_i at
// offset dpos = x_i - x_p = (o - f) dx (o = the node's offset in the stencil,
// f = the particle's fractional position) is  W * (c + M dpos)  per value;
// P2G's first value (mass) has no dpos term. The record stores the same
// affine map in the node offset o: c + M dpos = c' + M' o with M' = M dx and
// c' = c - M' f, so that step 3 needs no per-particle offset arithmetic.
#pragma once

#include <climits>

#include "common.cuh"

namespace mpm {

constexpr int kRecF4 = 5;  // float4 per particle record: 4 used, the fifth keeps 16-byte stores free of bank conflicts
// Resident threads per SM that the G2P adjoint is compiled for, 3 CTAs of 256 or 6 of
// 128 (80 registers a thread; the fused step, left to the compiler, takes 80 to
// 104), and, as a launch choice for both, 4 CTAs of 256 or 8 of 128 (64 registers).
constexpr int kScatterResidentThreads = 768;
constexpr int kScatterResidentThreadsHigh = 1024;

// NT = threads per CTA = particles per CTA (one each)
template <int NT>
struct alignas(16) ScatterSmem {
  float4 rec[NT * kRecF4];
};

// Quadratic B-spline weight of stencil offset o as a polynomial in the
// fractional position f in [0.5, 1.5): w_o(f) = k0 + k1 f + k2 f^2, from
// w_0 = (1.5 - f)^2 / 2, w_1 = 3/4 - (f - 1)^2, w_2 = (f - 0.5)^2 / 2.
__device__ inline void spline_poly(int o, float& k0, float& k1, float& k2) {
  k0 = o == 0 ? 1.125f : (o == 1 ? -0.25f : 0.125f);
  k1 = o == 0 ? -1.5f : (o == 1 ? 2.0f : -0.5f);
  k2 = o == 1 ? -1.0f : 0.5f;
}

// Activate grid block b: the first caller to set its flag appends it to the
// active-block list (the grid update clears the flag again).
__device__ inline void activate_block(int* __restrict__ flags, int* __restrict__ list,
                                      int* __restrict__ count, long long b) {
  if (flags[b] == 0 && atomicExch(&flags[b], 1) == 0) list[atomicAdd(count, 1)] = int(b);
}

// Activate the blocks of one cell's stencil.
__device__ inline void mark_stencil_blocks(const Params& P, int scene, const int* base,
                                           int* __restrict__ flags, int* __restrict__ list,
                                           int* __restrict__ count) {
  int b0[3], b1[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    b0[d] = base[d] / kBlockEdge;
    b1[d] = (base[d] + 2) / kBlockEdge;
  }
  for (int bx = b0[0]; bx <= b1[0]; ++bx)
    for (int by = b0[1]; by <= b1[1]; ++by)
      for (int bz = b0[2]; bz <= b1[2]; ++bz)
        activate_block(flags, list, count, (long long)scene * P.NB + (bx * P.nb + by) * P.nb + bz);
}

// Activate the grid blocks that the stencils of a warp's cells touch (every
// lane must call it; leaders: the lanes that hold one cell each). If the cells
// share a scene and the blocks around them form a box of at most 12, one lane
// marks each block of the box, so that a single load tests them all; a warp
// spread wider marks cell by cell. (One lane per cell walking its up to 8
// blocks put as many dependent loads in a row.)
__device__ inline void mark_warp_blocks(const Params& P, unsigned leaders, bool leader, int scene, const int* base,
                                        int* __restrict__ flags, int* __restrict__ list, int* __restrict__ count) {
  constexpr unsigned kAll = 0xffffffffu;
  if (leaders == 0u) return;
  int lo[3], nb[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    lo[d] = __reduce_min_sync(kAll, leader ? base[d] : INT_MAX) / kBlockEdge;
    nb[d] = (__reduce_max_sync(kAll, leader ? base[d] : 0) + 2) / kBlockEdge - lo[d] + 1;
  }
  const int smin = __reduce_min_sync(kAll, leader ? scene : INT_MAX);
  const int smax = __reduce_max_sync(kAll, leader ? scene : 0);
  // each factor is at least 1 and at most 256
  const int yz = nb[1] * nb[2], total = nb[0] * yz;
  if (smin == smax && total <= 12) {
    const int lane = threadIdx.x & 31;
    if (lane < total) {
      const int tx = lane / yz, r = lane - tx * yz, ty = r / nb[2];
      activate_block(flags, list, count, (long long)smin * P.NB +
                                             ((lo[0] + tx) * P.nb + lo[1] + ty) * P.nb + lo[2] + r - ty * nb[2]);
    }
  } else if (leader) {
    mark_stencil_blocks(P, scene, base, flags, list, count);
  }
}

// Scatter of the warp's particles (every lane must call it). rec: the warp's
// 32 records. valid: this lane holds a particle with stencil sc in `scene`, mass
// value cm (kMass) and coefficients c' (cp) and M' (Md, row-major 3 x 3) in
// node-offset form. The values travel as v0 (with the mass beside it) and the
// pair (v1, v2) through packed two-lane FP32 fused multiply-adds (per lane the
// rounding of the scalar fmaf). flags (nullable): activates the grid blocks
// the stencils touch.
template <bool kMass>
__device__ inline void warp_scatter(float4* rec, const Params& P, bool valid, int scene, const Stencil& sc, float cm,
                                    const float* cp, const float* Md, float4* __restrict__ grid,
                                    int* __restrict__ flags, int* __restrict__ list, int* __restrict__ count) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  // node index of the stencil origin (all scenes' nodes number fewer than 2^31)
  const int key = valid ? int(node_index(P, scene, sc.base[0], sc.base[1], sc.base[2])) : -1;
  if (valid) {
    float4* r = rec + lane * kRecF4;
    r[0] = make_float4(sc.f[0], sc.f[1], sc.f[2], cm);
    r[1] = make_float4(cp[0], Md[0], Md[1], Md[2]);
    r[2] = make_float4(cp[1], cp[2], Md[3], Md[6]);
    r[3] = make_float4(Md[4], Md[7], Md[5], Md[8]);
  }
  const unsigned peers = __match_any_sync(kAll, key);
  const bool leader = valid && (peers & ((1u << lane) - 1u)) == 0u;
  unsigned leaders = __ballot_sync(kAll, leader);
  __syncwarp();  // the records are written
  if (flags) mark_warp_blocks(P, leaders, leader, scene, sc.base, flags, list, count);
  // this lane's column (a, b) of the stencil and the column's weight polynomials
  const int sub = lane / 9, col = lane - 9 * sub;
  const int oa = col / 3, ob = col - 3 * oa;
  float ka0, ka1, ka2, kb0, kb1, kb2;
  spline_poly(oa, ka0, ka1, ka2);
  spline_poly(ob, kb0, kb1, kb2);
  const float2 k0 = make_float2(ka0, kb0), k1 = make_float2(ka1, kb1), k2 = make_float2(ka2, kb2);
  const float fa = float(oa), fb = float(ob);
  const float2 fa2 = make_float2(fa, fa), fb2 = make_float2(fb, fb);
  const int off = (oa * P.n + ob) * P.n;
  while (leaders) {
    // the next three cells, one per group of 9 lanes
    const unsigned rest1 = leaders & (leaders - 1u), rest2 = rest1 & (rest1 - 1u);
    const unsigned mine = sub == 0 ? leaders : sub == 1 ? rest1 : sub == 2 ? rest2 : 0u;
    const int l = mine ? __ffs(mine) - 1 : lane;
    unsigned m = __shfl_sync(kAll, peers, l);
    const int node = __shfl_sync(kAll, key, l);
    leaders = rest2 & (rest2 - 1u);
    if (!mine) m = 0u;
    float2 s01[3], s23[3];  // (mass, v0), (v1, v2) at the column's nodes c = 0, 1, 2
#pragma unroll
    for (int c = 0; c < 3; ++c) s01[c] = s23[c] = make_float2(0.0f, 0.0f);
    while (m) {
      const float4* r = rec + (__ffs(m) - 1) * kRecF4;
      m &= m - 1u;
      const float4 r0 = r[0], r1 = r[1], r2 = r[2], r3 = r[3];
      const float2 fxy = make_float2(r0.x, r0.y), fz = make_float2(r0.z, r0.z);
      const float2 wab = __ffma2_rn(__ffma2_rn(k2, fxy, k1), fxy, k0);  // (w_x(a), w_y(b))
      const float wxy = wab.x * wab.y;
      // z weights of offsets 0 and 1; the third is 1 minus their sum. f is a grid
      // coordinate less a whole number, a multiple of 2^-22 from the third cell
      // on: there the inner step is exact, and the polynomial is rounded once, to
      // the very bits of the stencil's (1.5 - f)^2 / 2 and 3/4 - (f - 1)^2.
      const float2 wz = __ffma2_rn(__ffma2_rn(make_float2(0.5f, -1.0f), fz, make_float2(-1.5f, 2.0f)), fz,
                                   make_float2(1.125f, -0.25f));
      const float2 W01 = __fmul2_rn(make_float2(wxy, wxy), wz);
      const float W[3] = {W01.x, W01.y, wxy - W01.x - W01.y};
      // values at c = 0, stepped by the third column of M' per node
      float v0 = fmaf(r1.z, fb, fmaf(r1.y, fa, r1.x));
      float2 v12 = __ffma2_rn(make_float2(r3.x, r3.y), fb2,
                              __ffma2_rn(make_float2(r2.z, r2.w), fa2, make_float2(r2.x, r2.y)));
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float2 w2 = make_float2(W[c], W[c]);
        if (kMass)
          s01[c] = __ffma2_rn(w2, make_float2(r0.w, v0), s01[c]);
        else
          s01[c].y = fmaf(W[c], v0, s01[c].y);
        s23[c] = __ffma2_rn(w2, v12, s23[c]);
        if (c < 2) {
          v0 += r1.w;
          v12 = __fadd2_rn(v12, make_float2(r3.z, r3.w));
        }
      }
    }
    if (mine) {
      float4* g = grid + node + off;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (kMass)
          red_add_v4(g + c, s01[c].x, s01[c].y, s23[c].x, s23[c].y);
        else
          red_add_v4(g + c, s01[c].y, s23[c].x, s23[c].y, 0.0f);
      }
    }
    __syncwarp();
  }
}

}  // namespace mpm
