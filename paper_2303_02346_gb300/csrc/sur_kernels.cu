// Surrogate kernels other than the tensor-core convolution and its weight
// gradient: weight layout preparation, grid features and their velocity
// adjoint, the 1x1x1 lift and projection (with loss, gradients and error
// sums), the lift backward, and Adam.
#include <cuda_bf16.h>

#include <algorithm>

#include "sur_kernels.h"

namespace sur {
namespace {

__device__ __forceinline__ void unpack8(const uint4& u, float (&f)[8]) {
  const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float2 t = __bfloat1622float2(p[i]);
    f[2 * i] = t.x;
    f[2 * i + 1] = t.y;
  }
}

__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
  uint4 u;
  __nv_bfloat162* p = reinterpret_cast<__nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) p[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
  return u;
}

__device__ __forceinline__ float rbf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// offsets into the flat parameter vector
__host__ __device__ inline long long conv_w_offset(int layer) {  // layer = 2 * block + (0: w1, 1: w2)
  return 288ll + static_cast<long long>(layer / 2) * 2 * (27 * 1024 + 32) + (layer % 2) * (27 * 1024 + 32);
}

// ---------------------------------------------------------------------------
// weights: FP32 master W[a][b][c][o][q] -> the BF16 UMMA A layout of the
// convolution (sur_conv.cu), [row c*32 + o][pair a*3+b][q]; the
// backward layout holds the mirrored taps with the channel roles swapped,
// W'[2-a][2-b][2-c][q][o] = W[a][b][c][o][q] (the input gradient of conv3 is
// conv3 of the output gradient with these weights). Rows 96..127 of every
// pair stay zero (set once at allocation).
// ---------------------------------------------------------------------------
__global__ void prep_weights_kernel(const float* params, int layers, __nv_bfloat16* wf, __nv_bfloat16* wb) {
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (i >= static_cast<long long>(layers) * 27 * 1024) return;
  const int L = static_cast<int>(i / (27 * 1024));
  const int rem = static_cast<int>(i % (27 * 1024));
  const int tap = rem / 1024, o = (rem / 32) % 32, q = rem % 32;
  const int pair = tap / 3, c = tap % 3;
  const int tapm = 26 - tap, pairm = tapm / 3, cm = tapm % 3;
  const __nv_bfloat16 w = __float2bfloat16_rn(params[conv_w_offset(L) + rem]);
  const long long base = static_cast<long long>(L) * kConvWElems;
  wf[base + ((c * 32 + o) * 9 + pair) * 32 + q] = w;
  wb[base + ((cm * 32 + q) * 9 + pairm) * 32 + o] = w;
}

// ---------------------------------------------------------------------------
// grid features: MLS-MPM quadratic B-spline transfer of m, m (v + C dpos) and
// the per-material mass, then normalisation and BF16 rounding.
// ---------------------------------------------------------------------------
struct Stencil {
  int base[3];
  float w[3][3];
  float fx[3];
};

__device__ __forceinline__ bool make_stencil(const float* x, int n, Stencil& s) {
  bool ok = true;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float xs = x[d] * n;
    const int b = static_cast<int>(floorf(xs - 0.5f));
    // one rounding, of f itself: x n rounded first would leave an error of its
    // own size in f wherever n is not a power of two (adjoint at n = 45: 1.4e-6
    // against 1.3e-7), and whether the compiler fuses the two is its own choice
    const float f = __fmaf_rn(x[d], static_cast<float>(n), -static_cast<float>(b));
    s.base[d] = b;
    s.fx[d] = f;
    s.w[0][d] = 0.5f * (1.5f - f) * (1.5f - f);
    s.w[1][d] = 0.75f - (f - 1.0f) * (f - 1.0f);
    s.w[2][d] = 0.5f * (f - 0.5f) * (f - 0.5f);
    ok = ok && b >= 0 && b <= n - 3;
  }
  return ok;
}

// four consecutive floats (16-byte aligned) reduced into memory at once
__device__ __forceinline__ void red_add_v4(float* addr, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d)
               : "memory");
}

// Bound by L2's reductions (the caller's particle order is arbitrary, so the 27
// nodes of neighbouring threads share nothing): the mass and the momentum go
// out as one vector reduction, the material's mass as a scalar, 2 a node
// instead of 5 (100k particles on 64^3: 124 -> 47 us).
__global__ void features_scatter_kernel(FeatArgs a, const float* __restrict__ x, const float* __restrict__ v,
                                        const float* __restrict__ C, const uint8_t* __restrict__ mat,
                                        float* acc, int* err) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= a.N) return;
  float xp[3] = {x[3 * p], x[3 * p + 1], x[3 * p + 2]};
  Stencil s;
  if (!make_stencil(xp, a.n, s)) {
    atomicOr(err, kErrDomain);
    return;
  }
  const int mt = mat[p];
  if (mt >= a.n_mat) {
    atomicOr(err, kErrArg);
    return;
  }
  const float mp = a.mmass[mt];
  float vp[3] = {v[3 * p], v[3 * p + 1], v[3 * p + 2]};
  float Cp[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) Cp[i] = C[9 * p + i];
  const float dx = 1.0f / a.n;
  const int n = a.n;
#pragma unroll
  for (int oi = 0; oi < 3; ++oi)
#pragma unroll
    for (int oj = 0; oj < 3; ++oj)
#pragma unroll
      for (int ok = 0; ok < 3; ++ok) {
        const float W = s.w[oi][0] * s.w[oj][1] * s.w[ok][2];
        const float d0 = (oi - s.fx[0]) * dx, d1 = (oj - s.fx[1]) * dx, d2 = (ok - s.fx[2]) * dx;
        const float wm = W * mp;
        const long long node =
            (static_cast<long long>(s.base[0] + oi) * n + (s.base[1] + oj)) * n + (s.base[2] + ok);
        float* dst = acc + node * 8;
        red_add_v4(dst, wm, wm * (vp[0] + Cp[0] * d0 + Cp[1] * d1 + Cp[2] * d2),
                   wm * (vp[1] + Cp[3] * d0 + Cp[4] * d1 + Cp[5] * d2),
                   wm * (vp[2] + Cp[6] * d0 + Cp[7] * d1 + Cp[8] * d2));
        if (mt < 3) atomicAdd(dst + 4 + mt, wm);
      }
}

__global__ void features_finalize_kernel(FeatArgs a, float* acc, uint16_t* frame) {
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  const long long n3 = static_cast<long long>(a.n) * a.n * a.n;
  if (i >= n3) return;
  float4* src = reinterpret_cast<float4*>(acc + i * 8);
  const float4 u = src[0], w = src[1];
  float o[8];
  const float m = u.x;
  o[0] = m * a.inv_mref;
  o[1] = u.y * a.inv_mvref;
  o[2] = u.z * a.inv_mvref;
  o[3] = u.w * a.inv_mvref;
  const float inv = m > 0.0f ? 1.0f / m : 0.0f;
  o[4] = w.x * inv;
  o[5] = w.y * inv;
  o[6] = w.z * inv;
  o[7] = 0.0f;
  reinterpret_cast<uint4*>(frame)[i] = pack8(o);
  src[0] = make_float4(0.f, 0.f, 0.f, 0.f);
  src[1] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// Adjoint of the mass and momentum channels of the transfer, for a cotangent
// g (FP32 [n^3][8]; channels 4..7 are not differentiated): with s = m_p /
// (m_ref v_ref), d = x_i - x_p and grad W the B-spline weight gradient,
//   dL/dv_p = s sum_i W g_i[1:4]
//   dL/dC_p = s sum_i W g_i[1:4] d^T
//   dL/dx_p = sum_i (s g_i[1:4] . (v_p + C_p d) + g_i[0] m_p / m_ref) grad W - s W C_p^T g_i[1:4]
__global__ void features_vjp_kernel(FeatArgs a, const float* __restrict__ x, const float* __restrict__ v,
                                    const float* __restrict__ C, const uint8_t* __restrict__ mat,
                                    const float* __restrict__ g, float* dLdx, float* dLdv, float* dLdC, int* err) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= a.N) return;
  float xp[3] = {x[3 * p], x[3 * p + 1], x[3 * p + 2]};
  Stencil st;
  if (!make_stencil(xp, a.n, st) || mat[p] >= a.n_mat) {
    atomicOr(err, kErrDomain);
    if (dLdx) dLdx[3 * p] = dLdx[3 * p + 1] = dLdx[3 * p + 2] = 0.0f;
    if (dLdv) dLdv[3 * p] = dLdv[3 * p + 1] = dLdv[3 * p + 2] = 0.0f;
    if (dLdC)
      for (int k = 0; k < 9; ++k) dLdC[9 * p + k] = 0.0f;
    return;
  }
  const float mp = a.mmass[mat[p]];
  const float sm = mp * a.inv_mvref, smass = mp * a.inv_mref;
  const float dx = 1.0f / a.n, inv_dx = static_cast<float>(a.n);
  float vp[3] = {0.f, 0.f, 0.f}, Cp[9];
  if (v) {
    vp[0] = v[3 * p];
    vp[1] = v[3 * p + 1];
    vp[2] = v[3 * p + 2];
  }
#pragma unroll
  for (int k = 0; k < 9; ++k) Cp[k] = C ? C[9 * p + k] : 0.0f;
  // B-spline weight derivatives w.r.t. f (= x inv_dx - base)
  float dw[3][3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float f = st.fx[d];
    dw[0][d] = -(1.5f - f);
    dw[1][d] = -2.0f * (f - 1.0f);
    dw[2][d] = f - 0.5f;
  }
  const int n = a.n;
  float gv[3] = {0.f, 0.f, 0.f}, gC[9], gx[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < 9; ++k) gC[k] = 0.0f;
#pragma unroll
  for (int oi = 0; oi < 3; ++oi)
#pragma unroll
    for (int oj = 0; oj < 3; ++oj)
#pragma unroll
      for (int ok = 0; ok < 3; ++ok) {
        const float W = st.w[oi][0] * st.w[oj][1] * st.w[ok][2];
        const float gW[3] = {dw[oi][0] * st.w[oj][1] * st.w[ok][2] * inv_dx,
                             st.w[oi][0] * dw[oj][1] * st.w[ok][2] * inv_dx,
                             st.w[oi][0] * st.w[oj][1] * dw[ok][2] * inv_dx};
        const float d[3] = {(oi - st.fx[0]) * dx, (oj - st.fx[1]) * dx, (ok - st.fx[2]) * dx};
        const long long node =
            (static_cast<long long>(st.base[0] + oi) * n + (st.base[1] + oj)) * n + (st.base[2] + ok);
        const float* gn = g + node * 8;
        const float g0 = gn[0], gm[3] = {gn[1], gn[2], gn[3]};
        float mom[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) mom[r] = vp[r] + Cp[3 * r] * d[0] + Cp[3 * r + 1] * d[1] + Cp[3 * r + 2] * d[2];
        const float coef = sm * (gm[0] * mom[0] + gm[1] * mom[1] + gm[2] * mom[2]) + g0 * smass;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          gx[c] += coef * gW[c] - sm * W * (Cp[c] * gm[0] + Cp[3 + c] * gm[1] + Cp[6 + c] * gm[2]);
          gv[c] += sm * W * gm[c];
        }
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
          for (int c = 0; c < 3; ++c) gC[3 * r + c] += sm * W * gm[r] * d[c];
      }
  if (dLdx)
    for (int c = 0; c < 3; ++c) dLdx[3 * p + c] = gx[c];
  if (dLdv)
    for (int c = 0; c < 3; ++c) dLdv[3 * p + c] = gv[c];
  if (dLdC)
    for (int k = 0; k < 9; ++k) dLdC[9 * p + k] = gC[k];
}

// (i, j, k) of node v = (i n + j) n + k of a frame: 32-bit divisions (a frame
// has n^3 < 2^32 nodes), far cheaper than 64-bit ones in these load-bound loops.
__device__ __forceinline__ void split_node(const SurGeom& g, long long v, int& i, int& j, int& k) {
  const unsigned n = static_cast<unsigned>(g.n), u = static_cast<unsigned>(v);
  const unsigned ij = u / n;
  k = static_cast<int>(u - ij * n);
  i = static_cast<int>(ij / n);
  j = static_cast<int>(ij - static_cast<unsigned>(i) * n);
}

// ---------------------------------------------------------------------------
// lift: h0 = bf16(W_l f + b_l) at every interior row. Memory moves 80 bytes a
// node; the weights' shared-memory loads were the bound (one word per product),
// so a thread reads the weights 16 bytes at a time and, where there are more nodes
// than threads, for two nodes (kTwo). 8 frames of 64^3: 46 -> 39 us; 3 frames of
// 40^3, where the second node would be none: 13.2 -> 12.5 us (15.3 with kTwo).
// ---------------------------------------------------------------------------
template <bool kTwo>
__global__ void __launch_bounds__(256) lift_kernel(SurGeom g, const uint16_t* __restrict__ frames,
                                                   const int* __restrict__ idx, const float* __restrict__ wl,
                                                   const float* __restrict__ bl, __nv_bfloat16* h0) {
  __shared__ float4 sw4[64 + 8];
  float* sw = reinterpret_cast<float*>(sw4);
  for (int i = threadIdx.x; i < 256 + 32; i += blockDim.x) sw[i] = i < 256 ? rbf(wl[i]) : bl[i - 256];
  __syncthreads();
  const int b = blockIdx.y;
  const long long n3 = static_cast<long long>(g.n) * g.n * g.n;
  const long long fr = idx ? idx[b] : b;
  const long long step = static_cast<long long>(gridDim.x) * blockDim.x;
  for (long long v0 = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; v0 < n3;
       v0 += (kTwo ? 2 : 1) * step) {
    const long long v1 = v0 + step;
    const bool two = kTwo && v1 < n3;
    const uint4 r0 = reinterpret_cast<const uint4*>(frames)[fr * n3 + v0];
    const uint4 r1 = two ? reinterpret_cast<const uint4*>(frames)[fr * n3 + v1] : r0;
    float f[2][8];
    unpack8(r0, f[0]);
    unpack8(r1, f[1]);
    int i, j, k;
    split_node(g, v0, i, j, k);
    const long long row0 = pad_row(g, b, i, j, k);
    split_node(g, two ? v1 : v0, i, j, k);
    const long long row1 = pad_row(g, b, i, j, k);
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
      float o0[8], o1[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int oc = c * 8 + e;
        const float4 wa = sw4[oc * 2], wb = sw4[oc * 2 + 1];
        const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
        float s0 = sw[256 + oc], s1 = s0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          s0 += w[q] * f[0][q];
          if (kTwo) s1 += w[q] * f[1][q];
        }
        o0[e] = s0;
        o1[e] = s1;
      }
      *reinterpret_cast<uint4*>(h0 + (c * g.plane + row0) * 8) = pack8(o0);
      if (two) *reinterpret_cast<uint4*>(h0 + (c * g.plane + row1) * 8) = pack8(o1);
    }
  }
}

// ---------------------------------------------------------------------------
// projection: pred = f[1:4] + W_p h + b_p, optionally with the loss, dL/dh
// (BF16), dL/dW_p, dL/db_p and per-frame error sums
// ---------------------------------------------------------------------------
constexpr int kProjThreads = 256;
constexpr int kRowWords = 17;  // words per node of a transposed channel row (16 of two BF16, one of padding)

// One thread per node. A warp's nodes are summed into dL/dW_p through a
// transpose in its own shared memory: each lane leaves its node's 32 channels
// there and takes one channel of all 32 nodes, so that a lane accumulates 3
// entries instead of 96 (which took 255 registers and spills); no barrier.
// The weights are read 16 bytes at a time. 8 frames of 64^3: training 170 -> 99
// us, inference 67 -> 46.
template <int MODE>
__global__ void __launch_bounds__(kProjThreads, (MODE & 2) ? 2 : (MODE & 4) ? 3 : 4) proj_kernel(SurGeom g, int batch,
                                                            const uint16_t* __restrict__ frames,
                                                            const int* __restrict__ idx,
                                                            const int* __restrict__ tgt,
                                                            const __nv_bfloat16* __restrict__ h,
                                                            const float* __restrict__ wp,
                                                            const float* __restrict__ bp, float* pred,
                                                            __nv_bfloat16* g_h, float* g_pred, float* grad_wp,
                                                            double* loss_acc, double* frame_sums) {
  constexpr bool want_grad = MODE & 2, want_sums = MODE & 4, given = MODE & 8;
  constexpr unsigned kAll = 0xffffffffu;
  __shared__ float4 sw4[24 + 1];
  __shared__ float red[kProjThreads / 32][101];
  __shared__ uint32_t rows[want_grad ? kProjThreads * kRowWords : 1];
  __shared__ float4 grads[want_grad ? kProjThreads : 1];
  float* sw = reinterpret_cast<float*>(sw4);
  for (int i = threadIdx.x; i < 99; i += blockDim.x) sw[i] = i < 96 ? rbf(wp[i]) : bp[i - 96];
  __syncthreads();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int b = blockIdx.y;
  const long long n3 = static_cast<long long>(g.n) * g.n * g.n;
  const long long fr = idx ? idx[b] : b;
  const long long ft = tgt ? tgt[b] : 0;
  const float inv_count = 1.0f / (static_cast<float>(batch) * static_cast<float>(n3) * 3.0f);
  float gw[3] = {0.f, 0.f, 0.f}, gb[3] = {0.f, 0.f, 0.f}, l2 = 0.f, t2 = 0.f;
  for (long long base = blockIdx.x * static_cast<long long>(blockDim.x); base < n3;
       base += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long vtx = base + threadIdx.x;
    const bool in = vtx < n3;
    float gp[3] = {0.f, 0.f, 0.f};
    uint4 raw[4] = {};
    if (in) {
      int i, j, k;
      split_node(g, vtx, i, j, k);
      const long long row = pad_row(g, b, i, j, k);
#pragma unroll
      for (int c = 0; c < 4; ++c) raw[c] = *reinterpret_cast<const uint4*>(h + (c * g.plane + row) * 8);
      const uint4 fraw = reinterpret_cast<const uint4*>(frames)[fr * n3 + vtx];
      float p[3] = {sw[96], sw[97], sw[98]};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float hv[8];
        unpack8(raw[c], hv);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const float4 wa = sw4[m * 8 + c * 2], wb = sw4[m * 8 + c * 2 + 1];
          const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
          for (int e = 0; e < 8; ++e) p[m] += w[e] * hv[e];
        }
      }
      float f[8];
      unpack8(fraw, f);
#pragma unroll
      for (int m = 0; m < 3; ++m) p[m] = f[1 + m] + p[m];
      if (MODE & 1) {
        float* dst = pred + (static_cast<long long>(b) * n3 + vtx) * 3;
        dst[0] = p[0];
        dst[1] = p[1];
        dst[2] = p[2];
      }
      if (given) {
        // cotangent of the prediction supplied by the caller: dL/dh only
        const float* src = g_pred + (static_cast<long long>(b) * n3 + vtx) * 3;
#pragma unroll
        for (int m = 0; m < 3; ++m) gp[m] = src[m];
      }
      if (want_grad || want_sums) {
        float tf[8];
        unpack8(reinterpret_cast<const uint4*>(frames)[ft * n3 + vtx], tf);
        const float d[3] = {p[0] - tf[1], p[1] - tf[2], p[2] - tf[3]};
        l2 += d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
        t2 += tf[1] * tf[1] + tf[2] * tf[2] + tf[3] * tf[3];
        if (want_grad) {
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            gp[m] = 2.0f * d[m] * inv_count;
            gb[m] += gp[m];
          }
          if (g_pred) {
            float* dst = g_pred + (static_cast<long long>(b) * n3 + vtx) * 3;
            dst[0] = gp[0];
            dst[1] = gp[1];
            dst[2] = gp[2];
          }
        }
      }
      if (want_grad || given) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float4 a0 = sw4[c * 2], a1 = sw4[c * 2 + 1], b0 = sw4[8 + c * 2], b1 = sw4[8 + c * 2 + 1],
                       c0 = sw4[16 + c * 2], c1 = sw4[16 + c * 2 + 1];
          const float wa[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
          const float wb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
          const float wc[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
          float o8[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) o8[e] = wa[e] * gp[0] + wb[e] * gp[1] + wc[e] * gp[2];
          *reinterpret_cast<uint4*>(g_h + (c * g.plane + row) * 8) = pack8(o8);
        }
      }
    }
    if (want_grad) {
      // lanes past the last node leave zeros
      uint32_t* mine = rows + threadIdx.x * kRowWords;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        mine[c * 4] = raw[c].x;
        mine[c * 4 + 1] = raw[c].y;
        mine[c * 4 + 2] = raw[c].z;
        mine[c * 4 + 3] = raw[c].w;
      }
      grads[threadIdx.x] = make_float4(gp[0], gp[1], gp[2], 0.f);
      __syncwarp();
      const uint32_t* col = rows + warp * 32 * kRowWords + lane / 2;
      const float4* gr = grads + warp * 32;
      // pairwise over the 32 nodes, so that the running sum takes one rounding
      // per 32 nodes, as many as when each thread summed its own nodes
      float part[3] = {0.f, 0.f, 0.f};
#pragma unroll 1
      for (int r0 = 0; r0 < 32; r0 += 16) {
        float s[2][3];
#pragma unroll
        for (int o = 0; o < 2; ++o) {
          float p[4][3];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int r = r0 + o * 8 + u * 2;
            const uint32_t wa = col[r * kRowWords], wb = col[(r + 1) * kRowWords];
            const float ha = __uint_as_float((lane & 1) ? (wa & 0xffff0000u) : (wa << 16));
            const float hb = __uint_as_float((lane & 1) ? (wb & 0xffff0000u) : (wb << 16));
            const float4 qa = gr[r], qb = gr[r + 1];
            p[u][0] = fmaf(qb.x, hb, qa.x * ha);
            p[u][1] = fmaf(qb.y, hb, qa.y * ha);
            p[u][2] = fmaf(qb.z, hb, qa.z * ha);
          }
#pragma unroll
          for (int m = 0; m < 3; ++m) s[o][m] = (p[0][m] + p[1][m]) + (p[2][m] + p[3][m]);
        }
#pragma unroll
        for (int m = 0; m < 3; ++m) part[m] += s[0][m] + s[1][m];
      }
#pragma unroll
      for (int m = 0; m < 3; ++m) gw[m] += part[m];
      __syncwarp();
    }
  }
  if (want_grad) {
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      red[warp][m * 32 + lane] = gw[m];
      const float s = warp_sum(gb[m]);
      if (lane == 0) red[warp][96 + m] = s;
    }
  }
  const float sl = warp_sum(l2), st = warp_sum(t2);
  if (lane == 0) {
    red[warp][99] = sl;
    red[warp][100] = st;
  }
  __syncthreads();
  if (want_grad && threadIdx.x < 99) {
    float s = 0.f;
    for (int w = 0; w < kProjThreads / 32; ++w) s += red[w][threadIdx.x];
    atomicAdd(grad_wp + threadIdx.x, s);  // w_proj (96) and b_proj (3) are adjacent
  }
  if (threadIdx.x == 128 && (want_grad || want_sums)) {
    double s = 0.0, t = 0.0;
    for (int w = 0; w < kProjThreads / 32; ++w) {
      s += red[w][99];
      t += red[w][100];
    }
    if (want_grad) atomicAdd(loss_acc, s);
    if (want_sums) {
      atomicAdd(frame_sums + 2 * b, s);
      atomicAdd(frame_sums + 2 * b + 1, t);
    }
  }
}

// ---------------------------------------------------------------------------
// lift backward: dW_l, db_l and optionally dL/dframe. As in the projection, a
// warp's nodes pass through its own shared memory, and lane o sums the 8
// entries of output channel o (and its bias) over the 32 nodes: 3 shared loads
// for 9 sums, where one entry a thread took 2 loads a sum behind two barriers
// per 256 nodes. 8 frames of 64^3: 162 -> 60 us.
// ---------------------------------------------------------------------------
constexpr int kLbThreads = 256;

__global__ void __launch_bounds__(kLbThreads) lift_bwd_kernel(SurGeom g, int batch,
                                                              const uint16_t* __restrict__ frames,
                                                              const int* __restrict__ idx,
                                                              const __nv_bfloat16* __restrict__ gh,
                                                              const float* __restrict__ wl,
                                                              const float* __restrict__ g_pred, float* grad_wl,
                                                              float* grad_bl, float* g_frames) {
  __shared__ float4 sw4[64];  // read 16 bytes at a time
  __shared__ uint32_t rows[kLbThreads * kRowWords];
  __shared__ float4 sf[kLbThreads * 2];
  float* sw = reinterpret_cast<float*>(sw4);
  for (int i = threadIdx.x; i < 256; i += blockDim.x) sw[i] = rbf(wl[i]);
  __syncthreads();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int b = blockIdx.y;
  const long long n3 = static_cast<long long>(g.n) * g.n * g.n;
  const long long fr = idx ? idx[b] : b;
  float accw[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, accb = 0.f;
  const long long step = static_cast<long long>(gridDim.x) * blockDim.x;
  for (long long base = blockIdx.x * static_cast<long long>(blockDim.x); base < n3; base += step) {
    const long long vtx = base + threadIdx.x;
    uint4 raw[4] = {};  // lanes past the last node leave zeros
    float f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (vtx < n3) {
      int i, j, k;
      split_node(g, vtx, i, j, k);
      const long long row = pad_row(g, b, i, j, k);
#pragma unroll
      for (int c = 0; c < 4; ++c) raw[c] = *reinterpret_cast<const uint4*>(gh + (c * g.plane + row) * 8);
      unpack8(reinterpret_cast<const uint4*>(frames)[fr * n3 + vtx], f);
      if (g_frames) {
        float gf[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float gv[8];
          unpack8(raw[c], gv);
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float4 wa = sw4[(c * 8 + e) * 2], wb = sw4[(c * 8 + e) * 2 + 1];
            const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
            for (int q = 0; q < 8; ++q) gf[q] += w[q] * gv[e];
          }
        }
        const float* gp = g_pred + (static_cast<long long>(b) * n3 + vtx) * 3;
        gf[1] += gp[0];
        gf[2] += gp[1];
        gf[3] += gp[2];
        float4* dst = reinterpret_cast<float4*>(g_frames + (static_cast<long long>(b) * n3 + vtx) * 8);
        dst[0] = make_float4(gf[0], gf[1], gf[2], gf[3]);
        dst[1] = make_float4(gf[4], gf[5], gf[6], gf[7]);
      }
    }
    uint32_t* mine = rows + threadIdx.x * kRowWords;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      mine[c * 4] = raw[c].x;
      mine[c * 4 + 1] = raw[c].y;
      mine[c * 4 + 2] = raw[c].z;
      mine[c * 4 + 3] = raw[c].w;
    }
    sf[threadIdx.x * 2] = make_float4(f[0], f[1], f[2], f[3]);
    sf[threadIdx.x * 2 + 1] = make_float4(f[4], f[5], f[6], f[7]);
    __syncwarp();
    const uint32_t* col = rows + warp * 32 * kRowWords + lane / 2;
    const float4* fw = sf + warp * 64;
#pragma unroll 8
    for (int r = 0; r < 32; ++r) {
      const uint32_t w2 = col[r * kRowWords];
      const float gv = __uint_as_float((lane & 1) ? (w2 & 0xffff0000u) : (w2 << 16));
      const float4 a = fw[r * 2], c = fw[r * 2 + 1];
      accw[0] += gv * a.x;
      accw[1] += gv * a.y;
      accw[2] += gv * a.z;
      accw[3] += gv * a.w;
      accw[4] += gv * c.x;
      accw[5] += gv * c.y;
      accw[6] += gv * c.z;
      accw[7] += gv * c.w;
      accb += gv;
    }
    __syncwarp();
  }
  // over the CTA's warps, then one atomic per entry
  __syncthreads();
  float* red = reinterpret_cast<float*>(rows);  // 8 warps x 288
#pragma unroll
  for (int q = 0; q < 8; ++q) red[warp * 288 + lane * 8 + q] = accw[q];
  red[warp * 288 + 256 + lane] = accb;
  __syncthreads();
  for (int i = threadIdx.x; i < 288; i += blockDim.x) {
    float s = 0.f;
    for (int w = 0; w < kLbThreads / 32; ++w) s += red[w * 288 + i];
    if (i < 256)
      atomicAdd(grad_wl + i, s);
    else
      atomicAdd(grad_bl + i - 256, s);
  }
}

// ---------------------------------------------------------------------------
// Adam (Kingma and Ba 2015) with bias correction
// ---------------------------------------------------------------------------
__global__ void adam_kernel(float* p, const float* __restrict__ gr, float* m, float* v, long long count, float lr,
                            float b1, float b2, float eps, float c1, float c2) {
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (i >= count) return;
  const float gi = gr[i];
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace

cudaError_t launch_prep_weights(const float* params, int blocks, __nv_bfloat16* wf, __nv_bfloat16* wb,
                                cudaStream_t st) {
  const long long total = 2ll * blocks * 27 * 1024;
  prep_weights_kernel<<<static_cast<unsigned>((total + 255) / 256), 256, 0, st>>>(params, 2 * blocks, wf, wb);
  return cudaGetLastError();
}

cudaError_t launch_lift(const SurGeom& g, int batch, const uint16_t* frames, const int* idx, const float* w_lift,
                        const float* b_lift, __nv_bfloat16* h0, cudaStream_t st) {
  const long long n3 = static_cast<long long>(g.n) * g.n * g.n;
  dim3 grid(static_cast<unsigned>(std::min<long long>((n3 + 255) / 256, 256)), batch);
  if (n3 > 256 * 256)
    lift_kernel<true><<<grid, 256, 0, st>>>(g, frames, idx, w_lift, b_lift, h0);
  else
    lift_kernel<false><<<grid, 256, 0, st>>>(g, frames, idx, w_lift, b_lift, h0);
  return cudaGetLastError();
}

// Nodes a thread walks through: 8 where parameter gradients are summed (fewer
// atomics per entry). Elsewhere only as many as leave four CTAs for every SM: the
// walk is a chain of loads (prediction of 3 frames of 40^3: 23.6 us with 8 nodes,
// 12.3 with 2; of one frame of 24^3: 16.4 with 8, 8.0 with one).
cudaError_t launch_proj(const SurGeom& g, int batch, int num_sms, int mode, const uint16_t* frames, const int* idx,
                        const int* tgt, const __nv_bfloat16* h, const float* w_proj, const float* b_proj,
                        float* pred, __nv_bfloat16* g_h, float* g_pred, float* grad_wp, double* loss_acc,
                        double* frame_sums, cudaStream_t st) {
  const long long n3 = static_cast<long long>(g.n) * g.n * g.n;
  const long long fill = 4LL * num_sms * kProjThreads;
  const long long walk = (mode & 2) ? 8 : std::min<long long>(std::max<long long>((n3 * batch + fill - 1) / fill, 1), 8);
  dim3 grid(static_cast<unsigned>(std::min<long long>((n3 + kProjThreads * walk - 1) / (kProjThreads * walk), 512)),
            batch);
  switch (mode) {
    case 1:
      proj_kernel<1><<<grid, kProjThreads, 0, st>>>(g, batch, frames, idx, tgt, h, w_proj, b_proj, pred, g_h, g_pred,
                                                    grad_wp, loss_acc, frame_sums);
      break;
    case 2:
      proj_kernel<2><<<grid, kProjThreads, 0, st>>>(g, batch, frames, idx, tgt, h, w_proj, b_proj, pred, g_h, g_pred,
                                                    grad_wp, loss_acc, frame_sums);
      break;
    case 4:
      proj_kernel<4><<<grid, kProjThreads, 0, st>>>(g, batch, frames, idx, tgt, h, w_proj, b_proj, pred, g_h, g_pred,
                                                    grad_wp, loss_acc, frame_sums);
      break;
    case 8:
      proj_kernel<8><<<grid, kProjThreads, 0, st>>>(g, batch, frames, idx, tgt, h, w_proj, b_proj, pred, g_h, g_pred,
                                                    grad_wp, loss_acc, frame_sums);
      break;
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_lift_bwd(const SurGeom& g, int batch, const uint16_t* frames, const int* idx,
                            const __nv_bfloat16* g_h0, const float* w_lift, const float* g_pred, float* grad_wl,
                            float* grad_bl, float* g_frames, cudaStream_t st) {
  const long long n3 = static_cast<long long>(g.n) * g.n * g.n;
  dim3 grid(static_cast<unsigned>(std::min<long long>((n3 + kLbThreads - 1) / kLbThreads, 128)), batch);
  lift_bwd_kernel<<<grid, kLbThreads, 0, st>>>(g, batch, frames, idx, g_h0, w_lift, g_pred, grad_wl, grad_bl,
                                               g_frames);
  return cudaGetLastError();
}

cudaError_t launch_adam(float* p, const float* grad, float* m, float* v, long long count, float lr, float beta1,
                        float beta2, float eps, int t, cudaStream_t st) {
  const float c1 = 1.0f - powf(beta1, static_cast<float>(t));
  const float c2 = 1.0f - powf(beta2, static_cast<float>(t));
  adam_kernel<<<static_cast<unsigned>((count + 255) / 256), 256, 0, st>>>(p, grad, m, v, count, lr, beta1, beta2,
                                                                          eps, c1, c2);
  return cudaGetLastError();
}

cudaError_t launch_features(const FeatArgs& a, const float* x, const float* v, const float* C, const uint8_t* mat,
                            float* acc, uint16_t* frame, int* err, cudaStream_t st) {
  if (a.N > 0) features_scatter_kernel<<<(a.N + 255) / 256, 256, 0, st>>>(a, x, v, C, mat, acc, err);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const long long n3 = static_cast<long long>(a.n) * a.n * a.n;
  features_finalize_kernel<<<static_cast<unsigned>((n3 + 255) / 256), 256, 0, st>>>(a, acc, frame);
  return cudaGetLastError();
}

cudaError_t launch_features_vjp(const FeatArgs& a, const float* x, const float* v, const float* C,
                                const uint8_t* mat, const float* g_frame, float* dLdx, float* dLdv, float* dLdC,
                                int* err, cudaStream_t st) {
  if (a.N > 0)
    features_vjp_kernel<<<(a.N + 255) / 256, 256, 0, st>>>(a, x, v, C, mat, g_frame, dLdx, dLdv, dLdC, err);
  return cudaGetLastError();
}

}  // namespace sur
