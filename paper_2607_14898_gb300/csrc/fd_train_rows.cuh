// Row-wise and element-wise kernels of the training step (fd_train.cu). All are bound by the
// memory they read and write once: four consecutive columns per thread (16-byte loads and stores),
// and what used to be separate passes over the same arrays rides along: the bf16 copy that the
// next products read, and the column sums of the bias and gain gradients. A block adds up the
// columns of its rows in registers (rows in order), stores one partial row, and sum_parts_kernel
// adds the partial rows in a fixed order: no atomics, so repeatable bits.
// 480p model, 2-chunk clip (24 + 2 blocks; 3328 and 13312 rows), device time of a step: column
// sums, casts and the norms' and GELU's backward 9.9 ms as separate passes, 3.0 ms here.
#pragma once
#include <cuda_runtime.h>

#include "fd_internal.h"

namespace fd {
namespace train {

using bf16 = __nv_bfloat16;
constexpr int kDh = kHeadDim;
constexpr int kRowBlock = 32;   // rows per block of the element-wise passes
constexpr int kNormRows = 16;   // rows per block of the RMSNorm backward

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ uint2 pack4(float a, float b, float c, float d) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&lo),
                    *reinterpret_cast<const uint32_t*>(&hi));
}
__device__ __forceinline__ void add4(float4& s, const float4& v) {
  s.x += v.x;
  s.y += v.y;
  s.z += v.z;
  s.w += v.w;
}

// ---------------------------------------------------------------- column sums
// out[c] = sum over k of part[k][c] (parts rows of `pitch` floats); gate > 0: the columns are a
// gated MLP layer 1's (gate and up units in alternating blocks of 32), out in the blob's order
// (gate, then up).
struct SumJob {
  const float* part;
  int parts, pitch, cols, gate;
  float* out;
};
struct SumJobs {
  SumJob job[3];
};
constexpr int kSumRows = 16;  // threads per column
__global__ void sum_parts_kernel(const __grid_constant__ SumJobs jobs) {
  __shared__ float acc[kSumRows][33];
  const SumJob j = jobs.job[blockIdx.y];
  const int c = blockIdx.x * 32 + threadIdx.x;
  if (blockIdx.x * 32 >= static_cast<unsigned>(j.cols)) return;
  float s = 0.f;
  if (c < j.cols)
#pragma unroll 4
    for (int k = threadIdx.y; k < j.parts; k += kSumRows)
      s += j.part[static_cast<size_t>(k) * j.pitch + c];
  acc[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y != 0 || c >= j.cols) return;
#pragma unroll
  for (int k = 1; k < kSumRows; ++k) s += acc[k][threadIdx.x];
  int o = c;
  if (j.gate > 0) {
    const int u = c / 64 * 32 + c % 32;
    o = c % 64 < 32 ? u : j.gate + u;
  }
  j.out[o] = s;
}

// ---------------------------------------------------------------- GELU, gated SiLU
// GELU, exact (erf) form, and its derivative Phi(z) + z phi(z)
__device__ __forceinline__ float gelu_exact(float v) {
  return 0.5f * v * (1.0f + erff(v * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_grad(float v, float da) {
  const float Phi = 0.5f * (1.0f + erff(v * 0.70710678118654752f));
  const float phi = 0.39894228040143268f * expf(-0.5f * v * v);
  return da * (Phi + v * phi);
}
// n4 groups of four elements
__global__ void gelu_fwd_kernel(const float4* __restrict__ z, long long n4, uint2* __restrict__ a) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < n4;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    const float4 v = z[i];
    a[i] = pack4(gelu_exact(v.x), gelu_exact(v.y), gelu_exact(v.z), gelu_exact(v.w));
  }
}
// dz = da GELU'(z) as bf16 [M][cols] and the partial column sums of the fp32 values
__global__ void gelu_bwd_sum_kernel(const float* __restrict__ z, const float* __restrict__ da,
                                    int M, int cols, bf16* __restrict__ dz16,
                                    float* __restrict__ part) {
  const int c = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (c >= cols) return;
  const int r0 = blockIdx.y * kRowBlock, r1 = min(r0 + kRowBlock, M);
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
  for (int r = r0; r < r1; ++r) {
    const size_t e = static_cast<size_t>(r) * cols + c;
    const float4 v = *reinterpret_cast<const float4*>(z + e);
    const float4 d = *reinterpret_cast<const float4*>(da + e);
    const float4 g = make_float4(gelu_grad(v.x, d.x), gelu_grad(v.y, d.y), gelu_grad(v.z, d.z),
                                 gelu_grad(v.w, d.w));
    *reinterpret_cast<uint2*>(dz16 + e) = pack4(g.x, g.y, g.z, g.w);
    add4(s, g);
  }
  *reinterpret_cast<float4*>(part + static_cast<size_t>(blockIdx.y) * cols + c) = s;
}
// the same values alone, fp32 and bf16 (V = 4: n % 4 == 0 and aligned pointers; else V = 1)
template <int V>
__global__ void gelu_bwd_kernel(const float* __restrict__ z, const float* __restrict__ da,
                                long long n, float* __restrict__ dz, bf16* __restrict__ dz16) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < n / V;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    if constexpr (V == 4) {
      const float4 v = reinterpret_cast<const float4*>(z)[i];
      const float4 d = reinterpret_cast<const float4*>(da)[i];
      const float4 g = make_float4(gelu_grad(v.x, d.x), gelu_grad(v.y, d.y), gelu_grad(v.z, d.z),
                                   gelu_grad(v.w, d.w));
      reinterpret_cast<float4*>(dz)[i] = g;
      reinterpret_cast<uint2*>(dz16)[i] = pack4(g.x, g.y, g.z, g.w);
    } else {
      const float g = gelu_grad(z[i], da[i]);
      dz[i] = g;
      dz16[i] = __float2bfloat16_rn(g);
    }
  }
}

// Gated MLP (the XL layout, reading R7): layer 1's output z [M][2 Dm] holds, on the device,
// the gate and up columns of 32 hidden units side by side in blocks of 64 (gate unit 32 j + i
// at column 64 j + i, its up column at 64 j + 32 + i); a = SiLU(gate) up, in unit order.
__device__ __forceinline__ float logistic(float x) { return 1.0f / (1.0f + expf(-x)); }
__device__ __forceinline__ float swiglu(float g, float up) { return g * logistic(g) * up; }
__global__ void swiglu_fwd_kernel(const float* __restrict__ z, long long M, int Dm,
                                  bf16* __restrict__ a) {
  const int q = Dm / 4;
  const long long n = M * q;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long m = i / q;
    const int u = 4 * static_cast<int>(i - m * q);
    const float* zr = z + m * 2 * Dm + u / 32 * 64 + u % 32;
    const float4 g = *reinterpret_cast<const float4*>(zr);
    const float4 up = *reinterpret_cast<const float4*>(zr + 32);
    *reinterpret_cast<uint2*>(a + m * Dm + u) =
        pack4(swiglu(g.x, up.x), swiglu(g.y, up.y), swiglu(g.z, up.z), swiglu(g.w, up.w));
  }
}
// its backward: d gate = da up SiLU'(gate) with SiLU'(x) = s(x) (1 + x (1 - s(x))), d up =
// da SiLU(gate)
__device__ __forceinline__ void swiglu_grad(float g, float up, float d, float& dg, float& du) {
  const float sg = logistic(g);
  dg = d * up * sg * (1.0f + g * (1.0f - sg));
  du = d * g * sg;
}
// dz in the interleaved layout as bf16 and its partial column sums
__global__ void swiglu_bwd_sum_kernel(const float* __restrict__ z, const float* __restrict__ da,
                                      int M, int Dm, bf16* __restrict__ dz16,
                                      float* __restrict__ part) {
  const int u = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (u >= Dm) return;
  const int c = u / 32 * 64 + u % 32;
  const int r0 = blockIdx.y * kRowBlock, r1 = min(r0 + kRowBlock, M);
  float4 sg = make_float4(0.f, 0.f, 0.f, 0.f), su = sg;
#pragma unroll 2
  for (int r = r0; r < r1; ++r) {
    const size_t e = static_cast<size_t>(r) * 2 * Dm + c;
    const float4 g = *reinterpret_cast<const float4*>(z + e);
    const float4 up = *reinterpret_cast<const float4*>(z + e + 32);
    const float4 d = *reinterpret_cast<const float4*>(da + static_cast<size_t>(r) * Dm + u);
    float4 dg, du;
    swiglu_grad(g.x, up.x, d.x, dg.x, du.x);
    swiglu_grad(g.y, up.y, d.y, dg.y, du.y);
    swiglu_grad(g.z, up.z, d.z, dg.z, du.z);
    swiglu_grad(g.w, up.w, d.w, dg.w, du.w);
    *reinterpret_cast<uint2*>(dz16 + e) = pack4(dg.x, dg.y, dg.z, dg.w);
    *reinterpret_cast<uint2*>(dz16 + e + 32) = pack4(du.x, du.y, du.z, du.w);
    add4(sg, dg);
    add4(su, du);
  }
  float* p = part + static_cast<size_t>(blockIdx.y) * 2 * Dm + c;
  *reinterpret_cast<float4*>(p) = sg;
  *reinterpret_cast<float4*>(p + 32) = su;
}
// rows of a gated layer 1's weight gradient from the device's interleaved order to the blob's
// (gate rows, then up rows): dst row r = src row of blob row r; len % 4 == 0
__global__ void gated_rows_kernel(const float4* __restrict__ src, int rows, int len4,
                                  float4* __restrict__ dst) {
  const long long n = static_cast<long long>(rows) * len4;
  const int gate = rows / 2;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int r = static_cast<int>(i / len4), k = static_cast<int>(i - static_cast<long long>(r) * len4);
    const int u = r < gate ? r : r - gate;
    const int dr = u / 32 * 64 + (r < gate ? 0 : 32) + u % 32;
    dst[i] = src[static_cast<size_t>(dr) * len4 + k];
  }
}

// ---------------------------------------------------------------- RMSNorm backward
// y = x r g, r = (mean(x^2) + eps)^(-1/2), n = D:
// dx = r (dy g) - x r^3 sum_j(dy_j g_j x_j) / n (+ add), fp32 and (dx16 non-null) bf16; partial
// column sums of dy x r (the gain's gradient) into part_g and (non-null) of dx into part_b.
// A block takes kNormRows rows: one warp per row for the row's two sums, then the columns, V per
// thread (V = 4: D % 4 == 0 and aligned pointers), the rows shared by `groups` thread groups when
// D is narrow; group q of block b stores partial row b groups + q.
template <int V>
__global__ void __launch_bounds__(256)
    rmsnorm_bwd_kernel(const float* __restrict__ x, const float* __restrict__ g,
                       const float* __restrict__ dy, const float* __restrict__ add, int M, int D,
                       float eps, int groups, float* __restrict__ dx, bf16* __restrict__ dx16,
                       float* __restrict__ part_g, float* __restrict__ part_b) {
  __shared__ float rs[kNormRows], cs[kNormRows];
  const int lane = threadIdx.x & 31;
  const int row0 = blockIdx.x * kNormRows, rows = min(kNormRows, M - row0);
  for (int i = threadIdx.x >> 5; i < rows; i += 8) {
    const float* xr = x + static_cast<size_t>(row0 + i) * D;
    const float* dr = dy + static_cast<size_t>(row0 + i) * D;
    float ss = 0.f, se = 0.f;
#pragma unroll 8
    for (int j = lane; j < D; j += 32) {
      const float v = xr[j];
      ss = fmaf(v, v, ss);
      se = fmaf(dr[j] * g[j], v, se);
    }
    ss = warp_sum(ss);
    se = warp_sum(se);
    if (lane == 0) {
      const float r = rsqrtf(ss / D + eps);
      rs[i] = r;
      cs[i] = r * r * r * se / D;
    }
  }
  __syncthreads();
  const int per = blockDim.x / groups;  // threads of a group
  const int q = threadIdx.x / per, t = threadIdx.x - q * per;
  if (q >= groups) return;
  for (int c = V * t; c < D; c += V * per) {
    float gg[V], st[V] = {}, sd[V] = {};
#pragma unroll
    for (int k = 0; k < V; ++k) gg[k] = g[c + k];
#pragma unroll 2
    for (int i = q; i < rows; i += groups) {
      const size_t e = static_cast<size_t>(row0 + i) * D + c;
      float xv[V], dv[V], av[V], o[V];
      if constexpr (V == 4) {
        *reinterpret_cast<float4*>(xv) = *reinterpret_cast<const float4*>(x + e);
        *reinterpret_cast<float4*>(dv) = *reinterpret_cast<const float4*>(dy + e);
        if (add != nullptr)
          *reinterpret_cast<float4*>(av) = *reinterpret_cast<const float4*>(add + e);
      } else {
        xv[0] = x[e];
        dv[0] = dy[e];
        if (add != nullptr) av[0] = add[e];
      }
      const float r = rs[i], cc = cs[i];
#pragma unroll
      for (int k = 0; k < V; ++k) {
        float v = r * dv[k] * gg[k] - xv[k] * cc;
        if (add != nullptr) v += av[k];
        o[k] = v;
        st[k] += dv[k] * xv[k] * r;
        sd[k] += v;
      }
      if constexpr (V == 4) {
        *reinterpret_cast<float4*>(dx + e) = make_float4(o[0], o[1], o[2], o[3]);
        if (dx16 != nullptr)
          *reinterpret_cast<uint2*>(dx16 + e) = pack4(o[0], o[1], o[2], o[3]);
      } else {
        dx[e] = o[0];
      }
    }
    const size_t pe = (static_cast<size_t>(blockIdx.x) * groups + q) * D + c;
#pragma unroll
    for (int k = 0; k < V; ++k) {
      part_g[pe + k] = st[k];
      if (part_b != nullptr) part_b[pe + k] = sd[k];
    }
  }
}

// ---------------------------------------------------------------- QKV
// RoPE tables (host-computed in double): temporal (cos, sin) [frames][kBandT], row and column
// [grid][kBandS]
constexpr int kBandS = kHeadDim / 6;               // pairs per spatial band (10)
constexpr int kBandT = kHeadDim / 2 - 2 * kBandS;  // temporal pairs (12)
struct Rope {
  const float2 *t, *y, *x;
};
// angle of pair i for frame f, grid row gy, column gx
__device__ __forceinline__ float2 rope_cs(const Rope& rp, int i, int f, int gy, int gx) {
  if (i < kBandT) return rp.t[f * kBandT + i];
  if (i < kBandT + kBandS) return rp.y[gy * kBandS + i - kBandT];
  return rp.x[gx * kBandS + i - kBandT - kBandS];
}

// Shapes of the QKV kernels: slot < N query heads, then G key groups, then G value groups; rows
// [M / Pc chunks][Pc], Lp rows per frame of which the first L are tokens on a grid of width gw.
// q2 / dq2 are head-major per chunk, [M / Pc][N][Pc][64] (the rows of one chunk's heads of a KV
// group are then contiguous); k2 / dk2 and v1 / dv1 [G][M][64].
struct QkvShape {
  int M, Pc, Lp, L, gw, N, G, qk_norm;
  __device__ size_t head_row(int row, int slot) const {  // row of q2, k2 or v1 (all [..][64])
    return slot < N ? static_cast<size_t>(row / Pc * N + slot) * Pc + row % Pc
                    : static_cast<size_t>((slot - N) % G) * M + row;
  }
  __device__ int key(int row) const {  // position of a token's row among the unpadded keys
    return (row / Pc * (Pc / Lp) + row % Pc / Lp) * L + row % Lp;
  }
};

// RMS over the 64 values of one head with gain g
__device__ __forceinline__ void head_rms(float (&v)[kDh], const float* g, float eps) {
  float ss = 0.f;
#pragma unroll
  for (int j = 0; j < kDh; ++j) ss = fmaf(v[j], v[j], ss);
  const float r = rsqrtf(ss / kDh + eps);
#pragma unroll
  for (int j = 0; j < kDh; ++j) v[j] = v[j] * r * g[j];
}
// One thread does one (row, slot): its 64 values in order, as the sums over a head are. A block
// stages kQkvBatch rows x up to kQkvSlots slots through shared memory (65 floats per unit: no bank
// conflicts where a thread walks its own unit; the stores in and the packed reads out of the forward
// meet 4-way conflicts, the backward's column sums 2-way), so that global memory is read and written in whole lines: a thread reading its own
// 256 bytes took 136 us forward and 89 us backward on average at 480p, staged 42 and 52. What is left
// is a block's chain of load, sums and store, so the loads of a batch are issued together (36 / 34
// us), the four rows of a slot sit in neighbouring threads (a warp then does one kind of slot: 31 /
// 33) and a block takes one batch (kQkvRows rows): 22 / 28, for 1.1 us more in each sum of the
// backward's partial rows; 8 rows a block 32 / 33.
constexpr int kQkvBatch = 4, kQkvSlots = 32, kQkvRows = 4, kQkvPad = 65;
constexpr int kQkvUnits = kQkvBatch * kQkvSlots;  // threads
constexpr int kQkvLoads = kQkvSlots * kDh / (4 * kQkvUnits);  // 16-byte loads a thread and row
__device__ __forceinline__ void put4(float* p, float4 v) {
  p[0] = v.x; p[1] = v.y; p[2] = v.z; p[3] = v.w;
}

// QKV forward: q2 = RoPE(q0) (RMS with g2 first when qk_norm), k2 = RoPE(RMS(k0; gk)),
// v1 = RMS(v0; g2) (v0 when qk_norm), in bf16. With qr non-null, also: q rows bf16 [M][N 64] (the
// attention kernel's layout), and the real tokens' K bf16 [G][pitch][64] and V^T fp16
// [G][64][pitch] without the padding rows (chunk c's Lu = Pc / Lp * L keys at c Lu ...), the keys
// of the fused band attention. V^T leaves as the block's kQkvRows
// keys of each dimension.
__global__ void __launch_bounds__(kQkvUnits)
    qkv_fwd_kernel(const float* __restrict__ qkv, QkvShape p, const float* __restrict__ gk,
                   const float* __restrict__ g2, float eps, Rope rp, bf16* __restrict__ q2,
                   bf16* __restrict__ k2, bf16* __restrict__ v1, bf16* __restrict__ qr,
                   bf16* __restrict__ ku, __half* __restrict__ vtu, int pitch) {
  extern __shared__ float sm[];
  float* const xs = sm;
  __half* const vts = reinterpret_cast<__half*>(sm + kQkvUnits * kQkvPad);
  const int slots = p.N + 2 * p.G, s0 = blockIdx.y * kQkvSlots;
  const int sc = min(kQkvSlots, slots - s0), units = kQkvBatch * sc;
  const int v0 = max(p.N + p.G, s0);  // first V slot of the block
  const int tid = threadIdx.x, lu = tid / 16, lj = tid % 16 * 4;
#pragma unroll 1
  for (int b = 0; b < kQkvRows / kQkvBatch; ++b) {
    const int row0 = blockIdx.x * kQkvRows + b * kQkvBatch;
    float4 x[kQkvBatch][kQkvLoads];
#pragma unroll
    for (int i = 0; i < kQkvBatch; ++i)
#pragma unroll
      for (int k = 0; k < kQkvLoads; ++k)
        if (lu + 8 * k < sc)
          x[i][k] = *reinterpret_cast<const float4*>(
              qkv + (static_cast<size_t>(row0 + i) * slots + s0 + lu + 8 * k) * kDh + lj);
#pragma unroll
    for (int i = 0; i < kQkvBatch; ++i)
#pragma unroll
      for (int k = 0; k < kQkvLoads; ++k)
        if (lu + 8 * k < sc) put4(xs + ((lu + 8 * k) * kQkvBatch + i) * kQkvPad + lj, x[i][k]);
    __syncthreads();
    if (tid < units) {
      const int row = row0 + tid % kQkvBatch, slot = s0 + tid / kQkvBatch;
      const int f = row / p.Lp, l = min(row % p.Lp, p.L - 1);  // padding rows: a real token's angles
      const int gy = l / p.gw, gx = l % p.gw;
      const bool is_q = slot < p.N, is_k = !is_q && slot < p.N + p.G;
      float v[kDh];
      float* px = xs + tid * kQkvPad;
#pragma unroll
      for (int j = 0; j < kDh; ++j) v[j] = px[j];
      if (is_k) head_rms(v, gk, eps);
      else if (is_q ? p.qk_norm != 0 : p.qk_norm == 0) head_rms(v, g2, eps);
      if (is_q || is_k) {
#pragma unroll
        for (int i = 0; i < kDh / 2; ++i) {
          const float2 cs = rope_cs(rp, i, f, gy, gx);
          const float a = v[2 * i], c = v[2 * i + 1];
          v[2 * i] = a * cs.x - c * cs.y;
          v[2 * i + 1] = a * cs.y + c * cs.x;
        }
      }
#pragma unroll
      for (int j = 0; j < kDh; ++j) px[j] = v[j];
    }
    __syncthreads();
    // eight values (16 bytes) each
#pragma unroll
    for (int i = 0; i < kQkvBatch * kQkvLoads / 2; ++i) {
      const int ri = i % kQkvBatch, su = tid / 8 + 16 * (i / kQkvBatch);
      if (su >= sc) break;
      const int j = tid % 8 * 8, row = row0 + ri, slot = s0 + su;
      const float* px = xs + (su * kQkvBatch + ri) * kQkvPad + j;
      const uint2 lo = pack4(px[0], px[1], px[2], px[3]), hi = pack4(px[4], px[5], px[6], px[7]);
      const uint4 w = make_uint4(lo.x, lo.y, hi.x, hi.y);
      const bool is_q = slot < p.N, is_k = !is_q && slot < p.N + p.G;
      bf16* dst = is_q ? q2 : (is_k ? k2 : v1);
      *reinterpret_cast<uint4*>(dst + p.head_row(row, slot) * kDh + j) = w;
      if (qr == nullptr) continue;
      if (is_q) {
        *reinterpret_cast<uint4*>(qr + (static_cast<size_t>(row) * p.N + slot) * kDh + j) = w;
      } else if (!is_k) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
          vts[((slot - v0) * kDh + j + k) * kQkvRows + row % kQkvRows] = __float2half_rn(px[k]);
      } else if (row % p.Lp < p.L) {  // padding rows are no keys
        *reinterpret_cast<uint4*>(
            ku + (static_cast<size_t>(slot - p.N) * pitch + p.key(row)) * kDh + j) = w;
      }
    }
    __syncthreads();
  }
  if (qr == nullptr) return;
  const int r0 = blockIdx.x * kQkvRows, nv = s0 + sc - v0;  // V slots of the block
  const int r = r0 + tid % kQkvRows;
  if (nv <= 0 || r % p.Lp >= p.L) return;
  __half* const dst = vtu + static_cast<size_t>(v0 - p.N - p.G) * kDh * pitch + p.key(r);
#pragma unroll 8
  for (int d = tid / kQkvRows; d < nv * kDh; d += kQkvUnits / kQkvRows)  // of group d / 64
    dst[static_cast<size_t>(d) * pitch] = vts[d * kQkvRows + tid % kQkvRows];
}

// RMS over one head, backward: x the pre-norm values in shared memory, overwritten by the gain's
// gradient terms dy x r; dy the gradient of the normed output, overwritten by dx
__device__ __forceinline__ void head_rms_bwd(float* x, float (&dy)[kDh], const float* g,
                                             float eps) {
  float ss = 0.f, se = 0.f;
#pragma unroll
  for (int j = 0; j < kDh; ++j) {
    ss = fmaf(x[j], x[j], ss);
    se = fmaf(dy[j] * g[j], x[j], se);
  }
  const float r = rsqrtf(ss / kDh + eps);
  const float c = r * r * r * se / kDh;
#pragma unroll
  for (int j = 0; j < kDh; ++j) {
    const float xv = x[j], t = dy[j] * xv * r;
    dy[j] = r * dy[j] * g[j] - xv * c;
    x[j] = t;
  }
}

// dq2, dk2, dv1 (fp32) -> dqkv bf16 [M][(N + 2G) 64]: inverse RoPE (the rotation by the negated
// angle), then the per-head RMS backward where the forward normalised. Partial sums: the columns
// of dqkv (the bias gradient) into part_b [blocks x][(N + 2G) 64]; the gains' terms into
// part_t [blocks x * blocks y][128], K's gain then V's (Q's with qk_norm).
__global__ void __launch_bounds__(kQkvUnits)
    qkv_bwd_kernel(const float* __restrict__ qkv, const float* __restrict__ dq2,
                   const float* __restrict__ dk2, const float* __restrict__ dv1, QkvShape p,
                   const float* __restrict__ gk, const float* __restrict__ g2, float eps, Rope rp,
                   bf16* __restrict__ dqkv16, float* __restrict__ part_b,
                   float* __restrict__ part_t) {
  extern __shared__ float sm[];
  float* const xs = sm;
  float* const ds = sm + kQkvUnits * kQkvPad;
  const int slots = p.N + 2 * p.G, s0 = blockIdx.y * kQkvSlots;
  const int sc = min(kQkvSlots, slots - s0), units = kQkvBatch * sc, cols = sc * kDh;
  const int tid = threadIdx.x, lu = tid / 16, lj = tid % 16 * 4;
  auto normed = [&](int slot) {
    const bool is_q = slot < p.N, is_k = !is_q && slot < p.N + p.G;
    return is_k || (is_q ? p.qk_norm != 0 : p.qk_norm == 0);
  };
  // column pairs 2 tid, 2 tid + 1 (+ 256 k) of the block's slots
  float sb[16] = {}, st[16] = {};
#pragma unroll 1
  for (int b = 0; b < kQkvRows / kQkvBatch; ++b) {
    const int row0 = blockIdx.x * kQkvRows + b * kQkvBatch;
#pragma unroll
    for (int h = 0; h < kQkvBatch; h += 2) {
      float4 x[2][kQkvLoads], d[2][kQkvLoads];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int k = 0; k < kQkvLoads; ++k) {
          const int row = row0 + h + i, slot = s0 + lu + 8 * k;
          if (lu + 8 * k >= sc) continue;
          const float* src = slot < p.N ? dq2 : (slot < p.N + p.G ? dk2 : dv1);
          x[i][k] = *reinterpret_cast<const float4*>(
              qkv + (static_cast<size_t>(row) * slots + slot) * kDh + lj);
          d[i][k] = *reinterpret_cast<const float4*>(src + p.head_row(row, slot) * kDh + lj);
        }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int k = 0; k < kQkvLoads; ++k) {
          if (lu + 8 * k >= sc) continue;
          const int e = ((lu + 8 * k) * kQkvBatch + h + i) * kQkvPad + lj;
          put4(xs + e, x[i][k]);
          put4(ds + e, d[i][k]);
        }
    }
    __syncthreads();
    if (tid < units) {
      const int row = row0 + tid % kQkvBatch, slot = s0 + tid / kQkvBatch;
      const int f = row / p.Lp, l = min(row % p.Lp, p.L - 1);  // padding rows: a real token's angles
      const int gy = l / p.gw, gx = l % p.gw;
      const bool is_q = slot < p.N, is_k = !is_q && slot < p.N + p.G;
      float d[kDh];
      float* pd = ds + tid * kQkvPad;
#pragma unroll
      for (int j = 0; j < kDh; ++j) d[j] = pd[j];
      if (is_q || is_k) {
#pragma unroll
        for (int i = 0; i < kDh / 2; ++i) {
          const float2 cs = rope_cs(rp, i, f, gy, gx);
          const float a = d[2 * i], c = d[2 * i + 1];
          d[2 * i] = a * cs.x + c * cs.y;
          d[2 * i + 1] = -a * cs.y + c * cs.x;
        }
      }
      if (normed(slot)) head_rms_bwd(xs + tid * kQkvPad, d, is_k ? gk : g2, eps);
#pragma unroll
      for (int j = 0; j < kDh; ++j) pd[j] = d[j];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int c = 2 * (tid + kQkvUnits * k);
      if (c >= cols) break;
      const int su = c / kDh, j = c % kDh;
      const bool t = normed(s0 + su);
#pragma unroll
      for (int i = 0; i < kQkvBatch; ++i) {
        const int e = (su * kQkvBatch + i) * kQkvPad + j;
        const float a = ds[e], d = ds[e + 1];
        const __nv_bfloat162 v = __floats2bfloat162_rn(a, d);
        *reinterpret_cast<__nv_bfloat162*>(
            dqkv16 + static_cast<size_t>(row0 + i) * slots * kDh + s0 * kDh + c) = v;
        sb[2 * k] += a;
        sb[2 * k + 1] += d;
        if (t) {
          st[2 * k] += xs[e];
          st[2 * k + 1] += xs[e + 1];
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int c = 2 * (tid + kQkvUnits * k);
    if (c >= cols) break;
    *reinterpret_cast<float2*>(part_b + static_cast<size_t>(blockIdx.x) * slots * kDh + s0 * kDh +
                               c) = make_float2(sb[2 * k], sb[2 * k + 1]);
    xs[c] = st[2 * k];
    xs[c + 1] = st[2 * k + 1];
  }
  __syncthreads();
  // the gains' terms over the block's slots of each kind (kQkvUnits = 2 x 64 threads)
  const int j = tid % kDh;
  float t = 0.f;
  for (int su = 0; su < sc; ++su) {
    const int slot = s0 + su;
    const bool is_k = slot >= p.N && slot < p.N + p.G;
    if (normed(slot) && is_k == (tid < kDh)) t += xs[su * kDh + j];
  }
  part_t[(static_cast<size_t>(blockIdx.y) * gridDim.x + blockIdx.x) * 2 * kDh + tid] = t;
}
static_assert(kQkvUnits == 2 * kDh && kQkvRows % kQkvBatch == 0 &&
                  kQkvSlots * kDh <= 16 * kQkvUnits, "column phase");
static_assert(kQkvUnits % kQkvRows == 0 && kQkvUnits == kQkvBatch * kQkvSlots, "V^T store");

// ---------------------------------------------------------------- L1 term, pixel shuffle
// L1 term of the pixels (reading T3: the mean of |x_hat - x| over the clip, unclamped output,
// reading T1) through the pixel shuffle: F [R][C rs^2] with refined row (c r_t + tau) Lp + l,
// target [T][C][r_t][H][W]; dF = sign(F - x) / total (0 on padding rows, and on chunk 0's
// frames tau >= first, which a one-frame first chunk does not emit); per-block sums of |F - x|
// into part[block] (a fixed-order tree)
struct PixelGrid {
  int T, rt, first, Lp, L, gh, gw, C, rs;
  float inv_total;
};
__device__ __forceinline__ float l1_grad(float diff, float inv_total) {
  return diff > 0.f ? inv_total : (diff < 0.f ? -inv_total : 0.f);
}
__device__ __forceinline__ void block_sum_256(float e, float* out) {
  __shared__ float red[256];
  red[threadIdx.x] = e;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}
// one element per thread, any rs and alignment
__global__ void l1_head_kernel(const float* __restrict__ F, const float* __restrict__ target,
                               PixelGrid p, float* __restrict__ dF, float* __restrict__ part) {
  const int cols = p.C * p.rs * p.rs;
  const long long total = static_cast<long long>(p.T) * p.rt * p.Lp * cols;
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  float e = 0.f;
  if (i < total) {
    const long long row = i / cols;
    const int col = static_cast<int>(i % cols);
    const int l = static_cast<int>(row % p.Lp);
    const long long ft = row / p.Lp;  // c r_t + tau
    float g = 0.f;
    const int c = static_cast<int>(ft / p.rt), tau = static_cast<int>(ft % p.rt);
    if (l < p.L && (c > 0 || tau < p.first)) {
      const int ch = col / (p.rs * p.rs), ij = col % (p.rs * p.rs);
      const int ii = ij / p.rs, jj = ij % p.rs;
      const int h = l / p.gw, w = l % p.gw;
      const int H = p.gh * p.rs, W = p.gw * p.rs;
      const float x = target[((static_cast<size_t>(c) * p.C + ch) * p.rt + tau) * H * W +
                             static_cast<size_t>(h * p.rs + ii) * W + w * p.rs + jj];
      const float diff = F[i] - x;
      e = fabsf(diff);
      g = l1_grad(diff, p.inv_total);
    }
    dF[i] = g;
  }
  block_sum_256(e, part + blockIdx.x);
}
// four pixels of one row of a token's block per thread (rs % 4 == 0, 16-byte aligned F, target and
// dF), kRowBlock rows per block: the integer divisions are one per row and one per thread, not
// four per element. dF in fp32 (dF32) or, for the training step, bf16 with its column sums.
__global__ void __launch_bounds__(256)
    l1_head4_kernel(const float* __restrict__ F, const float* __restrict__ target, PixelGrid p,
                    float* __restrict__ dF32, bf16* __restrict__ dF16,
                    float* __restrict__ part_cols, float* __restrict__ part) {
  __shared__ long long base[kRowBlock];  // target offset of the row's token, -1: not emitted
  const int cols = p.C * p.rs * p.rs;
  const int M = p.T * p.rt * p.Lp;
  const int r0 = blockIdx.y * kRowBlock, rows = min(kRowBlock, M - r0);
  const long long HW = static_cast<long long>(p.gh) * p.rs * p.gw * p.rs;
  const int W = p.gw * p.rs;
  if (threadIdx.x < rows) {
    const int row = r0 + threadIdx.x, l = row % p.Lp, ft = row / p.Lp;
    const int c = ft / p.rt, tau = ft % p.rt;
    base[threadIdx.x] = l < p.L && (c > 0 || tau < p.first)
                            ? (static_cast<long long>(c) * p.C * p.rt + tau) * HW +
                                  static_cast<long long>(l / p.gw * p.rs) * W + l % p.gw * p.rs
                            : -1;
  }
  __syncthreads();
  const int col = 4 * (blockIdx.x * 256 + threadIdx.x);
  float e = 0.f;
  if (col < cols) {
    const int ch = col / (p.rs * p.rs), ij = col % (p.rs * p.rs);
    const long long off = ch * p.rt * HW + static_cast<long long>(ij / p.rs) * W + ij % p.rs;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int i = 0; i < rows; ++i) {
      const size_t f = static_cast<size_t>(r0 + i) * cols + col;
      float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
      if (base[i] >= 0) {
        const float4 a = *reinterpret_cast<const float4*>(F + f);
        const float4 x = *reinterpret_cast<const float4*>(target + base[i] + off);
        const float4 d = make_float4(a.x - x.x, a.y - x.y, a.z - x.z, a.w - x.w);
        e += (fabsf(d.x) + fabsf(d.y)) + (fabsf(d.z) + fabsf(d.w));
        g = make_float4(l1_grad(d.x, p.inv_total), l1_grad(d.y, p.inv_total),
                        l1_grad(d.z, p.inv_total), l1_grad(d.w, p.inv_total));
      }
      if (dF16 != nullptr) {
        *reinterpret_cast<uint2*>(dF16 + f) = pack4(g.x, g.y, g.z, g.w);
        add4(s, g);
      } else {
        *reinterpret_cast<float4*>(dF32 + f) = g;
      }
    }
    if (dF16 != nullptr)
      *reinterpret_cast<float4*>(part_cols + static_cast<size_t>(blockIdx.y) * cols + col) = s;
  }
  block_sum_256(e, part + static_cast<size_t>(blockIdx.y) * gridDim.x + blockIdx.x);
}

// one block of kLossThreads: thread t sums parts t, t + kLossThreads, ... in fp64, then a
// fixed-order tree over the threads (the same bits every step)
constexpr int kLossThreads = 1024;
__global__ void finish_loss_kernel(const float* __restrict__ part, int n, float inv_total,
                                   float* __restrict__ loss) {
  __shared__ double acc[kLossThreads];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += kLossThreads) s += part[i];
  acc[threadIdx.x] = s;
  __syncthreads();
  for (int w = kLossThreads / 2; w > 0; w >>= 1) {
    if (static_cast<int>(threadIdx.x) < w) acc[threadIdx.x] += acc[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = static_cast<float>(acc[0] * inv_total);
}

// ---------------------------------------------------------------- temporal upsampling, backward
// refined row (c r_t + tau) Lp + l of dh [T r_t Lp][D] back to channel block tau of token row
// c Lp + l (Eq. temporal_upsample, reading R6): bf16 [T Lp][r_t D] and its partial column sums
__global__ void tup_bwd_kernel(const float* __restrict__ dh, int M, int rt, int Lp, int D,
                               bf16* __restrict__ de16, float* __restrict__ part) {
  const int cols = rt * D;
  const int c = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (c >= cols) return;
  const int tau = c / D, d = c - tau * D;
  const int r0 = blockIdx.y * kRowBlock, r1 = min(r0 + kRowBlock, M);
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
  for (int r = r0; r < r1; ++r) {
    const int chunk = r / Lp, l = r - chunk * Lp;
    const float4 v = *reinterpret_cast<const float4*>(
        dh + (static_cast<size_t>(chunk * rt + tau) * Lp + l) * D + d);
    *reinterpret_cast<uint2*>(de16 + static_cast<size_t>(r) * cols + c) =
        pack4(v.x, v.y, v.z, v.w);
    add4(s, v);
  }
  *reinterpret_cast<float4*>(part + static_cast<size_t>(blockIdx.y) * cols + c) = s;
}

}  // namespace train
}  // namespace fd
