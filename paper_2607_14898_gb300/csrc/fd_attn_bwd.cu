// Backward of the band attention (the training step, Sec. 3.3) on tcgen05: dQ, and dK with dV, in
// two launches that keep the scores on chip. Both recompute S = Q K^T and dP = dO V^T per 128 x
// 128 block and form P = exp(S / 8 - lse), dS = P (dP - delta) / 8 in registers.
//
//   dQ launch   one CTA per 128 query rows of a head: dQ += dS K over the key blocks of the
//               chunk's window
//   dK/dV launch one CTA per 128 keys of a KV group, on the transposed blocks S^T = K Q^T and
//               dP^T = V dO^T: dK += dS^T Q, dV += P^T dO over the query blocks (chunks whose
//               window holds the keys, then the group's heads, then rows)
//
// What bounds it: the issue of the arithmetic on the scores. At 480p refinement sizes (2 chunks of
// 6656 rows, 16 heads on 4 groups) a 128 x 128 block takes 2630 cycles of an SM in either launch: per
// scheduler 1940 (dK / dV, 15 instructions a score) and 1630 (dQ, 13) issue cycles, against 1024 and
// 768 of MMA; the FMA pipe is at 50 and 45 %, the transcendental one at 20 %. So S and dP are
// recomputed in both launches (2 of the 5 products twice) rather than stored: writing dS, dS^T and
// P^T (bf16) and reading them back in N = 64 products moved 12 bytes a score: 45.3 ms of what was
// then a 72.6 ms training step of the 480p model (2 chunks, 24 + 2 blocks) and 43.8 ms with these
// kernels, with the same bits as gradients. They are 9.0 ms of it (24 x 179 us, 2 x 2344 us).
// Every product's operands are the row-major tiles as they are: K-major for S and dP, and the same
// shared-memory tile read MN-major (the transpose bit of the instruction descriptor) as B of the
// gradient products, so nothing is transposed in memory.
//
// The sums' order is fixed: one TMEM accumulator chain per dQ tile over ascending keys; for dK /
// dV one chain per (query chunk, hs heads), the chains added in fp32 in that order. No atomics.
//
// Warps: 0 TMA (the CTA's own two tiles once, then the streamed pairs into a ring), 1 MMA issue,
// 2-17 element-wise: four warps per 32 TMEM lanes, 32 columns each; a warp takes S and dP into
// registers and releases them at once, so that the next block's S and dP run under its arithmetic.
#include "fd_internal.h"
#include "fd_ptx.cuh"

namespace fd {

namespace attn_bwd {
constexpr int kStages = 4;
constexpr int kTile = 128 * 128;  // bytes of a [128][64] bf16 tile
constexpr int kOffX = 0;          // the CTA's own tiles: Q, dO (dQ) or K, V (dK / dV)
constexpr int kOffY = 2 * kTile;  // ring of streamed pairs: K, V or Q, dO
constexpr int kOffL = kOffY + kStages * 2 * kTile;  // ring of lse[128], delta[128] (dK / dV)
constexpr int kOffBar = kOffL + kStages * 1024;
constexpr int kSmem = kOffBar + 256;
constexpr int kElemWarps = 16;
constexpr int kThreads = 64 + 32 * kElemWarps;
constexpr uint32_t kColS = 0, kColDp = 128, kColDs = 256, kColP = 320, kColAcc = 384;
enum Bar { kXFull, kFull, kEmpty = kFull + kStages, kSReady = kEmpty + kStages, kSFree, kPFull,
           kPFree, kAccDone, kAccFree, kDone, kNumBars };
static_assert(kNumBars * 8 + 8 <= 256 && kSmem <= 227 * 1024, "shared memory");
}  // namespace attn_bwd

// P and dS of two elements: the softmax and its derivative, given each one's row log-sum-exp
// (negated; -inf for a padding row: P = 0) and delta (negated). Packed fp32 pairs, each operation
// rounded as its scalar form.
__device__ __forceinline__ void score_grad2(uint32_t s0, uint32_t s1, uint32_t d0, uint32_t d1,
                                            uint64_t nlse, uint64_t ndelta, float (&pr)[2],
                                            float (&ds)[2]) {
  const uint64_t scale = pack_f32x2(0.125f, 0.125f);
  uint64_t x = pack_f32x2(__uint_as_float(s0), __uint_as_float(s1));
  uint64_t y = pack_f32x2(__uint_as_float(d0), __uint_as_float(d1));
  asm("fma.rn.f32x2 %0, %0, %1, %2;" : "+l"(x) : "l"(scale), "l"(nlse));
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x));
  pr[0] = expf(a);
  pr[1] = expf(b);
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(y) : "l"(ndelta));
  asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(y) : "l"(pack_f32x2(pr[0], pr[1])));
  asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(y) : "l"(scale));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(ds[0]), "=f"(ds[1]) : "l"(y));
}

// The unit of a CTA. dQ: query rows q0 .. of head h, chunk i; keys k0 .. of the window. dK / dV:
// keys of chunk jc in group g; query chunks jc .. jc + nq - 1.
template <bool KV>
__global__ void __launch_bounds__(attn_bwd::kThreads, 1)
    attn_bwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmdO,
                    const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                    const __grid_constant__ AttnBwdParams p) {
  using namespace attn_bwd;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int warp = warp_index();
  const int lane = threadIdx.x & 31;
  const uint32_t base = smem_u32(smem);
  const bool aligned = (base & 1023u) == 0;
  const uint32_t bar0 = base + kOffBar;
  auto bar = [&](int i) { return bar0 + 8u * static_cast<uint32_t>(i); };
  uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffBar + 8 * kNumBars);

  const int hpg = p.N / p.G;
  const int tiles = p.Pc / 128;  // 128-row tiles of a chunk (of one head)
  int xrow, g, i0, len, group;   // first row of the own tiles; group; first query chunk; blocks
  int yrow = 0;                  // dQ: first key row
  int key = 0;                   // dK / dV: first key's position in its chunk
  if constexpr (KV) {
    // longest first: keys of early chunks are in the window of more query chunks
    const int u = blockIdx.x / p.G;
    g = blockIdx.x % p.G;
    i0 = u / tiles;
    key = u % tiles * 128;
    xrow = g * p.M + u * 128;
    const int nq = p.T - i0 < p.W ? p.T - i0 : p.W;
    group = p.hs * tiles;
    len = nq * hpg * tiles;
  } else {
    const int per = p.N * tiles;
    const int u = blockIdx.x % per;
    i0 = p.T - 1 - blockIdx.x / per;  // longest first: late chunks have the full window
    const int h = u / tiles;
    g = h / hpg;
    xrow = (i0 * p.N + h) * p.Pc + u % tiles * 128;
    const int j0 = i0 - p.W + 1 > 0 ? i0 - p.W + 1 : 0;
    yrow = g * p.M + j0 * p.Pc;
    len = (i0 + 1 - j0) * tiles;
    group = len;
  }
  // first query row of block j (dK / dV): chunk-major, then the group's heads, then rows; one
  // head's blocks are contiguous, and so are a group's heads within a chunk
  auto y_row = [&](int j) -> int {
    if constexpr (KV) {
      const int c = j / (hpg * tiles);
      return ((i0 + c) * p.N + g * hpg) * p.Pc + (j - c * hpg * tiles) * 128;
    } else {
      return yrow + j * 128;
    }
  };

  if (threadIdx.x == 0) {
    if (!aligned) atomicOr(p.err, ERR_SMEM_ALIGN);
    for (int b = 0; b < kNumBars; ++b)
      mbar_init(bar(b), b == kSFree || b == kPFull || b == kAccFree ? kElemWarps : 1);
    fence_barrier_init();
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  // the dQ grid reads nothing that the dK / dV grid writes: its CTAs may take the SMs that this
  // grid leaves (both grids' sizes leave some idle)
  if (KV) grid_dep_launch();

  if (!aligned) {
    // error recorded above
  } else if (warp == 0) {
    // ------------------------------------------------------------ TMA loads
    if (elect_one()) {
      mbar_expect_tx(bar(kXFull), 2 * kTile);
      tma_load_2d(base + kOffX, KV ? &tmK : &tmQ, bar(kXFull), 0, xrow);
      tma_load_2d(base + kOffX + kTile, KV ? &tmV : &tmdO, bar(kXFull), 0, xrow);
    }
    int st = 0, j = 0;
    uint32_t ph = 1;
    for (; j < len; ++j) {
      const int row = y_row(j);
      if (!mbar_wait_warp(bar(kEmpty + st), ph, p.err, ERR_WAIT_MMA)) break;
      if (elect_one()) {
        const uint32_t b = bar(kFull + st), dst = base + kOffY + st * 2 * kTile;
        mbar_expect_tx(b, 2 * kTile + (KV ? 1024 : 0));
        tma_load_2d(dst, KV ? &tmQ : &tmK, b, 0, row);
        tma_load_2d(dst + kTile, KV ? &tmdO : &tmV, b, 0, row);
        if (KV) {
          bulk_load(base + kOffL + st * 1024, p.lse + row, 512, b);
          bulk_load(base + kOffL + st * 1024 + 512, p.delta + row, 512, b);
        }
      }
      if (++st == kStages) {
        st = 0;
        ph ^= 1;
      }
    }
    // nothing may be in flight when the CTA exits
    mbar_wait_warp(bar(kXFull), 0, p.err, ERR_WAIT_TMA);
    for (int k = j - 1; k >= 0 && k >= j - kStages; --k)
      mbar_wait_warp(bar(kFull + k % kStages), (k / kStages) & 1, p.err, ERR_WAIT_TMA);
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issue
    // S and dP of block j, then the gradient products of block j - 1
    const uint32_t id_s = idesc_bf16_f32(128, 128);
    const uint32_t id_g = idesc_bf16_f32(128, 64) | (1u << 16);  // B read MN-major
    const uint64_t dx = sdesc_k_sw128(base + kOffX), dy = sdesc_k_sw128(base + kOffY);
    constexpr uint64_t kT = kTile >> 4;
    bool ok = mbar_wait_warp(bar(kXFull), 0, p.err, ERR_WAIT_TMA);
    int st = 0, gst = 0, in_group = 0;
    uint32_t ph = 0, gph = 0;  // parity of the full barrier; of accFree
    for (int j = 0; j <= len && ok; ++j) {
      if (j < len) {
        ok = mbar_wait_warp(bar(kFull + st), ph, p.err, ERR_WAIT_TMA) &&
             (j == 0 || mbar_wait_warp(bar(kSFree), (j - 1) & 1, p.err, ERR_WAIT_EPI));
        if (!ok) break;
        tc_fence_after();
        const uint64_t y = dy + static_cast<uint64_t>(st) * 2 * kT;
        if (elect_one()) {
          mma4_bf16_ss(tmem + kColS, dx, y, id_s, 0u);
          mma4_bf16_ss(tmem + kColDp, dx + kT, y + kT, id_s, 0u);
          mma_commit(bar(kSReady));
        }
        if (++st == kStages) {
          st = 0;
          ph ^= 1;
        }
      }
      if (j > 0) {
        const bool first = in_group == 0, last = in_group + 1 == group;
        ok = mbar_wait_warp(bar(kPFull), (j - 1) & 1, p.err, ERR_WAIT_EPI);
        if (ok && first && j > 1) {  // the previous chain's sums have been read
          ok = mbar_wait_warp(bar(kAccFree), gph, p.err, ERR_WAIT_EPI);
          gph ^= 1;
        }
        if (!ok) break;
        tc_fence_after();
        const uint64_t y = dy + static_cast<uint64_t>(gst) * 2 * kT;
        if (elect_one()) {
          mma4_bf16_ts_mn(tmem + kColAcc, tmem + kColDs, y, id_g, first ? 0u : 1u);
          mma4_bf16_ts_mn(tmem + kColAcc, tmem + kColDs + 32, y + kT / 2, id_g, 1u);
          if (KV) {
            mma4_bf16_ts_mn(tmem + kColAcc + 64, tmem + kColP, y + kT, id_g, first ? 0u : 1u);
            mma4_bf16_ts_mn(tmem + kColAcc + 64, tmem + kColP + 32, y + kT + kT / 2, id_g, 1u);
          }
          mma_commit(bar(kPFree));
          mma_commit(bar(kEmpty + gst));
          if (last) mma_commit(bar(kAccDone));
        }
        in_group = last ? 0 : in_group + 1;
        if (++gst == kStages) gst = 0;
      }
    }
    if (elect_one()) mma_commit(bar(kDone));
    mbar_wait_warp(bar(kDone), 0, p.err, ERR_WAIT_MMA);
  } else {
    // ------------------------------------------------------------ element-wise
    const int quarter = warp & 3, hc = (warp - 2) >> 2;
    const int row = quarter * 32 + lane;  // TMEM lane: query row (dQ) or key (dK / dV)
    const uint32_t lanes = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
    uint64_t nlse = 0, ndelta = 0;
    bool key_live = true;
    if constexpr (KV) {
      key_live = (key + row) % p.Lp < p.L;
    } else {
      const float a = -__ldg(p.lse + xrow + row), b = -__ldg(p.delta + xrow + row);
      nlse = pack_f32x2(a, a);
      ndelta = pack_f32x2(b, b);
    }
    const bool all_live = __all_sync(0xffffffffu, key_live);
    int st = 0, in_group = 0, groups = 0;
    uint32_t ph = 0;
    int kpos = 0;  // dQ: the block's first key within its frame (Lp rows, the first L of them keys)
    for (int j = 0; j < len; ++j) {
      if (KV && !mbar_wait_warp(bar(kFull + st), ph, p.err, ERR_WAIT_TMA)) break;
      if (!mbar_wait_warp(bar(kSReady), j & 1, p.err, ERR_WAIT_MMA)) break;
      tc_fence_after();
      uint32_t s[32], d[32];
      tmem_ld_32x32b_x32(lanes + kColS + 32u * hc, s);
      tmem_ld_32x32b_x32(lanes + kColDp + 32u * hc, d);
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (elect_one()) mbar_arrive(bar(kSFree));
      uint32_t pd[16], pp[KV ? 16 : 1];
#pragma unroll
      for (int e = 0; e < 32; e += 4) {
        uint64_t nl[2] = {nlse, nlse}, nd[2] = {ndelta, ndelta};
        if constexpr (KV) {  // the block's lse and delta by column, the same for every lane
          const float4* q =
              reinterpret_cast<const float4*>(smem + kOffL + st * 1024) + 8 * hc + e / 4;
          const float4 l4 = q[0], d4 = q[32];
          nl[0] = pack_f32x2(-l4.x, -l4.y);
          nl[1] = pack_f32x2(-l4.z, -l4.w);
          nd[0] = pack_f32x2(-d4.x, -d4.y);
          nd[1] = pack_f32x2(-d4.z, -d4.w);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          float pr[2], ds[2];
          score_grad2(s[e + 2 * k], s[e + 2 * k + 1], d[e + 2 * k], d[e + 2 * k + 1], nl[k], nd[k],
                      pr, ds);
          pd[e / 2 + k] = pack_bf16x2(ds[0], ds[1]);
          if constexpr (KV) pp[e / 2 + k] = pack_bf16x2(pr[0], pr[1]);
        }
      }
      // padding keys take no part: their rows (dK / dV) or columns (dQ) are zero
      if constexpr (KV) {
        if (!all_live) {
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            pd[k] = key_live ? pd[k] : 0u;
            pp[k] = key_live ? pp[k] : 0u;
          }
        }
      } else {
        const int live = p.L - kpos - 32 * hc;  // keys among this warp's columns
        if (live < 32) {
#pragma unroll
          for (int k = 0; k < 16; ++k)
            pd[k] = 2 * k + 1 < live ? pd[k] : (2 * k < live ? pd[k] & 0xffffu : 0u);
        }
        kpos = kpos + 128 == p.Lp ? 0 : kpos + 128;
      }
      if (j > 0 && !mbar_wait_warp(bar(kPFree), (j - 1) & 1, p.err, ERR_WAIT_MMA)) break;
      tc_fence_after();
      __syncwarp();  // block 0 waits for nothing after the elected arrive above
      tmem_st_32x32b_x16(lanes + kColDs + 16u * hc, pd);
      if constexpr (KV) tmem_st_32x32b_x16(lanes + kColP + 16u * hc, pp);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (elect_one()) mbar_arrive(bar(kPFull));
      if (++st == kStages) {
        st = 0;
        ph ^= 1;
      }
      if (++in_group < group) continue;

      // the chain's sums: 16 columns per thread, the first chain stored, later ones added
      in_group = 0;
      if (!mbar_wait_warp(bar(kAccDone), groups & 1, p.err, ERR_WAIT_MMA)) break;
      tc_fence_after();
#pragma unroll
      for (int a = 0; a < (KV ? 2 : 1); ++a) {
        uint32_t o[16];
        tmem_ld_32x32b_x16(lanes + kColAcc + 64u * a + 16u * hc, o);
        tmem_ld_wait();
        float4* dst = reinterpret_cast<float4*>((a == 0 ? p.out0 : p.out1) +
                                                static_cast<size_t>(xrow + row) * 64 + 16 * hc);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          float4 v = make_float4(__uint_as_float(o[4 * k]), __uint_as_float(o[4 * k + 1]),
                                 __uint_as_float(o[4 * k + 2]), __uint_as_float(o[4 * k + 3]));
          if (KV && groups > 0) {
            const float4 w = dst[k];
            v = make_float4(w.x + v.x, w.y + v.y, w.z + v.z, w.w + v.w);
          }
          dst[k] = v;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (elect_one()) mbar_arrive(bar(kAccFree));
      ++groups;
    }
  }
  // this grid's end is also the dK / dV grid's: what follows on the stream needs both
  if (!KV && blockIdx.x == gridDim.x - 1) grid_dep_wait();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

cudaError_t launch_attention_bwd(const CUtensorMap& tmQ, const CUtensorMap& tmdO,
                                 const CUtensorMap& tmK, const CUtensorMap& tmV, AttnBwdParams p,
                                 float* dq, float* dk, float* dv, cudaStream_t s) {
  static const cudaError_t attr = [] {
    const cudaError_t e = cudaFuncSetAttribute(
        attn_bwd_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, attn_bwd::kSmem);
    return e != cudaSuccess
               ? e
               : cudaFuncSetAttribute(attn_bwd_kernel<false>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, attn_bwd::kSmem);
  }();
  if (attr != cudaSuccess) return attr;
  p.out0 = dk;
  p.out1 = dv;
  attn_bwd_kernel<true><<<p.G * (p.M / 128), attn_bwd::kThreads, attn_bwd::kSmem, s>>>(
      tmQ, tmdO, tmK, tmV, p);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  p.out0 = dq;
  p.out1 = nullptr;
  return launch_pdl(attn_bwd_kernel<false>, dim3(p.T * p.N * (p.Pc / 128)),
                    dim3(attn_bwd::kThreads), attn_bwd::kSmem, s, tmQ, tmdO, tmK, tmV, p);
}

}  // namespace fd
