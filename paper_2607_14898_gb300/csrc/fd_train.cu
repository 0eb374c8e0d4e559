// Streaming training step on the GPU (Sec. 3.3 "Training--Inference Consistency", Sec. 3.5
// Eq. loss, its L1 term): the loss of a clip of T latent frames and the gradient of every
// decoder parameter.
//
// Training through the rolling cache has the gradient of one pass over the whole clip under
// the block sliding-window mask (query chunk i sees key chunks i-W < j <= i), so the GPU runs
// all T chunks at once: the forward of every block with its activations kept, the L1 term of
// the pixels, then the backward block by block in reverse. Every product runs on the tensor
// cores with bf16 operands and fp32 accumulation:
//   - the linear layers and their input gradients dX = dY W (with the transposed weights): the
//     library's GEMM (gemm_view, gemm_tup); the weight gradients dW = dY^T X on dY and X as they
//     are (gemm_wgrad), or on transposed copies of a narrow input (the patch embedding of a
//     48-channel latent);
//   - the attention forward: the decode's batched attention kernel with one stream per query
//     chunk over the window of its key chunks, writing each row's log-sum-exp (attn_fwd);
//   - the attention backward (fd_attn_bwd.cu): two launches that recompute S = Q K^T and dP =
//     dO V^T on chip, one for dQ, one for dK and dV.
// Row-wise and element-wise steps (RMSNorm's backward, KV-norm / QK-norm with 3D-RoPE and their
// backward, GELU and GELU', the L1 term through the pixel shuffle, bias and gain sums) are the
// kernels of fd_train_rows.cuh; the attention backward's operands and what the materialised
// attention forward needs are below. That form (S, the band softmax, O = P V) runs where a stack's
// keys per chunk are not a multiple of 8.
//
// Rows: chunk c's L tokens sit at rows c Lp .. c Lp + L - 1 with Lp = 128 ceil(L / 128), the
// refined frame (c, tau) at rows (c r_t + tau) Lp ...; padding rows carry finite values
// forward (they are never keys: the softmax masks them) and exactly zero gradient backward, so
// they add nothing to any weight gradient.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <initializer_list>
#include <new>
#include <vector>

#include "fd_internal.h"
#include "fd_train_rows.cuh"
#include "flashdec.h"

namespace fd {
namespace train {


__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// y[c][r] = x[r][c] for a rows x cols block (pitches in elements), through a padded tile
template <typename T>
__global__ void transpose_kernel(const T* __restrict__ x, int rows, int cols, int ldx,
                                 T* __restrict__ y, int ldy) {
  __shared__ T tile[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    if (r < rows && c < cols) tile[i][threadIdx.x] = x[static_cast<size_t>(r) * ldx + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (r < rows && c < cols) y[static_cast<size_t>(c) * ldy + r] = tile[threadIdx.x][i];
  }
}

// Band softmax of one (query chunk, KV group): S fp32 [rows][n] (row pitch n), rows = the
// group's heads x the chunk's rows; column c is a key of a token (c mod Lp < L). P = softmax(S
// scale) over the valid columns (0 elsewhere) as bf16, and lse = log sum exp(S scale) of each
// row (natural log) for the backward. One warp per row: an online max / sum pass, then the
// write pass.
__global__ void softmax_lse_kernel(const float* __restrict__ S, int rows, int n, float scale,
                                   int Lp, int L, bf16* __restrict__ P16,
                                   float* __restrict__ lse) {
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const float* s = S + static_cast<size_t>(row) * n;
  float m = -INFINITY, sum = 0.f;
  for (int c = lane; c < n; c += 32) {
    if (c % Lp >= L) continue;
    const float v = s[c] * scale;
    if (v > m) {
      sum = sum * expf(m - v) + 1.0f;
      m = v;
    } else {
      sum += expf(v - m);
    }
  }
  const float mw = warp_max(m);
  sum = warp_sum(m == -INFINITY ? 0.f : sum * expf(m - mw));
  const float l = mw + logf(sum);
  for (int c = lane; c < n; c += 32) {
    const float p = c % Lp < L ? expf(s[c] * scale - l) : 0.f;
    P16[static_cast<size_t>(row) * n + c] = __float2bfloat16_rn(p);
  }
  if (lane == 0) lse[row] = l;
}

// Operands of the attention backward from dO fp32 rows [M][N 64], one warp per (row, head): dO
// head-major bf16 [M / Pc][N][Pc][64], delta[(c N + h) Pc + l] = sum_j dO O of the row and head
// (O bf16 rows), and lse of padding rows set to +inf (their P is then exp(-inf) = 0)
__global__ void attn_bwd_prep_kernel(const float* __restrict__ dO, const bf16* __restrict__ O,
                                     int M, int Pc, int Lp, int L, int N, bf16* __restrict__ do16,
                                     float* __restrict__ delta, float* __restrict__ lse) {
  const long long w = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= static_cast<long long>(M) * N) return;
  const int m = static_cast<int>(w / N), h = static_cast<int>(w % N);
  const size_t e = (static_cast<size_t>(m) * N + h) * kDh;
  const float* a = dO + e;
  const bf16* b = O + e;
  const float a0 = a[lane], a1 = a[lane + 32];
  float v = a0 * __bfloat162float(b[lane]) + a1 * __bfloat162float(b[lane + 32]);
  v = warp_sum(v);
  const int l = m % Pc;
  const size_t r = (static_cast<size_t>(m / Pc) * N + h) * Pc + l;
  do16[r * kDh + lane] = __float2bfloat16_rn(a0);
  do16[r * kDh + lane + 32] = __float2bfloat16_rn(a1);
  if (lane == 0) {
    delta[r] = v;
    if (l % Lp >= L) lse[r] = INFINITY;
  }
}

// head-major [M / Pc][N][Pc][64] fp32 -> bf16 rows [M][N 64]
__global__ void head_permute_kernel(const float* __restrict__ x, int M, int Pc, int N,
                                    bf16* __restrict__ y) {
  const long long total = static_cast<long long>(M) * N * kDh;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    // i indexes the rows layout: row m, head h, element j
    const long long m = i / (static_cast<long long>(N) * kDh);
    const int h = static_cast<int>(i / kDh % N), j = static_cast<int>(i % kDh);
    y[i] = __float2bfloat16_rn(x[((m / Pc * N + h) * Pc + m % Pc) * kDh + j]);
  }
}

}  // namespace train
}  // namespace fd

using fd::train::bf16;

// ---------------------------------------------------------------- the trainer object
struct fd_trainer_s {
  fd_config cfg;
  fd_weights w = nullptr;
  int T = 0;
  // shapes
  int C, H, W, p, D, N, G, NQ, QO, Dm, nb, nr, Wn, rt, rs, Cout, Cr, cin, gh, gw, L, Lp, MB, MR;
  int Dz = 0;          // MLP layer 1's outputs: Dm, or 2 Dm for the gated MLP (interleaved)
  bool gated = false;  // gated-SiLU MLP (the XL layout)
  bool f1 = false;     // chunk 0 emits one frame (first_chunk_frames = 1)
  float* dwz = nullptr;  // gated: layer 1's weight gradient (device order)
  float eps;
  std::vector<const void*> wt;   // device tensors of the weights, blob order
  std::vector<size_t> goff;      // element offset of each tensor in the gradient blob
  std::vector<void*> allocs;
  int* err = nullptr;
  float* zero_bias = nullptr;
  float2 *rope_t = nullptr, *rope_y = nullptr, *rope_x = nullptr;
  // transposed weights (bf16 [in][out]) of the linears used by the backward
  struct LinT {
    bf16 *qkv, *out, *mlp1, *mlp2;
  };
  std::vector<LinT> tB, tR;
  bf16 *t_tup = nullptr, *t_head1 = nullptr, *t_head2 = nullptr;
  // one stack's saved activations (per block) and its scratch
  struct Stack {
    int M, Pc;  // rows, rows per chunk
    std::vector<float*> h;  // block inputs (h[nblocks] = stack output), fp32 [M][D]
    std::vector<bf16*> u, q2, k2, v1, o, u2, a;
    std::vector<float*> qkv, hm, z, lse;  // lse [M / Pc][N][Pc]
    float* o32 = nullptr;  // head-major O of the materialised forward (scratch)
    // the fused band attention of the forward (the decode's batched attention kernel, one
    // stream per query chunk); off when its maps cannot be made
    struct {
      bool on = false;
      bf16* qr = nullptr;      // q rows [M][N 64]
      bf16* k = nullptr;       // K [G][pitch][64] of the real tokens
      __half* vt = nullptr;    // V^T [G][64][pitch]
      int pitch = 0, Lu = 0, parts = 1, pairs = 0;
      fd::AttnStream* streams = nullptr;  // device [T]
      int* steps = nullptr;               // device [T] = 0 .. T-1
      float* ws = nullptr;                // [T][ws_stride] partial results and counters
      size_t ws_stride = 0;
      CUtensorMap tmQ, tmQ8;
    } band;
  } sB, sR;
  // scratch
  bf16 *x0, *y16, *yh16, *a1, *vT, *do16, *P16, *dy16, *dyT = nullptr, *xT = nullptr,
      *dqkv16;
  float *z1, *F, *loss_part, *S, *delta, *dq2, *dk2, *dv1, *gA, *gB, *gC, *gtmp = nullptr;
  // heads of one KV group per product of the materialised attention forward, and per accumulator
  // chain of dK and dV (a divisor of N / G)
  int hs = 1;
  float *part_a = nullptr, *part_b = nullptr;  // partial column sums, two sets of part_elems
  size_t part_elems = 0;
  // per-kernel profile (fd_train_profile_enable): events around each launch, by kernel kind
  struct Rec {
    int kind;
    cudaEvent_t a, b;
  };
  bool prof = false;
  std::vector<cudaEvent_t> ev_free, ev_all;
  std::vector<Rec> rec;
  cudaEvent_t event() {
    if (!ev_free.empty()) {
      cudaEvent_t e = ev_free.back();
      ev_free.pop_back();
      return e;
    }
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    ev_all.push_back(e);
    return e;
  }
};

namespace {

template <typename T>
T* dalloc(fd_trainer_s* tr, size_t elems, bool& ok) {
  void* ptr = nullptr;
  if (!ok || cudaMalloc(&ptr, elems * sizeof(T) + 256) != cudaSuccess) {
    ok = false;
    return nullptr;
  }
  tr->allocs.push_back(ptr);
  if (cudaMemset(ptr, 0, elems * sizeof(T) + 256) != cudaSuccess) ok = false;
  return static_cast<T*>(ptr);
}

int blocks_for(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  return static_cast<int>(b < 1 ? 1 : (b > 65535 * 16 ? 65535 * 16 : b));
}

double rope_inv_freq(int i, double base) {
  using fd::train::kBandS;
  using fd::train::kBandT;
  int j, d;
  if (i < kBandT) { j = i; d = 2 * kBandT; }
  else if (i < kBandT + kBandS) { j = i - kBandT; d = 2 * kBandS; }
  else { j = i - kBandT - kBandS; d = 2 * kBandS; }
  return std::pow(base, -2.0 * j / d);
}

constexpr int kQkvBwdSmem = 2 * fd::train::kQkvUnits * fd::train::kQkvPad * 4;
// + the block's V^T: at most kQkvSlots groups
int qkv_fwd_smem(int G) {
  using namespace fd::train;
  return kQkvUnits * kQkvPad * 4 + std::min(G, kQkvSlots) * kDh * kQkvRows * 2;
}

// thread groups that share a block's rows in the RMSNorm backward (one for D >= 1024)
int norm_groups(int D) {
  const int threads = (D + 3) / 4;
  return threads >= 256 ? 1 : std::min(fd::train::kNormRows, 256 / threads);
}

// the launches of one step, in order on one stream; any failure ends the step
struct Run {
  fd_trainer_s* tr;
  cudaStream_t s;
  bool ok = true;
  cudaEvent_t t0 = nullptr;  // start event of the launch being profiled
  int t_kind = 0;

  void check(cudaError_t e) {
    if (e != cudaSuccess) ok = false;
  }
  // bracket the next launch with profile events (when the profile is enabled)
  bool begin(int kind) {
    if (!ok) return false;
    if (tr->prof) {
      t0 = tr->event();
      t_kind = kind;
      if (t0 != nullptr) check(cudaEventRecord(t0, s));
    }
    return ok;
  }
  void end() {
    if (t0 == nullptr) return;
    cudaEvent_t t1 = tr->event();
    if (t1 != nullptr) {
      check(cudaEventRecord(t1, s));
      tr->rec.push_back({t_kind, t0, t1});
    } else {
      tr->ev_free.push_back(t0);
    }
    t0 = nullptr;
  }
  void gemm(int kind, int epi, int M, int N, int K, const bf16* A, int lda, const bf16* Wm,
            int ldw, const float* bias, float* out, int ldo) {
    if (!begin(kind)) return;
    check(fd::gemm_view(epi, M, N, K, A, lda, Wm, ldw, bias ? bias : tr->zero_bias, out, ldo,
                        tr->err, s));
    end();
  }
  template <typename T>
  void transpose(const T* x, int rows, int cols, int ldx, T* y, int ldy) {
    if (!begin(FD_TK_TRANSPOSE)) return;
    dim3 grid((cols + 31) / 32, (rows + 31) / 32);
    fd::train::transpose_kernel<T><<<grid, dim3(32, 8), 0, s>>>(x, rows, cols, ldx, y, ldy);
    check(cudaGetLastError());
    end();
  }
  // room for `parts` partial rows of `cols` columns
  bool room(size_t parts, size_t cols) {
    if (parts * cols > tr->part_elems) ok = false;
    return ok;
  }
  // the last step of up to three column sums, in the same launch bracket as their partial sums
  void sum_parts(std::initializer_list<fd::train::SumJob> jobs) {
    fd::train::SumJobs js{};
    int n = 0, cols = 0;
    for (const fd::train::SumJob& j : jobs) {
      if (j.out == nullptr) continue;
      js.job[n++] = j;
      cols = std::max(cols, j.cols);
    }
    if (n == 0) return;
    fd::train::sum_parts_kernel<<<dim3((cols + 31) / 32, n), dim3(32, fd::train::kSumRows), 0, s>>>(
        js);
    check(cudaGetLastError());
  }
  void copy(float* dst, const float* src, size_t n) {
    if (!begin(FD_TK_POINTWISE)) return;
    check(cudaMemcpyAsync(dst, src, sizeof(float) * n, cudaMemcpyDeviceToDevice, s));
    end();
  }
  void rmsnorm(const float* x, const float* g, int M, bf16* u) {
    if (!begin(FD_TK_NORM)) return;
    check(fd::launch_rmsnorm(x, g, M, tr->D, tr->eps, u, s));
    end();
  }
  // dx = RMSNorm backward (+ add) in fp32 and bf16, the gain's gradient into grad, the column sums
  // of dx (the bias gradient of the linear whose output gradient dx is) into bias_grad if non-null
  void rmsnorm_bwd(const float* x, const float* g, const float* dy, const float* add, int M,
                   float* dx, bf16* dx16, float* grad, float* bias_grad) {
    using namespace fd::train;
    const int D = tr->D, groups = norm_groups(D);
    const int blocks = (M + kNormRows - 1) / kNormRows, parts = blocks * groups;
    if (!room(parts, D) || !begin(FD_TK_NORM)) return;
    rmsnorm_bwd_kernel<4><<<blocks, 256, 0, s>>>(x, g, dy, add, M, D, tr->eps, groups, dx, dx16,
                                                tr->part_a, bias_grad ? tr->part_b : nullptr);
    check(cudaGetLastError());
    sum_parts({{tr->part_a, parts, D, D, 0, grad}, {tr->part_b, parts, D, D, 0, bias_grad}});
    end();
  }
  // dz16 = da GELU'(z) (bf16) and the bias gradient, its column sums; cols % 4 == 0
  void gelu_bwd(const float* z, const float* da, int M, int cols, bf16* dz16, float* bias_grad) {
    using namespace fd::train;
    const int parts = (M + kRowBlock - 1) / kRowBlock;
    if (!room(parts, cols) || !begin(FD_TK_POINTWISE)) return;
    gelu_bwd_sum_kernel<<<dim3((cols + 1023) / 1024, parts), 256, 0, s>>>(z, da, M, cols, dz16,
                                                                         tr->part_a);
    check(cudaGetLastError());
    sum_parts({{tr->part_a, parts, cols, cols, 0, bias_grad}});
    end();
  }
  // weight gradient of a linear out = X W^T: dW [n_out][n_in] = dY^T X with dY16 [M][n_out]
  // and X16 [M][n_in] (bf16; K of the product = M rows, padding rows of dY are zero), on the
  // matrices as they are when both widths are whole 64-column groups
  void wgrad(const bf16* dY16, int n_out, const bf16* X16, int n_in, int M, float* dW) {
    if (n_out % 64 == 0 && n_in % 64 == 0) {
      if (!begin(FD_TK_WGRAD)) return;
      check(fd::gemm_wgrad(n_out, n_in, M, dY16, X16, tr->zero_bias, dW, tr->err, s));
      end();
      return;
    }
    // narrow inputs (the patch embedding of a 48-channel latent)
    bf16* dyT = tr->dyT;
    bf16* xT = tr->xT;
    transpose(dY16, M, n_out, n_out, dyT, M);
    transpose(X16, M, n_in, n_in, xT, M);
    if (n_in % 32 == 0) {
      gemm(FD_TK_WGRAD, fd::EPI_F32, n_out, n_in, M, dyT, M, xT, M, nullptr, dW, n_in);
    } else {  // the product in the other orientation (its N = n_out), then transposed
      gemm(FD_TK_WGRAD, fd::EPI_F32, n_in, n_out, M, xT, M, dyT, M, nullptr, tr->gtmp, n_out);
      transpose(tr->gtmp, n_in, n_out, n_out, dW, n_in);
    }
  }
  float* grad(float* g, size_t entry) { return g + tr->goff[entry]; }
  const float* wf(size_t entry) { return static_cast<const float*>(tr->wt[entry]); }
  const bf16* wb(size_t entry) { return static_cast<const bf16*>(tr->wt[entry]); }
};

// blob entries of block b of a stack starting at entry e0: norm1.g, qkv.w, qkv.b, knorm.g,
// (vnorm|qnorm).g, out.w, out.b, norm2.g, mlp1.w, mlp1.b, mlp2.w, mlp2.b
enum { kN1 = 0, kQW, kQB, kKG, kG2, kOW, kOB, kN2, kM1W, kM1B, kM2W, kM2B, kBlockEntries };

// attention forward of one block (Sec. 3.3, Eq. attention over the chunk window): O rows (bf16)
// into st.o and each row's log-sum-exp into st.lse. On the batched attention kernel when the
// stack's band maps exist; else materialised per (query chunk i, KV group g): the rows of the
// group's heads form one product with the window's keys (chunks max(0, i - W + 1) .. i,
// contiguous in k2 / v1): S = Q K^T, band softmax (P bf16 and the log-sum-exp), O = P V (head-
// major fp32 in st.o32, then permuted into st.o). A group's heads go tr->hs at a time (all of
// them unless S would pass its size bound).
void attn_fwd(Run& r, fd_trainer_s::Stack& st, int b) {
  fd_trainer_s* tr = r.tr;
  const int M = st.M, Pc = st.Pc, N = tr->N, hpg = N / tr->G, rows = tr->hs * Pc;
  if (st.band.on) {
    // the decode's batched attention kernel, one stream per query chunk: stream i's queries are
    // its Pc rows (padding rows computed, not used), its keys the window's real tokens; O as
    // bf16 rows into st.o, each row's log-sum-exp into st.lse
    auto& bd = st.band;
    fd::AttnParams a{};
    a.Lq = Pc; a.heads = N; a.groups = tr->G; a.ring_pitch = bd.pitch;
    a.rows_per_chunk = bd.Lu; a.window = tr->Wn; a.step_dev = bd.steps; a.n_keys_host = 0;
    a.out = st.o[b]; a.ld_out = tr->NQ;
    a.scale_log2 = static_cast<float>(1.4426950408889634 / 8.0);
    a.err = tr->err;
    a.lq_pad = fd::attention_lq_pad(Pc);
    a.parts = bd.parts;
    fd::attention_workspace_split(bd.ws, bd.parts, bd.pairs, a);
    a.streams = bd.streams; a.n_streams = tr->T; a.q_rows_stream = Pc;
    a.ws_stride = bd.ws_stride;
    a.lse = st.lse[b]; a.lse_pitch = Pc;
    if (r.begin(FD_TK_ATTN_GEMM)) {
      r.check(fd::launch_attention(bd.tmQ, bd.tmQ8, bd.tmQ, bd.tmQ, a, r.s));
      r.end();
    }
    return;
  }
  // V^T [G][64][M] for the P V products
  for (int g = 0; g < tr->G; ++g)
    r.transpose(st.v1[b] + static_cast<size_t>(g) * M * 64, M, 64, 64,
                tr->vT + static_cast<size_t>(g) * 64 * M, M);
  for (int i = 0; i < tr->T; ++i) {
    const int j0 = i - tr->Wn + 1 > 0 ? i - tr->Wn + 1 : 0;
    const int k0 = j0 * Pc, nk = (i + 1) * Pc - k0;
    for (int h0 = 0; h0 < N; h0 += tr->hs) {  // tr->hs heads of group h0 / hpg at a time
      const int g = h0 / hpg;
      const size_t q0 = (static_cast<size_t>(i) * N + h0) * Pc;  // first row, head-major
      r.gemm(FD_TK_ATTN_GEMM, fd::EPI_F32, rows, nk, 64, st.q2[b] + q0 * 64, 64,
             st.k2[b] + (static_cast<size_t>(g) * M + k0) * 64, 64, nullptr, tr->S, nk);
      if (r.begin(FD_TK_SOFTMAX)) {
        fd::train::softmax_lse_kernel<<<(rows + 7) / 8, 256, 0, r.s>>>(
            tr->S, rows, nk, 0.125f, tr->Lp, tr->L, tr->P16, st.lse[b] + q0);
        r.check(cudaGetLastError());
        r.end();
      }
      r.gemm(FD_TK_ATTN_GEMM, fd::EPI_F32, rows, 64, nk, tr->P16, nk,
             tr->vT + static_cast<size_t>(g) * 64 * M + k0, M, nullptr, st.o32 + q0 * 64, 64);
    }
  }
  if (r.begin(FD_TK_POINTWISE)) {  // O rows (bf16) for the output projection
    const long long n = static_cast<long long>(M) * tr->NQ;
    fd::train::head_permute_kernel<<<blocks_for(n, 256), 256, 0, r.s>>>(st.o32, M, Pc, N,
                                                                         st.o[b]);
    r.check(cudaGetLastError());
    r.end();
  }
}

// attention backward of one block: dq2 (fp32, the head-major layout of q2), dk2, dv1 (fp32
// [G][M][64], summed over the query chunks whose windows hold each key and the group's heads)
// from dO (tr->gA, fp32 rows [M][N 64])
void attn_bwd(Run& r, fd_trainer_s::Stack& st, int b) {
  fd_trainer_s* tr = r.tr;
  const int M = st.M, Pc = st.Pc, N = tr->N;
  if (r.begin(FD_TK_SOFTMAX)) {
    const long long threads = static_cast<long long>(M) * N * 32;
    fd::train::attn_bwd_prep_kernel<<<static_cast<unsigned>((threads + 255) / 256), 256, 0, r.s>>>(
        tr->gA, st.o[b], M, Pc, tr->Lp, tr->L, N, tr->do16, tr->delta, st.lse[b]);
    r.check(cudaGetLastError());
    r.end();
  }
  if (r.begin(FD_TK_ATTN_GEMM)) {
    const fd::AttnBwdParams p{st.lse[b], tr->delta, nullptr, nullptr, tr->T, N, tr->G, tr->Wn, Pc,
                              tr->Lp, tr->L, M, tr->hs, tr->err};
    r.check(fd::attention_bwd(st.q2[b], tr->do16, st.k2[b], st.v1[b], p, tr->dq2, tr->dk2, tr->dv1,
                              r.s));
    r.end();
  }
}

// one block forward (Sec. 3.2): st.h[b] -> st.h[b + 1], activations kept
void block_fwd(Run& r, fd_trainer_s::Stack& st, int b, size_t e0) {
  fd_trainer_s* tr = r.tr;
  const int M = st.M;
  r.rmsnorm(st.h[b], r.wf(e0 + kN1), M, st.u[b]);
  r.gemm(FD_TK_LINEAR, fd::EPI_F32, M, tr->QO, tr->D, st.u[b], tr->D, r.wb(e0 + kQW), tr->D, r.wf(e0 + kQB),
         st.qkv[b], tr->QO);
  if (r.begin(FD_TK_NORM)) {
    using namespace fd::train;
    const Rope rp{tr->rope_t, tr->rope_y, tr->rope_x};
    const QkvShape sh{M, st.Pc, tr->Lp, tr->L, tr->gw, tr->N, tr->G, tr->cfg.qk_norm};
    const int slots = tr->N + 2 * tr->G;
    qkv_fwd_kernel<<<dim3(M / kQkvRows, (slots + kQkvSlots - 1) / kQkvSlots), kQkvUnits,
                     qkv_fwd_smem(tr->G), r.s>>>(
        st.qkv[b], sh, r.wf(e0 + kKG), r.wf(e0 + kG2), tr->eps, rp, st.q2[b], st.k2[b], st.v1[b],
        st.band.on ? st.band.qr : nullptr, st.band.k, st.band.vt, st.band.pitch);
    r.check(cudaGetLastError());
    r.end();
  }
  attn_fwd(r, st, b);
  r.copy(st.hm[b], st.h[b], static_cast<size_t>(M) * tr->D);
  r.gemm(FD_TK_LINEAR, fd::EPI_RESID, M, tr->D, tr->NQ, st.o[b], tr->NQ, r.wb(e0 + kOW), tr->NQ,
         r.wf(e0 + kOB), st.hm[b], tr->D);
  r.rmsnorm(st.hm[b], r.wf(e0 + kN2), M, st.u2[b]);
  r.gemm(FD_TK_LINEAR, fd::EPI_F32, M, tr->Dz, tr->D, st.u2[b], tr->D, r.wb(e0 + kM1W), tr->D,
         r.wf(e0 + kM1B), st.z[b], tr->Dz);
  if (r.begin(FD_TK_POINTWISE)) {
    const long long n = static_cast<long long>(M) * tr->Dm;
    if (tr->gated)
      fd::train::swiglu_fwd_kernel<<<blocks_for(n / 4, 256), 256, 0, r.s>>>(st.z[b], M, tr->Dm,
                                                                             st.a[b]);
    else
      fd::train::gelu_fwd_kernel<<<blocks_for(n / 4, 256), 256, 0, r.s>>>(
          reinterpret_cast<const float4*>(st.z[b]), n / 4, reinterpret_cast<uint2*>(st.a[b]));
    r.check(cudaGetLastError());
    r.end();
  }
  r.copy(st.h[b + 1], st.hm[b], static_cast<size_t>(M) * tr->D);
  r.gemm(FD_TK_LINEAR, fd::EPI_RESID, M, tr->D, tr->Dm, st.a[b], tr->Dm, r.wb(e0 + kM2W), tr->Dm,
         r.wf(e0 + kM2B), st.h[b + 1], tr->D);
}

// one block backward: dho (tr->gB, fp32 [M][D], and its bf16 copy tr->dy16; the gradient of this
// block's second MLP bias is its column sums, already taken) -> dh_in (tr->gB and tr->dy16),
// gradients into g; prev_bias: where the column sums of dh_in belong (the bias gradient of what
// produced the block's input), or null
void block_bwd(Run& r, fd_trainer_s::Stack& st, int b, size_t e0,
               const fd_trainer_s::LinT& lt, float* g, float* prev_bias) {
  fd_trainer_s* tr = r.tr;
  const int M = st.M, D = tr->D, Dm = tr->Dm, NQ = tr->NQ, QO = tr->QO;
  // MLP layer 2
  r.gemm(FD_TK_DGRAD, fd::EPI_F32, M, Dm, D, tr->dy16, D, lt.mlp2, D, nullptr, tr->gC, Dm);  // da
  r.wgrad(tr->dy16, D, st.a[b], Dm, M, r.grad(g, e0 + kM2W));
  // GELU' (or the gated SiLU's derivative into the interleaved dz)
  const int Dz = tr->Dz;
  if (tr->gated) {
    const int parts = (M + fd::train::kRowBlock - 1) / fd::train::kRowBlock;
    if (r.room(parts, Dz) && r.begin(FD_TK_POINTWISE)) {
      fd::train::swiglu_bwd_sum_kernel<<<dim3((Dm + 1023) / 1024, parts), 256, 0, r.s>>>(
          st.z[b], tr->gC, M, Dm, tr->dqkv16, tr->part_a);
      r.check(cudaGetLastError());
      r.sum_parts({{tr->part_a, parts, Dz, Dz, Dm, r.grad(g, e0 + kM1B)}});
      r.end();
    }
  } else {
    r.gelu_bwd(st.z[b], tr->gC, M, Dm, tr->dqkv16, r.grad(g, e0 + kM1B));
  }
  // MLP layer 1
  r.gemm(FD_TK_DGRAD, fd::EPI_F32, M, D, Dz, tr->dqkv16, Dz, lt.mlp1, Dz, nullptr, tr->gA, D);  // du2
  if (tr->gated) {  // the weight gradient in the device's interleaved rows, then in the blob's order
    r.wgrad(tr->dqkv16, Dz, st.u2[b], D, M, tr->dwz);
    if (r.begin(FD_TK_POINTWISE)) {
      const long long n = static_cast<long long>(Dz) * D / 4;
      fd::train::gated_rows_kernel<<<blocks_for(n, 256), 256, 0, r.s>>>(
          reinterpret_cast<const float4*>(tr->dwz), Dz, D / 4,
          reinterpret_cast<float4*>(r.grad(g, e0 + kM1W)));
      r.check(cudaGetLastError());
      r.end();
    }
  } else {
    r.wgrad(tr->dqkv16, Dz, st.u2[b], D, M, r.grad(g, e0 + kM1W));
  }
  // RMSNorm 2, plus the residual: dhm (gC, dy16); its column sums are the output bias's gradient
  r.rmsnorm_bwd(st.hm[b], r.wf(e0 + kN2), tr->gA, tr->gB, M, tr->gC, tr->dy16,
                r.grad(g, e0 + kN2), r.grad(g, e0 + kOB));
  // output projection
  r.gemm(FD_TK_DGRAD, fd::EPI_F32, M, NQ, D, tr->dy16, D, lt.out, D, nullptr, tr->gA, NQ);  // dO (fp32)
  r.wgrad(tr->dy16, D, st.o[b], NQ, M, r.grad(g, e0 + kOW));
  // attention (reads dO from gA)
  attn_bwd(r, st, b);
  // KV-norm / QK-norm and RoPE backward, the bias's and the two gains' gradients
  const int slots = tr->N + 2 * tr->G;
  const int bx = M / fd::train::kQkvRows;
  const int by = (slots + fd::train::kQkvSlots - 1) / fd::train::kQkvSlots;
  if (r.room(bx, QO) && r.room(static_cast<size_t>(bx) * by, 128) && r.begin(FD_TK_NORM)) {
    const fd::train::Rope rp{tr->rope_t, tr->rope_y, tr->rope_x};
    const fd::train::QkvShape sh{M, st.Pc, tr->Lp, tr->L, tr->gw, tr->N, tr->G, tr->cfg.qk_norm};
    fd::train::qkv_bwd_kernel<<<dim3(bx, by), fd::train::kQkvUnits, kQkvBwdSmem, r.s>>>(
        st.qkv[b], tr->dq2, tr->dk2, tr->dv1, sh, r.wf(e0 + kKG), r.wf(e0 + kG2), tr->eps, rp,
        tr->dqkv16, tr->part_a, tr->part_b);
    r.check(cudaGetLastError());
    r.sum_parts({{tr->part_a, bx, QO, QO, 0, r.grad(g, e0 + kQB)},
                 {tr->part_b, bx * by, 128, 64, 0, r.grad(g, e0 + kKG)},
                 {tr->part_b + 64, bx * by, 128, 64, 0, r.grad(g, e0 + kG2)}});
    r.end();
  }
  // QKV projection
  r.gemm(FD_TK_DGRAD, fd::EPI_F32, M, D, QO, tr->dqkv16, QO, lt.qkv, QO, nullptr, tr->gA, D);  // du
  r.wgrad(tr->dqkv16, QO, st.u[b], D, M, r.grad(g, e0 + kQW));
  // RMSNorm 1, plus the residual: dh_in
  r.rmsnorm_bwd(st.h[b], r.wf(e0 + kN1), tr->gA, tr->gC, M, tr->gB, tr->dy16,
                r.grad(g, e0 + kN1), prev_bias);
}

}  // namespace

extern "C" {

size_t fd_train_grad_elems(const fd_config* cfg) { return fd_weights_blob_elems(cfg); }

fd_status fd_train_create(const fd_config* cfg, fd_weights w, int chunks, fd_trainer* out) {
  if (out == nullptr || w == nullptr || cfg == nullptr) return FD_ERR_INVALID_ARG;
  *out = nullptr;
  const fd_config* wc = fd::weights_config(w);
  if (fd_weights_blob_elems(cfg) == 0 || std::memcmp(cfg, wc, sizeof(fd_config)) != 0)
    return FD_ERR_CONFIG;
  // the bf16-valued decoder: GELU or gated-SiLU MLPs, r_t frames per chunk or one from chunk 0
  if (cfg->mlp_fp8) return FD_ERR_CONFIG;
  if (chunks < 1 || chunks > 256) return FD_ERR_INVALID_ARG;
  static const cudaError_t attr[2] = {
      cudaFuncSetAttribute(fd::train::qkv_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           kQkvBwdSmem),
      cudaFuncSetAttribute(fd::train::qkv_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           qkv_fwd_smem(fd::train::kQkvSlots))};
  if (attr[0] != cudaSuccess || attr[1] != cudaSuccess) return FD_ERR_CUDA;
  fd_trainer tr = new (std::nothrow) fd_trainer_s;
  if (tr == nullptr) return FD_ERR_OOM;
  tr->cfg = *cfg;
  tr->w = w;
  tr->T = chunks;
  tr->C = cfg->latent_channels; tr->H = cfg->latent_h; tr->W = cfg->latent_w; tr->p = cfg->patch;
  tr->D = cfg->hidden; tr->N = cfg->heads; tr->G = cfg->kv_groups; tr->NQ = tr->N * 64;
  tr->QO = (tr->N + 2 * tr->G) * 64; tr->Dm = cfg->mlp_ratio * tr->D; tr->nb = cfg->n_blocks;
  tr->gated = cfg->mlp_gated != 0;
  tr->Dz = tr->gated ? 2 * tr->Dm : tr->Dm;
  tr->f1 = cfg->first_chunk_frames == 1;
  tr->nr = cfg->n_refine; tr->Wn = cfg->window; tr->rt = cfg->r_t;
  tr->rs = cfg->vae_spatial * cfg->patch; tr->Cout = cfg->out_channels;
  tr->Cr = tr->Cout * tr->rs * tr->rs; tr->cin = tr->C * tr->p * tr->p;
  tr->gh = tr->H / tr->p; tr->gw = tr->W / tr->p; tr->L = tr->gh * tr->gw;
  tr->Lp = (tr->L + 127) / 128 * 128;
  tr->MB = tr->T * tr->Lp;
  tr->MR = tr->T * tr->rt * tr->Lp;
  tr->eps = cfg->norm_eps;
  // tensors of the weights and their offsets in the gradient blob
  const size_t n_ent = fd::weights_entries(w, nullptr, 0);
  tr->wt.resize(n_ent);
  fd::weights_entries(w, tr->wt.data(), n_ent);
  {
    const size_t D = tr->D, blk[kBlockEntries] = {
        D, static_cast<size_t>(tr->QO) * D, static_cast<size_t>(tr->QO), 64, 64,
        D * tr->NQ, D, D, static_cast<size_t>(tr->Dz) * D, static_cast<size_t>(tr->Dz),
        D * tr->Dm, D};
    std::vector<size_t> elems = {D * tr->cin, D};
    for (int b = 0; b < tr->nb; ++b) elems.insert(elems.end(), blk, blk + kBlockEntries);
    elems.push_back(D);
    elems.push_back(static_cast<size_t>(tr->rt) * D * D);
    elems.push_back(static_cast<size_t>(tr->rt) * D);
    for (int b = 0; b < tr->nr; ++b) elems.insert(elems.end(), blk, blk + kBlockEntries);
    elems.insert(elems.end(), {D, D * D, D, static_cast<size_t>(tr->Cr) * D,
                               static_cast<size_t>(tr->Cr)});
    if (elems.size() != n_ent) {
      delete tr;
      return FD_ERR_CONFIG;
    }
    size_t off = 0;
    for (size_t e : elems) {
      tr->goff.push_back(off);
      off += e;
    }
  }
  bool ok = true;
  const int D = tr->D, Dm = tr->Dm, QO = tr->QO, NQ = tr->NQ, G = tr->G, MB = tr->MB,
            MR = tr->MR;
  const int Mmax = MB > MR ? MB : MR;
  const int Pmax = tr->rt > 1 ? tr->rt * tr->Lp : tr->Lp;
  const int Kmax = std::min(tr->T, tr->Wn) * Pmax;  // keys of one query chunk's window
  // heads per product of the materialised forward: all of a KV group's, unless its S (fp32
  // [heads Pmax][Kmax]) would pass 512 M elements; then the largest divisor of the group size that
  // stays within it. The attention backward stores no scores, but adds dK and dV up in chains of
  // the same heads: they are the sums of the products that it replaced, to the bit.
  {
    const int hpg = tr->N / tr->G;
    tr->hs = 1;
    for (int d = hpg; d >= 1; --d)
      if (hpg % d == 0 && static_cast<size_t>(d) * Pmax * Kmax <= (static_cast<size_t>(1) << 29)) {
        tr->hs = d;
        break;
      }
  }
  const size_t RK = static_cast<size_t>(tr->hs) * Pmax * Kmax;  // one product's scores
  tr->err = dalloc<int>(tr, 4, ok);
  tr->zero_bias = dalloc<float>(tr, std::max({Kmax, Dm, QO, NQ, tr->rt * D, tr->Cr, D}), ok);
  // RoPE tables, fp64 on the host (frames 0 .. T r_t - 1; rows; columns)
  {
    const int F = tr->T * tr->rt;
    const double base = cfg->rope_base;
    std::vector<float2> ht(static_cast<size_t>(F) * fd::train::kBandT),
        hy(static_cast<size_t>(tr->gh) * fd::train::kBandS),
        hx(static_cast<size_t>(tr->gw) * fd::train::kBandS);
    for (int f = 0; f < F; ++f)
      for (int i = 0; i < fd::train::kBandT; ++i) {
        const double a = f * rope_inv_freq(i, base);
        ht[f * fd::train::kBandT + i] = make_float2(static_cast<float>(std::cos(a)),
                                                    static_cast<float>(std::sin(a)));
      }
    for (int y = 0; y < tr->gh; ++y)
      for (int i = 0; i < fd::train::kBandS; ++i) {
        const double a = y * rope_inv_freq(fd::train::kBandT + i, base);
        hy[y * fd::train::kBandS + i] = make_float2(static_cast<float>(std::cos(a)),
                                                    static_cast<float>(std::sin(a)));
      }
    for (int x = 0; x < tr->gw; ++x)
      for (int i = 0; i < fd::train::kBandS; ++i) {
        const double a = x * rope_inv_freq(fd::train::kBandT + fd::train::kBandS + i, base);
        hx[x * fd::train::kBandS + i] = make_float2(static_cast<float>(std::cos(a)),
                                                    static_cast<float>(std::sin(a)));
      }
    tr->rope_t = dalloc<float2>(tr, ht.size(), ok);
    tr->rope_y = dalloc<float2>(tr, hy.size(), ok);
    tr->rope_x = dalloc<float2>(tr, hx.size(), ok);
    if (ok)
      ok = cudaMemcpy(tr->rope_t, ht.data(), ht.size() * sizeof(float2), cudaMemcpyHostToDevice) ==
               cudaSuccess &&
           cudaMemcpy(tr->rope_y, hy.data(), hy.size() * sizeof(float2), cudaMemcpyHostToDevice) ==
               cudaSuccess &&
           cudaMemcpy(tr->rope_x, hx.data(), hx.size() * sizeof(float2), cudaMemcpyHostToDevice) ==
               cudaSuccess;
  }
  auto alloc_stack = [&](fd_trainer_s::Stack& st, int M, int Pc, int nblocks) {
    st.M = M;
    st.Pc = Pc;
    for (int b = 0; b <= nblocks; ++b) st.h.push_back(dalloc<float>(tr, static_cast<size_t>(M) * D, ok));
    for (int b = 0; b < nblocks; ++b) {
      st.u.push_back(dalloc<bf16>(tr, static_cast<size_t>(M) * D, ok));
      st.qkv.push_back(dalloc<float>(tr, static_cast<size_t>(M) * QO, ok));
      st.q2.push_back(dalloc<bf16>(tr, static_cast<size_t>(M) * NQ, ok));
      st.k2.push_back(dalloc<bf16>(tr, static_cast<size_t>(G) * M * 64, ok));
      st.v1.push_back(dalloc<bf16>(tr, static_cast<size_t>(G) * M * 64, ok));
      st.lse.push_back(dalloc<float>(tr, static_cast<size_t>(M) * tr->N, ok));
      st.o.push_back(dalloc<bf16>(tr, static_cast<size_t>(M) * NQ, ok));
      st.hm.push_back(dalloc<float>(tr, static_cast<size_t>(M) * D, ok));
      st.u2.push_back(dalloc<bf16>(tr, static_cast<size_t>(M) * D, ok));
      st.z.push_back(dalloc<float>(tr, static_cast<size_t>(M) * tr->Dz, ok));
      st.a.push_back(dalloc<bf16>(tr, static_cast<size_t>(M) * Dm, ok));
    }
  };
  alloc_stack(tr->sB, MB, tr->Lp, tr->nb);
  alloc_stack(tr->sR, MR, tr->rt * tr->Lp, tr->nr);
  // the forward's band attention: per stack, the query rows, unpadded K / V^T (allocated
  // zeroed: keys past the clip read zeros), the kernel's per-chunk stream table and its
  // workspace (counters zero); else the materialised forward with its head-major O scratch
  int sms = 0, dev = 0;
  if (ok) ok = cudaGetDevice(&dev) == cudaSuccess &&
               cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
  auto setup_band = [&](fd_trainer_s::Stack& st, int Lu) {
    auto& bd = st.band;
    const int T = tr->T, M = st.M;
    bd.Lu = Lu;
    bd.pitch = (T * Lu + 127) / 128 * 128;
    bd.on = ok && (Lu % 8 == 0 || T == 1);
    if (bd.on) {
      bd.qr = dalloc<bf16>(tr, static_cast<size_t>(M) * NQ, ok);
      bd.k = dalloc<bf16>(tr, static_cast<size_t>(G) * bd.pitch * 64, ok);
      bd.vt = dalloc<__half>(tr, static_cast<size_t>(G) * 64 * bd.pitch, ok);
      bd.steps = dalloc<int>(tr, T, ok);
      bd.streams = dalloc<fd::AttnStream>(tr, T, ok);
      const int keys = std::min(T, tr->Wn) * Lu;
      bd.pairs = fd::attention_units(st.Pc, tr->N, G);
      const long long units = static_cast<long long>(bd.pairs) * ((keys + 127) / 128);
      bd.parts = static_cast<int>(std::max(1LL, std::min<long long>(std::max(1, sms / T), units)));
      bd.ws_stride = (fd::attention_workspace_floats(bd.parts, bd.pairs) + 63) / 64 * 64;
      bd.ws = dalloc<float>(tr, bd.ws_stride * T, ok);
    }
    if (bd.on && ok) {
      std::vector<fd::AttnStream> host(T);
      std::vector<int> steps(T);
      for (int i = 0; i < T; ++i) steps[i] = i;
      bd.on = fd::band_attention_maps(host.data(), T, tr->Wn, Lu, G, bd.pitch, bd.k, bd.vt,
                                      bd.steps, tr->err) &&
              fd::attention_q_maps(&bd.tmQ, &bd.tmQ8, bd.qr, M, tr->N);
      if (bd.on)
        ok = cudaMemcpy(bd.streams, host.data(), T * sizeof(fd::AttnStream),
                        cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(bd.steps, steps.data(), T * sizeof(int), cudaMemcpyHostToDevice) ==
                 cudaSuccess;
    }
    if (!bd.on) st.o32 = dalloc<float>(tr, static_cast<size_t>(M) * NQ, ok);
  };
  setup_band(tr->sB, tr->L);
  setup_band(tr->sR, tr->rt * tr->L);
  const size_t wide = static_cast<size_t>(Mmax) *
                      std::max({D, tr->Dz, QO, NQ, tr->rt * D, tr->Cr});
  tr->x0 = dalloc<bf16>(tr, static_cast<size_t>(MB) * tr->cin, ok);
  tr->y16 = dalloc<bf16>(tr, static_cast<size_t>(MB) * D, ok);
  tr->yh16 = dalloc<bf16>(tr, static_cast<size_t>(MR) * D, ok);
  tr->a1 = dalloc<bf16>(tr, static_cast<size_t>(MR) * D, ok);
  tr->vT = dalloc<bf16>(tr, static_cast<size_t>(G) * 64 * Mmax, ok);
  tr->do16 = dalloc<bf16>(tr, static_cast<size_t>(Mmax) * NQ, ok);
  // S and P of the materialised forward (a stack whose band attention is off)
  const bool materialised = !tr->sB.band.on || !tr->sR.band.on;
  if (materialised) tr->P16 = dalloc<bf16>(tr, RK, ok);
  tr->dy16 = dalloc<bf16>(tr, wide, ok);
  if (tr->cin % 64) {
    tr->dyT = dalloc<bf16>(tr, static_cast<size_t>(MB) * D, ok);
    tr->xT = dalloc<bf16>(tr, static_cast<size_t>(MB) * tr->cin, ok);
  }
  tr->dqkv16 = dalloc<bf16>(tr, wide, ok);
  tr->z1 = dalloc<float>(tr, static_cast<size_t>(MR) * D, ok);
  tr->F = dalloc<float>(tr, static_cast<size_t>(MR) * tr->Cr, ok);
  tr->loss_part = dalloc<float>(
      tr,
      static_cast<size_t>((MR + fd::train::kRowBlock - 1) / fd::train::kRowBlock) *
          ((tr->Cr + 1023) / 1024),
      ok);
  if (materialised) tr->S = dalloc<float>(tr, RK, ok);
  tr->delta = dalloc<float>(tr, static_cast<size_t>(Mmax) * tr->N, ok);
  {  // partial rows of the column sums: per kRowBlock rows, per kNormRows rows and group, per
     // kQkvRows rows (and kQkvSlots slots, 128 columns)
    using namespace fd::train;
    const size_t m = Mmax, slots = tr->N + 2 * G;
    tr->part_elems = std::max({(m + kRowBlock - 1) / kRowBlock *
                                   std::max({tr->Dz, tr->rt * D, tr->Cr, D}),
                               (m + kNormRows - 1) / kNormRows * norm_groups(D) * D,
                               m / kQkvRows * QO,
                               m / kQkvRows * ((slots + kQkvSlots - 1) / kQkvSlots) * 128});
    tr->part_a = dalloc<float>(tr, tr->part_elems, ok);
    tr->part_b = dalloc<float>(tr, tr->part_elems, ok);
  }
  tr->dq2 = dalloc<float>(tr, static_cast<size_t>(Mmax) * NQ, ok);
  tr->dk2 = dalloc<float>(tr, static_cast<size_t>(G) * Mmax * 64, ok);
  tr->dv1 = dalloc<float>(tr, static_cast<size_t>(G) * Mmax * 64, ok);
  tr->gA = dalloc<float>(tr, wide, ok);
  tr->gB = dalloc<float>(tr, wide, ok);
  tr->gC = dalloc<float>(tr, wide, ok);
  if (tr->cin % 64) tr->gtmp = dalloc<float>(tr, static_cast<size_t>(D) * tr->cin, ok);
  if (tr->gated) {
    tr->dwz = dalloc<float>(tr, static_cast<size_t>(tr->Dz) * D, ok);
  }
  // transposed weights [in][out] for the input gradients dX = dY W
  auto wT = [&](size_t entry, int n_out, int n_in) -> bf16* {
    bf16* t = dalloc<bf16>(tr, static_cast<size_t>(n_out) * n_in, ok);
    if (ok) {
      dim3 grid((n_in + 31) / 32, (n_out + 31) / 32);
      fd::train::transpose_kernel<bf16><<<grid, dim3(32, 8)>>>(
          static_cast<const bf16*>(tr->wt[entry]), n_out, n_in, n_in, t, n_out);
      ok = cudaGetLastError() == cudaSuccess;
    }
    return t;
  };
  auto stackT = [&](std::vector<fd_trainer_s::LinT>& v, size_t e0, int nblocks) {
    for (int b = 0; b < nblocks; ++b) {
      const size_t e = e0 + static_cast<size_t>(b) * kBlockEntries;
      v.push_back({wT(e + kQW, QO, D), wT(e + kOW, D, NQ), wT(e + kM1W, tr->Dz, D),
                   wT(e + kM2W, D, Dm)});
    }
  };
  const size_t eB = 2, eF = eB + static_cast<size_t>(tr->nb) * kBlockEntries;
  const size_t eR = eF + 3, eH = eR + static_cast<size_t>(tr->nr) * kBlockEntries;
  stackT(tr->tB, eB, tr->nb);
  tr->t_tup = wT(eF + 1, tr->rt * D, D);
  stackT(tr->tR, eR, tr->nr);
  tr->t_head1 = wT(eH + 1, D, D);
  tr->t_head2 = wT(eH + 3, tr->Cr, D);
  if (ok) ok = cudaDeviceSynchronize() == cudaSuccess;
  if (!ok) {
    for (void* ptr : tr->allocs) cudaFree(ptr);
    delete tr;
    return FD_ERR_OOM;
  }
  fd::weights_add_user(w, 1);
  *out = tr;
  return FD_OK;
}

fd_status fd_train_step(fd_trainer tr, const float* latents, const float* targets, float* loss,
                        float* grads, void* stream) {
  if (tr == nullptr || latents == nullptr || targets == nullptr || loss == nullptr ||
      grads == nullptr)
    return FD_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(latents) | reinterpret_cast<uintptr_t>(targets) |
       reinterpret_cast<uintptr_t>(grads)) & 15u)
    return FD_ERR_INVALID_ARG;
  Run r{tr, static_cast<cudaStream_t>(stream)};
  const int D = tr->D, MB = tr->MB, MR = tr->MR, rt = tr->rt;
  const size_t eB = 2, eF = eB + static_cast<size_t>(tr->nb) * kBlockEntries;
  const size_t eR = eF + 3, eH = eR + static_cast<size_t>(tr->nr) * kBlockEntries;
  if (r.begin(FD_TK_POINTWISE)) {
    r.check(cudaMemsetAsync(tr->err, 0, sizeof(int), r.s));
    r.end();
  }
  // ---- forward
  // patch-embedding (Eq. projection) of every chunk: PixelUnshuffle rows, then the linear
  const size_t chw = static_cast<size_t>(tr->C) * tr->H * tr->W;
  for (int c = 0; c < tr->T && r.begin(FD_TK_POINTWISE); ++c) {
    r.check(fd::launch_unshuffle(latents + c * chw, tr->C, tr->H, tr->W, tr->p,
                                 tr->x0 + static_cast<size_t>(c) * tr->Lp * tr->cin, r.s));
    r.end();
  }
  r.gemm(FD_TK_LINEAR, fd::EPI_F32, MB, D, tr->cin, tr->x0, tr->cin, r.wb(0), tr->cin, r.wf(1), tr->sB.h[0], D);
  for (int b = 0; b < tr->nb; ++b)
    block_fwd(r, tr->sB, b, eB + static_cast<size_t>(b) * kBlockEntries);
  // final norm and temporal upsampling (Eq. temporal_upsample): channel block tau -> frame tau
  const float* hBo = tr->sB.h[tr->nb];
  r.rmsnorm(hBo, r.wf(eF), MB, tr->y16);
  if (r.begin(FD_TK_LINEAR)) {
    r.check(fd::gemm_tup(MB, rt, tr->Lp, D, tr->y16, r.wb(eF + 1), r.wf(eF + 2), tr->sR.h[0],
                         tr->err, r.s));
    r.end();
  }
  for (int b = 0; b < tr->nr; ++b)
    block_fwd(r, tr->sR, b, eR + static_cast<size_t>(b) * kBlockEntries);
  // head (Sec. 3.4 Step 3): RMSNorm, Linear + GELU, Linear to C r_s^2 per refined token
  const float* hRo = tr->sR.h[tr->nr];
  r.rmsnorm(hRo, r.wf(eH), MR, tr->yh16);
  r.gemm(FD_TK_LINEAR, fd::EPI_F32, MR, D, D, tr->yh16, D, r.wb(eH + 1), D, r.wf(eH + 2), tr->z1, D);
  if (r.begin(FD_TK_POINTWISE)) {
    const long long n4 = static_cast<long long>(MR) * D / 4;
    fd::train::gelu_fwd_kernel<<<blocks_for(n4, 256), 256, 0, r.s>>>(
        reinterpret_cast<const float4*>(tr->z1), n4, reinterpret_cast<uint2*>(tr->a1));
    r.check(cudaGetLastError());
    r.end();
  }
  r.gemm(FD_TK_LINEAR, fd::EPI_F32, MR, tr->Cr, D, tr->a1, D, r.wb(eH + 3), D, r.wf(eH + 4), tr->F, tr->Cr);
  // ---- loss (L1 over every pixel of the clip) and its gradient through the pixel shuffle
  const int first = tr->f1 ? 1 : rt;  // frames chunk 0 emits (reading R16)
  const double total = (static_cast<double>(tr->T - 1) * rt + first) * tr->Cout * tr->gh *
                       tr->rs * tr->gw * tr->rs;
  const float inv_total = static_cast<float>(1.0 / total);
  float* g = grads;
  using fd::train::kRowBlock;
  {
    const int parts = (MR + kRowBlock - 1) / kRowBlock, strips = (tr->Cr + 1023) / 1024;
    if (r.room(parts, tr->Cr) && r.begin(FD_TK_POINTWISE)) {
      const fd::train::PixelGrid pg{tr->T, rt, first, tr->Lp, tr->L, tr->gh, tr->gw, tr->Cout,
                                    tr->rs, inv_total};
      fd::train::l1_head4_kernel<<<dim3(strips, parts), 256, 0, r.s>>>(
          tr->F, targets, pg, nullptr, tr->dy16, tr->part_a, tr->loss_part);
      r.check(cudaGetLastError());
      fd::train::finish_loss_kernel<<<1, fd::train::kLossThreads, 0, r.s>>>(
          tr->loss_part, parts * strips, inv_total, loss);
      r.check(cudaGetLastError());
      r.sum_parts({{tr->part_a, parts, tr->Cr, tr->Cr, 0, r.grad(g, eH + 4)}});
      r.end();
    }
  }
  // ---- backward
  // head layer 2
  r.gemm(FD_TK_DGRAD, fd::EPI_F32, MR, D, tr->Cr, tr->dy16, tr->Cr, tr->t_head2, tr->Cr, nullptr, tr->gC, D);
  r.wgrad(tr->dy16, tr->Cr, tr->a1, D, MR, r.grad(g, eH + 3));
  // head layer 1 (GELU')
  r.gelu_bwd(tr->z1, tr->gC, MR, D, tr->dqkv16, r.grad(g, eH + 2));
  r.gemm(FD_TK_DGRAD, fd::EPI_F32, MR, D, D, tr->dqkv16, D, tr->t_head1, D, nullptr, tr->gA, D);
  r.wgrad(tr->dqkv16, D, tr->yh16, D, MR, r.grad(g, eH + 1));
  // the gradient of a block's second MLP bias: the column sums of the block's output gradient
  auto mlp_bias = [&](size_t e0, int b) {
    return r.grad(g, e0 + static_cast<size_t>(b) * kBlockEntries + kM2B);
  };
  // the head's RMSNorm
  r.rmsnorm_bwd(hRo, r.wf(eH), tr->gA, nullptr, MR, tr->gB, tr->dy16, r.grad(g, eH),
                tr->nr > 0 ? mlp_bias(eR, tr->nr - 1) : nullptr);
  for (int b = tr->nr - 1; b >= 0; --b)
    block_bwd(r, tr->sR, b, eR + static_cast<size_t>(b) * kBlockEntries, tr->tR[b], g,
              b > 0 ? mlp_bias(eR, b - 1) : nullptr);
  // temporal upsampling: refined frame tau back to channel block tau
  {
    const int parts = (MB + kRowBlock - 1) / kRowBlock, cols = rt * D;
    if (r.room(parts, cols) && r.begin(FD_TK_POINTWISE)) {
      fd::train::tup_bwd_kernel<<<dim3((cols + 1023) / 1024, parts), 256, 0, r.s>>>(
          tr->gB, MB, rt, tr->Lp, D, tr->dqkv16, tr->part_a);
      r.check(cudaGetLastError());
      r.sum_parts({{tr->part_a, parts, cols, cols, 0, r.grad(g, eF + 2)}});
      r.end();
    }
  }
  r.gemm(FD_TK_DGRAD, fd::EPI_F32, MB, D, rt * D, tr->dqkv16, rt * D, tr->t_tup, rt * D, nullptr, tr->gA, D);
  r.wgrad(tr->dqkv16, rt * D, tr->y16, D, MB, r.grad(g, eF + 1));
  r.rmsnorm_bwd(hBo, r.wf(eF), tr->gA, nullptr, MB, tr->gB, tr->dy16, r.grad(g, eF),
                mlp_bias(eB, tr->nb - 1));
  // the first block's input gradient sums to the patch-embedding's bias gradient
  for (int b = tr->nb - 1; b >= 0; --b)
    block_bwd(r, tr->sB, b, eB + static_cast<size_t>(b) * kBlockEntries, tr->tB[b], g,
              b > 0 ? mlp_bias(eB, b - 1) : r.grad(g, 1));
  // patch-embedding: the weight gradient
  r.wgrad(tr->dy16, D, tr->x0, tr->cin, MB, r.grad(g, 0));
  return r.ok ? FD_OK : FD_ERR_CUDA;
}

// ---- single kernels of the step, for per-kernel checks (include/flashdec_ops.h)
fd_status fd_op_scores_bwd(int M, int N, const void* Q, const void* dO, const void* K,
                           const void* V, const float* lse, const float* delta, int Pc, int Lp,
                           int L, void* dS, void* dST, void* PT, int* err_dev, void* stream) {
  if (!Q || !dO || !K || !V || !lse || !delta || !dS || !dST || !PT || !err_dev || M < 1 ||
      N < 32 || N % 32 || Lp < 1 || Pc < Lp || Pc % Lp || L < 1 || L > Lp)
    return FD_ERR_INVALID_ARG;
  const void* const ptrs[7] = {Q, dO, K, V, dS, dST, PT};
  for (const void* ptr : ptrs)
    if (reinterpret_cast<uintptr_t>(ptr) & 15u) return FD_ERR_INVALID_ARG;
  const fd::DsEpi ds{lse, delta, 0.125f, Pc, Lp, L, static_cast<bf16*>(dS),
                     static_cast<bf16*>(dST), static_cast<bf16*>(PT)};
  const cudaError_t e = fd::scores_bwd(M, N, static_cast<const bf16*>(Q),
                                       static_cast<const bf16*>(dO), 64,
                                       static_cast<const bf16*>(K), static_cast<const bf16*>(V),
                                       64, ds, err_dev, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? FD_OK : FD_ERR_CUDA;
}

fd_status fd_op_attention_bwd(int T, int N, int G, int W, int Pc, int Lp, int L, int hs,
                              const void* q, const void* dO, const void* k, const void* v,
                              const float* lse, const float* delta, float* dq, float* dk, float* dv,
                              int* err_dev, void* stream) {
  if (!err_dev || T < 1 || N < 1 || G < 1 || N % G || W < 1 || Lp < 128 || Lp % 128 || Pc < Lp ||
      Pc % Lp || L < 1 || L > Lp || hs < 1 || N / G % hs)
    return FD_ERR_INVALID_ARG;
  if (static_cast<long long>(T) * Pc > (1LL << 30) / N) return FD_ERR_INVALID_ARG;  // int rows
  const void* const ptrs[9] = {q, dO, k, v, lse, delta, dq, dk, dv};
  for (const void* ptr : ptrs)
    if (!ptr || reinterpret_cast<uintptr_t>(ptr) & 15u) return FD_ERR_INVALID_ARG;
  const fd::AttnBwdParams p{lse, delta, nullptr, nullptr, T, N, G, W, Pc, Lp, L, T * Pc, hs, err_dev};
  const cudaError_t e = fd::attention_bwd(
      static_cast<const bf16*>(q), static_cast<const bf16*>(dO), static_cast<const bf16*>(k),
      static_cast<const bf16*>(v), p, dq, dk, dv, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? FD_OK : FD_ERR_CUDA;
}

fd_status fd_op_rmsnorm_bwd(const float* x, const float* g, const float* dy, int M, int D,
                            float eps, float* dx, float* dg, float* work, void* stream) {
  if (!x || !g || !dy || !dx || !dg || !work || M < 1 || D < 1 || D > 65536)
    return FD_ERR_INVALID_ARG;
  using namespace fd::train;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // partial rows of dg in the caller's scratch (at most M of them)
  const int blocks = (M + kNormRows - 1) / kNormRows;
  int groups = norm_groups(D);
  if (blocks * groups > M) groups = 1;
  const bool vec = D % 4 == 0 && ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(dy) |
                                   reinterpret_cast<uintptr_t>(dx)) & 15u) == 0;
  if (vec)
    rmsnorm_bwd_kernel<4><<<blocks, 256, 0, s>>>(x, g, dy, nullptr, M, D, eps, groups, dx, nullptr,
                                                work, nullptr);
  else
    rmsnorm_bwd_kernel<1><<<blocks, 256, 0, s>>>(x, g, dy, nullptr, M, D, eps, groups, dx, nullptr,
                                                work, nullptr);
  if (cudaGetLastError() != cudaSuccess) return FD_ERR_CUDA;
  SumJobs js{};
  js.job[0] = {work, blocks * groups, D, D, 0, dg};
  sum_parts_kernel<<<dim3((D + 31) / 32, 1), dim3(32, kSumRows), 0, s>>>(js);
  return cudaGetLastError() == cudaSuccess ? FD_OK : FD_ERR_CUDA;
}

fd_status fd_op_gelu_bwd(const float* z, const float* da, int64_t n, float* dz, void* dz_bf16,
                         void* stream) {
  if (!z || !da || !dz || !dz_bf16 || n < 1) return FD_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  bf16* const dz16 = static_cast<bf16*>(dz_bf16);
  const bool vec =
      n % 4 == 0 && ((reinterpret_cast<uintptr_t>(z) | reinterpret_cast<uintptr_t>(da) |
                      reinterpret_cast<uintptr_t>(dz)) & 15u) == 0 &&
      (reinterpret_cast<uintptr_t>(dz16) & 7u) == 0;
  if (vec)
    fd::train::gelu_bwd_kernel<4><<<blocks_for(n / 4, 256), 256, 0, s>>>(z, da, n, dz, dz16);
  else
    fd::train::gelu_bwd_kernel<1><<<blocks_for(n, 256), 256, 0, s>>>(z, da, n, dz, dz16);
  return cudaGetLastError() == cudaSuccess ? FD_OK : FD_ERR_CUDA;
}

fd_status fd_op_l1_pixel_bwd(const float* F, const float* target, int frames, int grid_h,
                             int grid_w, int channels, int rs, float* dF, float* loss,
                             float* work, void* stream) {
  if (!F || !target || !dF || !loss || !work || frames < 1 || grid_h < 1 || grid_w < 1 ||
      channels < 1 || rs < 1)
    return FD_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int L = grid_h * grid_w;
  const long long n = static_cast<long long>(frames) * L * channels * rs * rs;
  const int blocks = static_cast<int>((n + 255) / 256);
  const float inv_total = static_cast<float>(1.0 / static_cast<double>(n));
  // one chunk of `frames` refined frames, rows unpadded (Lp = L)
  const fd::train::PixelGrid pg{1, frames, frames, L, L, grid_h, grid_w, channels, rs, inv_total};
  const int cols = channels * rs * rs;
  const bool vec = rs % 4 == 0 && L <= 65535 * fd::train::kRowBlock / frames &&  // grid y
                   ((reinterpret_cast<uintptr_t>(F) | reinterpret_cast<uintptr_t>(target) |
                     reinterpret_cast<uintptr_t>(dF)) & 15u) == 0;
  int parts = blocks;
  if (vec) {  // no more partial sums than the caller's scratch holds: a row has cols >= 16 elements
    const int strips = (cols + 1023) / 1024;
    const int rows = (frames * L + fd::train::kRowBlock - 1) / fd::train::kRowBlock;
    parts = strips * rows;
    fd::train::l1_head4_kernel<<<dim3(strips, rows), 256, 0, s>>>(F, target, pg, dF, nullptr,
                                                                 nullptr, work);
  } else {
    fd::train::l1_head_kernel<<<blocks, 256, 0, s>>>(F, target, pg, dF, work);
  }
  if (cudaGetLastError() != cudaSuccess) return FD_ERR_CUDA;
  fd::train::finish_loss_kernel<<<1, fd::train::kLossThreads, 0, s>>>(work, parts, inv_total, loss);
  return cudaGetLastError() == cudaSuccess ? FD_OK : FD_ERR_CUDA;
}

fd_status fd_train_status(fd_trainer tr, void* stream) {
  if (tr == nullptr) return FD_ERR_INVALID_ARG;
  if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) return FD_ERR_CUDA;
  int e = 0;
  if (cudaMemcpy(&e, tr->err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    return FD_ERR_CUDA;
  return e ? FD_ERR_DEVICE_TIMEOUT : FD_OK;
}

fd_status fd_train_profile_enable(fd_trainer tr, int enable) {
  if (tr == nullptr) return FD_ERR_INVALID_ARG;
  tr->prof = enable != 0;
  return FD_OK;
}

fd_status fd_train_profile_collect(fd_trainer tr, int64_t* launches, double* ms) {
  if (tr == nullptr || launches == nullptr || ms == nullptr) return FD_ERR_INVALID_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return FD_ERR_CUDA;
  fd_status st = FD_OK;
  for (const fd_trainer_s::Rec& e : tr->rec) {
    float t = 0.f;
    if (cudaEventElapsedTime(&t, e.a, e.b) != cudaSuccess) st = FD_ERR_CUDA;
    if (e.kind >= 0 && e.kind < FD_TK_COUNT) {
      launches[e.kind] += 1;
      ms[e.kind] += t;
    }
    tr->ev_free.push_back(e.a);
    tr->ev_free.push_back(e.b);
  }
  tr->rec.clear();
  return st;
}

fd_status fd_train_destroy(fd_trainer tr) {
  if (tr == nullptr) return FD_ERR_INVALID_ARG;
  cudaDeviceSynchronize();
  for (cudaEvent_t e : tr->ev_all) cudaEventDestroy(e);
  for (void* ptr : tr->allocs) cudaFree(ptr);
  fd::weights_add_user(tr->w, -1);
  delete tr;
  return FD_OK;
}

}  // extern "C"
