// Stage 5 — dense in-block attention and the online-softmax merge (Section 4.3, Section 2.2);
// stage 6 — cache maintenance (Section 4.3, Section 2.1) and the page summaries (Section 2.3).
//
// These stages touch O(B * H * d) data: they are latency-bound.  In bf16 mode the in-block attention
// runs on the tensor cores (block_attn_mma_kernel); the fp32 mode and the cache kernels are plain
// CUDA-core code laid out for coalesced global access and conflict-free shared-memory access.
#include "kernels.h"
#include "block_attn_mma.cuh"

namespace losa {
namespace {

constexpr int kThreads = 256;
constexpr int kTokTile = 4;        // block tokens per CTA of the in-block attention
constexpr int kBaThreads = 128;
constexpr int kBaRows = 4;         // query rows a warp works on together

// One CTA per (four block tokens, KV head, sequence): K_b, V_b of the KV head and the CTA's query
// rows staged in shared memory as fp32.  A warp takes four query rows at a time (with G = 4 the
// heads of one token), so every K_b / V_b element read from shared memory feeds four multiply-adds:
// the kernel is bound by shared-memory reads, and this is what keeps it short enough to hide beside
// stages 1-3.  Scores: lane = block key (rows of K_b padded by four floats: conflict-free 16-byte
// reads), the four query rows read as broadcasts; P V: lane = output column, probabilities by shuffle.
// MERGE = false (whole-step path): only the in-block part, normalised o_b to `ob_out` and L_b to
// `lse_out`; the prefix statistics are not touched, so this can run beside stages 1-4.
template <typename T, int D, bool MERGE>
__global__ void __launch_bounds__(kBaThreads)
block_attn_merge_kernel(const T* __restrict__ q, const T* __restrict__ k_blk, const T* __restrict__ v_blk,
                        const float* __restrict__ o_p, const float* __restrict__ lse_p,
                        T* __restrict__ out, float* __restrict__ lse_out, float* __restrict__ ob_out,
                        int B, int Hq, int Hkv, float sm_scale) {
  grid_dep_wait();
  constexpr int KS = D + 4;         // padded row of K_b
  constexpr int C = D / 32;
  constexpr int U = 2;              // block keys per lane (B <= 64)
  extern __shared__ __align__(16) float smem[];
  float* Ks = smem;                 // [B][D + 4]
  float* Vs = Ks + B * KS;          // [B][D]
  float* Qs = Vs + B * D;           // [kTokTile * G][D]
  const int t0 = blockIdx.x * kTokTile, kh = blockIdx.y, s = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = Hq / Hkv;
  const int nrow = min(kTokTile, B - t0) * G;
  auto row_of = [&](int r) { return (static_cast<size_t>(s) * B + t0 + r / G) * Hq + kh * G + r % G; };
  for (int idx = tid * 8; idx < nrow * D; idx += kBaThreads * 8) {
    float a[8];
    load8(q + row_of(idx / D) * D + idx % D, a);
    *reinterpret_cast<float4*>(Qs + idx) = make_float4(a[0], a[1], a[2], a[3]);
    *reinterpret_cast<float4*>(Qs + idx + 4) = make_float4(a[4], a[5], a[6], a[7]);
  }
  for (int idx = tid * 8; idx < B * D; idx += kBaThreads * 8) {
    const int t = idx / D, j = idx % D;
    const size_t src = ((static_cast<size_t>(s) * B + t) * Hkv + kh) * D + j;
    float a[8], b[8];
    load8(k_blk + src, a);
    load8(v_blk + src, b);
    *reinterpret_cast<float4*>(Ks + t * KS + j) = make_float4(a[0], a[1], a[2], a[3]);
    *reinterpret_cast<float4*>(Ks + t * KS + j + 4) = make_float4(a[4], a[5], a[6], a[7]);
    *reinterpret_cast<float4*>(Vs + idx) = make_float4(b[0], b[1], b[2], b[3]);
    *reinterpret_cast<float4*>(Vs + idx + 4) = make_float4(b[4], b[5], b[6], b[7]);
  }
  __syncthreads();
  for (int r0 = warp * kBaRows; r0 < nrow; r0 += (kBaThreads / 32) * kBaRows) {
    const int nr = min(kBaRows, nrow - r0);
    // prefix statistics of the rows (MERGE): requested now, used after the arithmetic
    float opv[kBaRows][C], Lp[kBaRows];
#pragma unroll
    for (int r = 0; r < kBaRows; ++r) {
      const size_t row = row_of(r0 + min(r, nr - 1));
#pragma unroll
      for (int c = 0; c < C; ++c) opv[r][c] = MERGE ? o_p[row * D + lane + 32 * c] : 0.f;
      Lp[r] = MERGE ? lse_p[row] : 0.f;
    }
    // ---- scores: lane = block key (two keys per lane when B > 32)
    float sc[U][kBaRows];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < kBaRows; ++r) sc[u][r] = 0.f;
    const float* qr = Qs + r0 * D;
#pragma unroll 4
    for (int j = 0; j < D; j += 4) {
      float4 kv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int t = lane + 32 * u;
        kv[u] = (t < B) ? *reinterpret_cast<const float4*>(Ks + t * KS + j) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int r = 0; r < kBaRows; ++r) {
        const float4 qv = *reinterpret_cast<const float4*>(qr + min(r, nr - 1) * D + j);
#pragma unroll
        for (int u = 0; u < U; ++u)
          sc[u][r] = fmaf(qv.w, kv[u].w, fmaf(qv.z, kv[u].z, fmaf(qv.y, kv[u].y, fmaf(qv.x, kv[u].x, sc[u][r]))));
      }
    }
    // ---- softmax over the block keys, per row
    float p[U][kBaRows], sum[kBaRows], Lb[kBaRows];
#pragma unroll
    for (int r = 0; r < kBaRows; ++r) {
      float mx = -INFINITY;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        sc[u][r] = (lane + 32 * u < B) ? sc[u][r] * sm_scale : -INFINITY;
        mx = fmaxf(mx, sc[u][r]);
      }
      const float M = warp_max(mx);
      float ps = 0.f;
#pragma unroll
      for (int u = 0; u < U; ++u) { p[u][r] = expf(sc[u][r] - M); ps += p[u][r]; }
      sum[r] = warp_sum(ps);
      Lb[r] = M + logf(sum[r]);
    }
    // ---- P V: lane = output column
    float ob[kBaRows][C];
#pragma unroll
    for (int r = 0; r < kBaRows; ++r)
#pragma unroll
      for (int c = 0; c < C; ++c) ob[r][c] = 0.f;
#pragma unroll 2
    for (int t = 0; t < B; ++t) {
      float v[C];
#pragma unroll
      for (int c = 0; c < C; ++c) v[c] = Vs[t * D + lane + 32 * c];
#pragma unroll
      for (int r = 0; r < kBaRows; ++r) {
        const float pt = __shfl_sync(0xffffffffu, t < 32 ? p[0][r] : p[1][r], t & 31);
#pragma unroll
        for (int c = 0; c < C; ++c) ob[r][c] = fmaf(pt, v[c], ob[r][c]);
      }
    }
#pragma unroll
    for (int r = 0; r < kBaRows; ++r) {
      if (r < nr) {
        const size_t row = row_of(r0 + r);
        if (MERGE) {
          const float M2 = fmaxf(Lp[r], Lb[r]);
          const float L = M2 + logf(expf(Lp[r] - M2) + expf(Lb[r] - M2));
          const float wp = expf(Lp[r] - L), wb = expf(Lb[r] - L) / sum[r];
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const float v = (wp > 0.f ? wp * opv[r][c] : 0.f) + wb * ob[r][c];
            out[row * D + lane + 32 * c] = from_f32<T>(v);
          }
          if (lse_out && lane == 0) lse_out[row] = L;
        } else {
          const float inv = 1.f / sum[r];
#pragma unroll
          for (int c = 0; c < C; ++c) ob_out[row * D + lane + 32 * c] = ob[r][c] * inv;
          if (lane == 0) lse_out[row] = Lb[r];
        }
      }
    }
  }
}

// Stage 5 of the six-call path, bf16 (MERGE), and the in-block part of a whole step whose selection does
// not carry it.
template <int D, int BK, bool MERGE>
__global__ void __launch_bounds__(kMmaThreads) block_attn_mma_kernel(BlockAttnParams p) {
  grid_dep_wait();
  __shared__ __align__(16) BlockAttnSmem<D, BK> sm;
  block_attn_mma_cta<D, BK, MERGE, D>(p, sm, blockIdx.x, blockIdx.y, blockIdx.z);
}

template <typename T>
__global__ void __launch_bounds__(kThreads)
commit_step_kernel(const uint4* __restrict__ q, uint4* __restrict__ q_prev, size_t n_vec,
                   int32_t* __restrict__ step, int N) {
  grid_dep_wait();
  for (size_t i = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x; i < n_vec;
       i += static_cast<size_t>(gridDim.x) * kThreads)
    q_prev[i] = q[i];
  if (blockIdx.x == 0)
    for (int s = threadIdx.x; s < N; s += kThreads) step[s] += 1;
}

// min / max of column j of logical page p over its valid tokens; tokens at prefix positions >=
// new_from are taken from the block being appended (k_blk) instead of the pool.
template <typename T>
__device__ __forceinline__ void summarise_column(const T* __restrict__ k_pages, const T* __restrict__ k_blk,
                                                 T* __restrict__ kmin, T* __restrict__ kmax,
                                                 size_t page_off, int64_t stride_tok, int valid,
                                                 int page_start, int new_from, size_t blk_off,
                                                 int blk_stride, size_t sum_off, int j) {
  float lo = INFINITY, hi = -INFINITY;
  for (int t = 0; t < valid; ++t) {
    const int pos = page_start + t;
    const float v = (pos >= new_from)
                        ? to_f32(k_blk[blk_off + static_cast<size_t>(pos - new_from) * blk_stride + j])
                        : to_f32(k_pages[page_off + static_cast<size_t>(t) * stride_tok + j]);
    lo = fminf(lo, v);
    hi = fmaxf(hi, v);
  }
  kmin[sum_off + j] = from_f32<T>(lo);
  kmax[sum_off + j] = from_f32<T>(hi);
}

// One warp per (logical page, KV head, sequence).  One pass over the keys, so HBM bounds it: a lane
// takes 16 bytes of a row per load with up to 16 loads in flight, the warps of a CTA take
// neighbouring heads of a page (neighbours in the pool).  184 MB of bf16 keys: 54 us with a thread
// per column (two bytes a load), 40 us now.
constexpr int kSumWarps = 8;

template <typename T, int D>
__global__ void __launch_bounds__(kSumWarps * 32)
build_summaries_kernel(const T* __restrict__ k_pages, T* __restrict__ kmin,
                       T* __restrict__ kmax, const int32_t* __restrict__ page_table,
                       const int32_t* __restrict__ kv_len, int64_t stride_page,
                       int64_t stride_head, int64_t stride_tok, int Hkv, int g,
                       int Pmax, int n_phys, int32_t* __restrict__ status) {
  constexpr int V = 16 / sizeof(T), LPR = D / V, RPI = 32 / LPR, U = 16;   // elements per load, lanes per row, rows per load, loads in flight
  grid_dep_wait();
  const int lane = threadIdx.x & 31, w = blockIdx.x * kSumWarps + (threadIdx.x >> 5);
  const int kh = w % Hkv, p = w / Hkv, s = blockIdx.z;
  if (p >= Pmax) return;
  const int len = kv_len[s], phys = page_table[static_cast<size_t>(s) * Pmax + p];   // (a table entry past the prefix is not used)
  const int valid = min(g, len - p * g);
  if (valid <= 0) return;
  if (phys < 0 || phys >= n_phys) { if (lane == 0) set_status(status, LOSA_ERR_BOUNDS); return; }
  const int t0 = lane / LPR, j = (lane % LPR) * V;
  const T* src = k_pages + static_cast<size_t>(phys) * stride_page + static_cast<size_t>(kh) * stride_head + j;
  float lo[V], hi[V];
#pragma unroll
  for (int x = 0; x < V; ++x) { lo[x] = INFINITY; hi[x] = -INFINITY; }
  for (int base = 0; base < valid; base += U * RPI) {
    uint4 raw[U];
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int t = base + t0 + i * RPI;
      if (t < valid) raw[i] = __ldcs(reinterpret_cast<const uint4*>(src + static_cast<size_t>(t) * stride_tok));
    }
#pragma unroll
    for (int i = 0; i < U; ++i) {
      if (base + t0 + i * RPI < valid) {
        const T* e = reinterpret_cast<const T*>(&raw[i]);
#pragma unroll
        for (int x = 0; x < V; ++x) { lo[x] = fminf(lo[x], to_f32(e[x])); hi[x] = fmaxf(hi[x], to_f32(e[x])); }
      }
    }
  }
#pragma unroll
  for (int o = LPR; o < 32; o <<= 1)
#pragma unroll
    for (int x = 0; x < V; ++x) {
      lo[x] = fminf(lo[x], __shfl_xor_sync(0xffffffffu, lo[x], o));
      hi[x] = fmaxf(hi[x], __shfl_xor_sync(0xffffffffu, hi[x], o));
    }
  if (t0 == 0) {
    alignas(16) T a[V], b[V];
#pragma unroll
    for (int x = 0; x < V; ++x) { a[x] = from_f32<T>(lo[x]); b[x] = from_f32<T>(hi[x]); }
    const size_t at = (static_cast<size_t>(phys) * Hkv + kh) * D + j;
    *reinterpret_cast<uint4*>(kmin + at) = *reinterpret_cast<const uint4*>(a);
    *reinterpret_cast<uint4*>(kmax + at) = *reinterpret_cast<const uint4*>(b);
  }
}

// Block finalisation: one CTA per (touched page, KV head, sequence) writes the block tokens that
// fall into the page and recomputes the page's summaries; kv_len / step are bumped by a second
// kernel so that every CTA here sees the old length.
template <typename T>
__global__ void append_block_kernel(T* __restrict__ k_pages, T* __restrict__ v_pages, T* __restrict__ kmin,
                                    T* __restrict__ kmax, const T* __restrict__ k_blk,
                                    const T* __restrict__ v_blk, const int32_t* __restrict__ page_table,
                                    const int32_t* __restrict__ kv_len, int64_t stride_page,
                                    int64_t stride_head, int64_t stride_tok, int B, int Hkv, int D,
                                    int g, int Pmax, int n_phys, int32_t* __restrict__ status) {
  grid_dep_wait();
  const int kh = blockIdx.y, s = blockIdx.z, j = threadIdx.x;
  const int L0 = kv_len[s];
  const int p = L0 / g + blockIdx.x;
  if (p > (L0 + B - 1) / g) return;
  if (p >= Pmax) { set_status(status, LOSA_ERR_BOUNDS); return; }
  const int phys = page_table[static_cast<size_t>(s) * Pmax + p];
  if (phys < 0 || phys >= n_phys) { set_status(status, LOSA_ERR_BOUNDS); return; }
  const size_t page_off = static_cast<size_t>(phys) * stride_page + static_cast<size_t>(kh) * stride_head;
  const size_t blk_off = (static_cast<size_t>(s) * B * Hkv + kh) * D;
  const int blk_stride = Hkv * D;
  const int first = max(L0, p * g), last = min(L0 + B, p * g + g);   // prefix positions written here
  for (int pos = first; pos < last; ++pos) {
    const size_t dst = page_off + static_cast<size_t>(pos - p * g) * stride_tok + j;
    const size_t src = blk_off + static_cast<size_t>(pos - L0) * blk_stride + j;
    k_pages[dst] = k_blk[src];
    v_pages[dst] = v_blk[src];
  }
  summarise_column<T>(k_pages, k_blk, kmin, kmax, page_off, stride_tok, last - p * g, p * g, L0,
                      blk_off, blk_stride, (static_cast<size_t>(phys) * Hkv + kh) * D, j);
}

// A sequence whose block did not fit its page-table row (the append kernel reported it and wrote
// nothing beyond the row) keeps its length: later steps must not index pages past P_max.
__global__ void finalize_counters_kernel(int32_t* __restrict__ kv_len, int32_t* __restrict__ step, int N, int B,
                                         int g, int Pmax) {
  grid_dep_wait();
  const int s = threadIdx.x;
  if (s < N) {
    const long long cap = static_cast<long long>(Pmax) * g;
    if (static_cast<long long>(kv_len[s]) + B <= cap) kv_len[s] += B;
    step[s] = 0;
  }
}

template <typename T, int D, bool MERGE>
int32_t launch_merge_t(losa_ctx* c, const void* q, const void* k_blk, const void* v_blk,
                       const losa_state_t* state, void* out, float* lse_out, float* ob_out, cudaStream_t st) {
  const losa_shape_t& sh = c->shape;
  const int G = sh.n_q_heads / sh.n_kv_heads;
  const size_t smem = (static_cast<size_t>(sh.block_size) * (2 * D + 4) + static_cast<size_t>(kTokTile) * G * D) * sizeof(float);
  constexpr int most = (LOSA_MAX_BLOCK * (2 * D + 4) + kTokTile * 16 * D) * static_cast<int>(sizeof(float));   // (16 heads per KV head)
  if (smem > 48 * 1024)               // (the most that any context asks for: the attribute is shared by all of them)
    LOSA_CUDA_TRY(c, cudaFuncSetAttribute(block_attn_merge_kernel<T, D, MERGE>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
  dim3 grid((sh.block_size + kTokTile - 1) / kTokTile, sh.n_kv_heads, sh.batch);
  launch_k(block_attn_merge_kernel<T, D, MERGE>, grid, kBaThreads, smem, st, 
      static_cast<const T*>(q), static_cast<const T*>(k_blk), static_cast<const T*>(v_blk),
      state ? static_cast<const float*>(state->o_p) : nullptr, state ? state->lse_p : nullptr, static_cast<T*>(out), lse_out, ob_out,
      sh.block_size, sh.n_q_heads, sh.n_kv_heads, sh.sm_scale);
  return after_launch(c);
}

template <typename T>
int32_t launch_update_t(losa_ctx* c, losa_kv_t* kv, losa_state_t* state, const void* q,
                        const void* k_blk, const void* v_blk, int32_t finalize_block, cudaStream_t st) {
  const losa_shape_t& sh = c->shape;
  if (!finalize_block) {
    const size_t n_vec = static_cast<size_t>(sh.batch) * sh.block_size * sh.n_q_heads * sh.head_dim * sizeof(T) / 16;
    const int blocks = static_cast<int>(std::min<size_t>((n_vec + kThreads - 1) / kThreads, static_cast<size_t>(c->n_sms) * 4));
    launch_k(commit_step_kernel<T>, std::max(blocks, 1), kThreads, 0, st, 
        static_cast<const uint4*>(q), static_cast<uint4*>(state->q_prev), n_vec, state->step, sh.batch);
    return after_launch(c);
  }
  if (kv->kv_format == LOSA_KV_FP8_E4M3) {
    // FP8 pages: the touched pages are re-quantised from their dequantised old rows and the new rows
    int32_t rc = launch_fp8_append(c, kv, k_blk, v_blk, st);
    if (rc != LOSA_OK) return rc;
    launch_k(finalize_counters_kernel, 1, std::max(32, sh.batch), 0, st, kv->kv_len, state->step, sh.batch, sh.block_size,
             sh.page_size, sh.max_pages_per_seq);
    return after_launch(c);
  }
  dim3 grid((sh.block_size + sh.page_size - 1) / sh.page_size + 1, sh.n_kv_heads, sh.batch);
  // (the driver's split leaves its loads in flight more L1 than the steps' split: an append between two steps of one
  // sequence with pages of 64 costs 7.8 us, else 9.7)
  launch_split(cudaSharedmemCarveoutDefault, append_block_kernel<T>, grid, sh.head_dim, 0, st, 
      static_cast<T*>(kv->k_pages), static_cast<T*>(kv->v_pages), static_cast<T*>(kv->kmin),
      static_cast<T*>(kv->kmax), static_cast<const T*>(k_blk), static_cast<const T*>(v_blk),
      kv->page_table, kv->kv_len, kv->stride_page, kv->stride_head, kv->stride_tok, sh.block_size,
      sh.n_kv_heads, sh.head_dim, sh.page_size, sh.max_pages_per_seq, kv->n_phys_pages, status_ptr(c));
  int32_t rc = after_launch(c);
  if (rc != LOSA_OK) return rc;
  launch_k(finalize_counters_kernel, 1, std::max(32, sh.batch), 0, st, kv->kv_len, state->step, sh.batch, sh.block_size,
           sh.page_size, sh.max_pages_per_seq);
  return after_launch(c);
}

template <typename T, int D>
int32_t launch_summaries_t(losa_ctx* c, losa_kv_t* kv, cudaStream_t st) {
  const losa_shape_t& sh = c->shape;
  if (sh.max_pages_per_seq == 0) return LOSA_OK;
  const dim3 grid((sh.max_pages_per_seq * sh.n_kv_heads + kSumWarps - 1) / kSumWarps, 1, sh.batch);
  launch_streaming(build_summaries_kernel<T, D>, grid, kSumWarps * 32, 0, st, 
      static_cast<const T*>(kv->k_pages), static_cast<T*>(kv->kmin), static_cast<T*>(kv->kmax),
      kv->page_table, kv->kv_len, kv->stride_page, kv->stride_head, kv->stride_tok, sh.n_kv_heads,
      sh.page_size, sh.max_pages_per_seq, kv->n_phys_pages, status_ptr(c));
  return after_launch(c);
}

}  // namespace

int32_t launch_block_attn_merge(losa_ctx* c, const void* q, const void* k_blk, const void* v_blk,
                                const losa_state_t* state, void* out, float* lse_out_opt, cudaStream_t st) {
  const bool bf = c->shape.dtype == LOSA_BF16;
  if (bf) {
    const losa_shape_t& sh = c->shape;
    BlockAttnParams p = block_attn_params(c, q, k_blk, v_blk);
    p.o_p = state->o_p;
    p.o_p_bf16 = state->o_p_format == LOSA_STATE_BF16 ? 1 : 0;
    p.lse_p = state->lse_p;
    p.out = static_cast<__nv_bfloat16*>(out);
    p.lse_out = lse_out_opt;
    const dim3 grid(block_attn_tiles(sh), sh.n_kv_heads, sh.batch);
    with_block_attn_shape(sh, [&](auto d, auto bk) {
      launch_k(block_attn_mma_kernel<decltype(d)::value, decltype(bk)::value, true>, grid, kMmaThreads, 0, st, p);
    });
    return after_launch(c);
  }
  if (c->shape.head_dim == 128) return launch_merge_t<float, 128, true>(c, q, k_blk, v_blk, state, out, lse_out_opt, nullptr, st);
  return launch_merge_t<float, 64, true>(c, q, k_blk, v_blk, state, out, lse_out_opt, nullptr, st);
}

int32_t launch_block_attn(losa_ctx* c, const void* q, const void* k_blk, const void* v_blk, cudaStream_t st) {
  float* ob = reinterpret_cast<float*>(c->ws + c->lay.block_o);
  float* lb = reinterpret_cast<float*>(c->ws + c->lay.block_lse);
  if (c->shape.dtype == LOSA_BF16) {
    const BlockAttnParams p = block_attn_params(c, q, k_blk, v_blk);
    const dim3 grid(block_attn_tiles(c->shape), c->shape.n_kv_heads, c->shape.batch);
    with_block_attn_shape(c->shape, [&](auto d, auto bk) {
      launch_k(block_attn_mma_kernel<decltype(d)::value, decltype(bk)::value, false>, grid, kMmaThreads, 0, st, p);
    });
    return after_launch(c);
  }
  if (c->shape.head_dim == 128) return launch_merge_t<float, 128, false>(c, q, k_blk, v_blk, nullptr, nullptr, lb, ob, st);
  return launch_merge_t<float, 64, false>(c, q, k_blk, v_blk, nullptr, nullptr, lb, ob, st);
}

int32_t launch_update_prefix_cache(losa_ctx* c, losa_kv_t* kv, losa_state_t* state, const void* q,
                                   const void* k_blk, const void* v_blk, int32_t finalize_block, cudaStream_t st) {
  return c->shape.dtype == LOSA_BF16
             ? launch_update_t<__nv_bfloat16>(c, kv, state, q, k_blk, v_blk, finalize_block, st)
             : launch_update_t<float>(c, kv, state, q, k_blk, v_blk, finalize_block, st);
}

int32_t launch_build_page_summaries(losa_ctx* c, losa_kv_t* kv, cudaStream_t st) {
  if (kv->kv_format == LOSA_KV_FP8_E4M3) return launch_fp8_summaries(c, kv, st);
  if (c->shape.dtype == LOSA_BF16)
    return c->shape.head_dim == 128 ? launch_summaries_t<__nv_bfloat16, 128>(c, kv, st) : launch_summaries_t<__nv_bfloat16, 64>(c, kv, st);
  return c->shape.head_dim == 128 ? launch_summaries_t<float, 128>(c, kv, st) : launch_summaries_t<float, 64>(c, kv, st);
}

}  // namespace losa
