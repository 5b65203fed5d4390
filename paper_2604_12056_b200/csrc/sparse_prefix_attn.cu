// Stage 4 — paged sparse prefix attention for the active tokens (Section 2.2, Section 4.2).
//
// Work decomposition (both element types).  The pages to read form a flat list of items
// (segment = (sequence, KV head, row group), position in that segment's union list).  The list is
// cut into one contiguous, equally long range per CTA (one CTA per SM), so ragged unions never
// leave an SM idle.  A CTA produces, for every segment its range touches, an un-normalised partial
// (row max, row sum, sum p*v) in the workspace; a small combine kernel merges the partials of a
// segment by log-sum-exp — the same merge Section 2.2 uses between prefix and block — and writes
// (o_p, L_p) of the ACTIVE tokens only, which is what keeps the reuse rule exact for the others.
//
// bf16 kernel (sparse_prefix_attn_tc5.cuh): TMA streams the pages of K and V into rings of shared
//   memory; Q K^T and P V run on the tcgen05 tensor cores with S, P and O in tensor memory; the
//   softmax warps own one query row per thread.  Query rows are the GQA-grouped (active token,
//   head) pairs of the KV head, up to 128 per row group.
// fp32 kernel: CUDA cores, fp32 FMA (bf16 tensor cores cannot meet the 1e-5 fp32 tolerance).
//
// Every wait on an mbarrier is bounded; when a bound runs out the CTA records LOSA_ERR_TIMEOUT,
// raises its abort flag (which ends every other wait of the CTA) and leaves through the common exit.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <type_traits>

#include "kernels.h"

namespace losa {
namespace {

struct AttnParams {
  const void* q;
  const void* k_pages;
  const void* v_pages;
  int64_t stride_page, stride_head, stride_tok;
  const int32_t* page_table;
  const int32_t* kv_len;
  const int32_t* active_idx;
  const int32_t* n_active;
  const int32_t* union_pages;
  const int32_t* union_count;
  const uint32_t* union_bits;   // whole step: the lists as page bitmaps [n_sk][W], to be written to ...
  int32_t* union_pages_out;     // ... these (fp32 kernel); null: the lists are in union_pages / union_count
  int32_t* union_count_out;
  int W;
  float* partials;
  int2* seg_records;    // per segment: first CTA and number of its partial records (written by the main kernels)
  void* o_p;                // cached prefix output, fp32 or bf16 (o_p_bf16)
  int o_p_bf16;
  float* lse_p;
  int32_t* status;
  const float* k_scale;   // FP8 pages: [n_phys, H_kv] power-of-two scales (else null)
  const float* v_scale;
  int N, B, Hq, Hkv, G, Pmax, n_phys, n_rg, n_sk, n_seg, n_ctas;   // n_sk = N * Hkv, n_seg = n_rg * n_sk
  float sm_scale;
  int early;              // the kernels before this one are stages 1 to 3 of the same step: what is older may be read before they end
  long long wait_cycles;  // bound of every mbarrier wait of the bf16 main kernel, in SM clock cycles
};


// Partial results.  A slot (CTA b, segment seg -> b + seg) holds eight records, record t for the
// rows 16t .. 16t+15 of the row group: m[16], l[16], o[16][D] (un-normalised, relative to m).
constexpr int kTileRows = 16;
__device__ __forceinline__ float* record_base(float* partials, int slot, int w, int D) {
  return partials + (static_cast<size_t>(slot) * 8 + w) * kTileRows * (D + 2);
}

__device__ __forceinline__ int clamp_active(int na, int B) { return na < 0 ? 0 : (na > B ? B : na); }

// Whole step: the lists as page bitmaps [n_sk][W] (written by the selection) in shared memory, with the number of
// set bits of the list before every word, so that a page is found by its position in the list.  (16 bits hold it: a context
// has at most topk_max_sortable() pages per sequence, 16,384, or is refused.)
struct UnionBits {
  uint32_t* bits;
  uint16_t* before;
  int W;
  // all lists, by the warps of the CTA (the caller synchronises)
  __device__ __forceinline__ void load(const uint32_t* __restrict__ src, int n_sk, int warp, int n_warps, int lane) const {
    for (int sk = warp; sk < n_sk; sk += n_warps) {
      int run = 0;
      for (int w0 = 0; w0 < W; w0 += 32) {
        const int w = w0 + lane;
        const uint32_t v = w < W ? src[sk * W + w] : 0u;
        const int c = __popc(v);
        int inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += t;
        }
        if (w < W) {
          bits[sk * W + w] = v;
          before[sk * W + w] = static_cast<uint16_t>(run + inc - c);
        }
        run += __shfl_sync(0xffffffffu, inc, 31);
      }
    }
  }
  __device__ __forceinline__ int count(int sk) const {
    const int e = (sk + 1) * W - 1;
    return before[e] + __popc(bits[e]);
  }
  __device__ __forceinline__ int page(int sk, int u) const {     // entry u of list sk: its word, then the bit in the word
    const uint16_t* first = before + sk * W;
    int a = 0, b = W;                               // first[a] <= u (< first[b])
    while (b - a > 1) {
      const int m = (a + b) >> 1;
      if (first[m] <= u) a = m; else b = m;
    }
    uint32_t v = bits[sk * W + a];
    int n = u - first[a], at = 0;                   // the bit with n set bits below it
#pragma unroll
    for (int half = 16; half > 0; half >>= 1) {
      const int c = __popc(v & ((1u << half) - 1u));
      if (n >= c) { n -= c; at += half; v >>= half; }
    }
    return a * 32 + at;
  }
  // stage 3's output for the lists of this CTA, by one warp
  __device__ __forceinline__ void write(const AttnParams& p, int lane) const {
    for (int sk = blockIdx.x; sk < p.n_sk; sk += gridDim.x) {
      int32_t* out = p.union_pages_out + static_cast<size_t>(sk) * p.Pmax;
      for (int w = lane; w < W; w += 32) {
        uint32_t v = bits[sk * W + w];
        int pos = before[sk * W + w];
        while (v) {
          out[pos++] = w * 32 + __ffs(v) - 1;
          v &= v - 1;
        }
      }
      const int n = count(sk);
      for (int t = n + lane; t < p.Pmax; t += 32) out[t] = -1;
      if (lane == 0) p.union_count_out[sk] = n;
    }
  }
};

// C (2 or 4) consecutive elements as one vector access; a lane of the row-wise kernels below owns
// columns lane * C .. lane * C + C - 1 of a row of D = 32 C elements.
template <int C> __device__ __forceinline__ void ldv(const float* p, float (&v)[C]) {
  if constexpr (C == 4) { const float4 t = *reinterpret_cast<const float4*>(p); v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w; }
  else { const float2 t = *reinterpret_cast<const float2*>(p); v[0] = t.x; v[1] = t.y; }
}
template <int C> __device__ __forceinline__ void stv(float* p, const float (&v)[C]) {
  if constexpr (C == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  else *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
}
template <int C> struct RawRow;                      // C elements of the I/O type, moved as they are
template <> struct RawRow<4> { uint2 bits; };
template <> struct RawRow<2> { uint32_t bits; };
template <int C> __device__ __forceinline__ RawRow<C> ld_raw(const __nv_bfloat16* p) { return *reinterpret_cast<const RawRow<C>*>(p); }
template <int C> __device__ __forceinline__ void st_raw(__nv_bfloat16* p, const RawRow<C>& r) { *reinterpret_cast<RawRow<C>*>(p) = r; }
template <int C> __device__ __forceinline__ void st_bf16(__nv_bfloat16* p, const float (&v)[C]) {
  RawRow<C> r;
  if constexpr (C == 4) {
    __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    r.bits = make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
  } else {
    __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]);
    r.bits = *reinterpret_cast<uint32_t*>(&a);
  }
  st_raw<C>(p, r);
}

// C elements of the cached prefix output (fp32 or bf16 storage) at element offset i
template <int C> __device__ __forceinline__ void ld_state(const void* base, int bf16, size_t i, float (&v)[C]) {
  if (bf16) {
    const RawRow<C> r = ld_raw<C>(static_cast<const __nv_bfloat16*>(base) + i);
    if constexpr (C == 4) {
      v[0] = __uint_as_float(r.bits.x << 16); v[1] = __uint_as_float(r.bits.x & 0xffff0000u);
      v[2] = __uint_as_float(r.bits.y << 16); v[3] = __uint_as_float(r.bits.y & 0xffff0000u);
    } else {
      v[0] = __uint_as_float(r.bits << 16); v[1] = __uint_as_float(r.bits & 0xffff0000u);
    }
  } else {
    ldv<C>(static_cast<const float*>(base) + i, v);
  }
}
// ... stored; with bf16 storage v comes back holding the stored (rounded) values, which is what every
// later use must see
template <int C> __device__ __forceinline__ void st_state(void* base, int bf16, size_t i, float (&v)[C]) {
  if (bf16) {
#pragma unroll
    for (int c = 0; c < C; ++c) v[c] = __bfloat162float(__float2bfloat16_rn(v[c]));
    st_bf16<C>(static_cast<__nv_bfloat16*>(base) + i, v);
  } else {
    stv<C>(static_cast<float*>(base) + i, v);
  }
}

#include "sparse_prefix_attn_f32.cuh"

// ===================================================================== combine kernel
// grid (n_seg, kCombineTiles): warp = one query row of the segment's row group at a time.  The CTAs whose
// item range meets the segment are consecutive; each of them left one record for the row's 16-row tile.
// The merge is a chain of dependent reads: latency bounds it.  LOG2: partial maxima in base-2 units
// (tensor-core kernel) or natural units (fp32 kernel).
// Merge of the partial records of row r of segment sg by one warp: returns the un-normalised output
// columns lane * C + c in acc, the reference maximum M and the sum of weights Lsum.  The outputs of up
// to kMergeBatch records are copied to `buf` (that many rows of D floats of this warp) while their
// maxima are read; with up to 40 KB per CTA and few registers, five CTAs are resident per SM, more than with
// outputs in registers, and the rolled loops keep the code short.  A lane reads back only what it
// copied itself.  20: a list cut over 148 CTAs leaves each of
// eight segments 19 or 20 records, one round trip instead of two with 16 (eight steps of one 8K sequence 293 us against 298); more segments have
// fewer records each, and five resident CTAs instead of six cost them nothing (four steps of eight 32K sequences 436 and 435 us).
constexpr int kMergeBatch = 20;
template <int D, bool LOG2>
__device__ __forceinline__ void merge_records(const AttnParams& p, float* buf, int sg, int r, int2 records, int lane,
                                              float (&acc)[D / 32], float& M, float& Lsum) {
  constexpr int C = D / 32;
  constexpr size_t kSlot = static_cast<size_t>(8) * kTileRows * (D + 2);     // consecutive CTAs, consecutive slots
  const int rr = r % kTileRows;
#pragma unroll
  for (int c = 0; c < C; ++c) acc[c] = 0.f;
  M = -INFINITY;
  Lsum = 0.f;
  const uint32_t dst = smem_u32(buf + lane * C);
  for (int base = 0; base < records.y; base += kMergeBatch) {
    const int n = min(kMergeBatch, records.y - base);
    const float* rec = record_base(p.partials, records.x + base + sg, r / kTileRows, D);
    const float mj = lane < n ? rec[lane * kSlot + rr] : -INFINITY, lj = lane < n ? rec[lane * kSlot + kTileRows + rr] : 0.f;
    const float* src = rec + 2 * kTileRows + rr * D + lane * C;
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      if constexpr (C == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i * D * 4), "l"(src + i * kSlot) : "memory");
      else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst + i * D * 4), "l"(src + i * kSlot) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float M_new = fmaxf(M, warp_max(mj));
    const float keep = (M == -INFINITY) ? 0.f : (LOG2 ? exp2f(M - M_new) : expf(M - M_new));
    const float wj = (mj == -INFINITY) ? 0.f : (LOG2 ? exp2f(mj - M_new) : expf(mj - M_new));
    M = M_new;
    Lsum = Lsum * keep + warp_sum(lj * wj);
#pragma unroll
    for (int c = 0; c < C; ++c) acc[c] *= keep;
    cp_async_wait<0>();
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      const float w = __shfl_sync(0xffffffffu, wj, i);
      float v[C];
      ldv<C>(buf + i * D + lane * C, v);
      if (w != 0.f) {
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c] = fmaf(v[c], w, acc[c]);
      }
    }
  }
}

constexpr int kCombineThreads = 128, kCombineTiles = 16;

template <int D, bool LOG2>
__global__ void __launch_bounds__(kCombineThreads) attn_combine_kernel(AttnParams p) {
  grid_dep_wait();
  __shared__ __align__(16) float buf[kCombineThreads / 32][kMergeBatch * D];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sg = blockIdx.x;
  const int rg = sg / p.n_sk, sk = sg % p.n_sk, s = sk / p.Hkv, kh = sk % p.Hkv;
  const int2 records = p.seg_records[sg];
  const int rows = rows_in_group(clamp_active(p.n_active[s], p.B), p.G, rg);
  constexpr int C = D / 32;
  for (int r = blockIdx.y * (kCombineThreads / 32) + warp; r < rows; r += gridDim.y * (kCombineThreads / 32)) {   // few CTAs per segment: most row blocks are empty on most steps
    const int row = rg * kRowsPerGroup + r, a = row / p.G, gi = row % p.G;
    const int tok = p.active_idx[s * p.B + a];
    if (tok < 0 || tok >= p.B) { set_status(p.status, LOSA_ERR_BOUNDS); continue; }
    const size_t orow = (static_cast<size_t>(s) * p.B + tok) * p.Hq + kh * p.G + gi;
    float acc[C], M, Lsum;
    merge_records<D, LOG2>(p, buf[warp], sg, r, records, lane, acc, M, Lsum);
    const bool empty = !(Lsum > 0.f);
    const float inv = empty ? 0.f : 1.f / Lsum;
#pragma unroll
    for (int c = 0; c < C; ++c) acc[c] *= inv;
    st_state<C>(p.o_p, p.o_p_bf16, orow * D + lane * C, acc);
    if (lane == 0) p.lse_p[orow] = empty ? -INFINITY : (LOG2 ? (M + log2f(Lsum)) * kLn2 : M + logf(Lsum));
  }
}

// Whole-step path, last kernel: one warp per (sequence, block token, head) row.
// An active row merges its partial records (as the combine kernel does) and stores the new prefix
// statistics; a stable row reads its cached ones (reuse rule, Section 4.2).  Either way the row is
// then merged with the in-block part by log-sum-exp (Section 2.2 / 4.3), the output is written and
// the row's query kept for the next step's Eq. 1; block 0 also bumps the step counters.
struct FinishParams {
  const void* q;
  void* q_prev;
  const float* o_b;
  const float* lse_b;
  void* out;
  float* lse_out;
  int32_t* step;
  const int32_t* slot_map;   // [N*B] slot of a block token in the active list, -1 = stable
  size_t n_rows;
};

constexpr int kFinishThreads = 128;

template <typename T, int D>
__global__ void __launch_bounds__(kFinishThreads) attn_finish_kernel(AttnParams p, FinishParams f) {
  constexpr bool LOG2 = !std::is_same_v<T, float>;     // partial maxima in base-2 units (tensor-core kernel)
  __shared__ __align__(16) float buf[kFinishThreads / 32][kMergeBatch * D];
  grid_dep_trigger();
  if constexpr (!LOG2) grid_dep_wait();                 // (fp32: launched behind an event, nothing runs beside it)
  constexpr int C = D / 32;
  const int lane = threadIdx.x & 31;
  const uint32_t row_i = blockIdx.x * (kFinishThreads / 32) + (threadIdx.x >> 5);
  const size_t row = row_i;
  const bool mine = row < f.n_rows;
  // The queries and the cached prefix statistics are older than the step, whose stage 1 has waited for all that is: they
  // are requested beside the kernels before this one.  Nine rows in ten are stable; an active row overwrites the
  // statistics below.  What the step itself writes, also in stage 1 (the slots), is read behind the wait: the kernels in
  // between release their dependents before they wait themselves.
  const int hq = static_cast<int>(row_i % p.Hq), st = static_cast<int>(row_i / p.Hq), tok = st % p.B, s = st / p.B;   // (32-bit divisions)
  const int kh = hq / p.G, gi = hq % p.G;
  const T* q = static_cast<const T*>(f.q);
  RawRow<C> qv;                                         // (fp32: qf)
  float qf[C];
  float a[C], Lp = 0.f;
  if (mine) {
    if constexpr (LOG2) qv = ld_raw<C>(q + row * D + lane * C);
    else ldv<C>(q + row * D + lane * C, qf);
    ld_state<C>(p.o_p, p.o_p_bf16, row * D + lane * C, a);
    Lp = p.lse_p[row];
  }
  if constexpr (LOG2) grid_dep_wait();
  if (blockIdx.x == 0)
    for (int s = threadIdx.x; s < p.N; s += kFinishThreads) f.step[s] += 1;
  if (!mine) return;
  // the slot in the active list (at most B entries), -1 = stable, and an active row's records, for the first row group, are
  // requested together (volatile: the records would sink below the look at the slot)
  int slot;
  asm volatile("ld.global.s32 %0, [%1];" : "=r"(slot) : "l"(f.slot_map + s * p.B + tok));
  float b[C];
  ldv<C>(f.o_b + row * D + lane * C, b);
  const float Lb = f.lse_b[row];
  int sg = s * p.Hkv + kh;
  int2 records;
  asm volatile("ld.global.v2.s32 {%0, %1}, [%2];" : "=r"(records.x), "=r"(records.y) : "l"(p.seg_records + sg));
  if (slot >= 0 && slot < p.B) {
    const int rowk = slot * p.G + gi, rg = rowk / kRowsPerGroup, r = rowk % kRowsPerGroup;
    if (rg > 0) {
      sg += rg * p.n_sk;
      records = p.seg_records[sg];
    }
    float acc[C], M, Lsum;
    merge_records<D, LOG2>(p, buf[threadIdx.x >> 5], sg, r, records, lane, acc, M, Lsum);
    const bool empty = !(Lsum > 0.f);
    const float inv = empty ? 0.f : 1.f / Lsum;
    Lp = empty ? -INFINITY : (LOG2 ? (M + log2f(Lsum)) * kLn2 : M + logf(Lsum));
#pragma unroll
    for (int c = 0; c < C; ++c) a[c] = acc[c] * inv;
    st_state<C>(p.o_p, p.o_p_bf16, row * D + lane * C, a);
    if (lane == 0) p.lse_p[row] = Lp;
  }
  const float Mx = fmaxf(Lp, Lb);
  const float L = Mx + logf(expf(Lp - Mx) + expf(Lb - Mx));
  const float wp = expf(Lp - L), wb = expf(Lb - L);
  T* out = static_cast<T*>(f.out);
  T* q_prev = static_cast<T*>(f.q_prev);
  float o[C];
#pragma unroll
  for (int c = 0; c < C; ++c) o[c] = (wp > 0.f ? wp * a[c] : 0.f) + wb * b[c];
  if constexpr (LOG2) {
    st_bf16<C>(out + row * D + lane * C, o);
    st_raw<C>(q_prev + row * D + lane * C, qv);
  } else {
    stv<C>(out + row * D + lane * C, o);
    stv<C>(q_prev + row * D + lane * C, qf);
  }
  if (f.lse_out && lane == 0) f.lse_out[row] = L;
}

// ===================================================================== bf16 TMA + tensor-core kernel: shared pieces
constexpr int kSmemBudget = 232448;                // 227 KB opt-in limit per CTA

constexpr int kStageIdx = 1024;     // active_idx entries (N * B) cached in shared memory when they fit
constexpr int kStageSeq = 64;       // ... together with n_active and kv_len of up to this many sequences
constexpr int kTailBytes = 512 + (kMaxSegments + 1) * 4 + 4 + kStageIdx * 4 + 2 * kStageSeq * 4;   // barriers, meta, prefix, index cache
// The K / V pages are read once per launch: they are marked evict-first in L2, so that the stream
// does not push out the small arrays the following kernels read (partial records, in-block output).
__device__ __forceinline__ unsigned long long l2_evict_first_policy() {
  unsigned long long pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0,
                                            int c1, int c2, int c3, unsigned long long policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(policy) : "memory");
}
// Loads whose issue point must stay where it is written (they are prefetches): volatile asm.
__device__ __forceinline__ int ld_nc_s32(const int32_t* ptr) {
  int v;
  asm volatile("ld.global.nc.s32 %0, [%1];" : "=r"(v) : "l"(ptr));
  return v;
}
// 2^x, one MUFU instruction (ex2.approx: 2 ulp; -inf -> 0); the bf16 rounding of P dwarfs its error
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
  const __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}


#include "sparse_prefix_attn_tc5.cuh"

// ===================================================================== host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

int32_t encode_pool_map(losa_ctx* c, unsigned char* blob, const void* pool, const losa_kv_t* kv, bool plain) {
  const losa_shape_t& sh = c->shape;
  if (!c->encode_fn) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    LOSA_CUDA_TRY(c, cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres));
    if (!fn || qres != cudaDriverEntryPointSuccess) return cuda_fail(c, cudaErrorSymbolNotFound);
    c->encode_fn = fn;
  }
  const cuuint64_t dims[4] = {static_cast<cuuint64_t>(sh.head_dim), static_cast<cuuint64_t>(sh.page_size),
                              static_cast<cuuint64_t>(sh.n_kv_heads), static_cast<cuuint64_t>(kv->n_phys_pages)};
  // bf16 pages: 64-element (128-byte) boxes with the 128-byte swizzle, as the MMA descriptors expect them;
  // FP8 pages: whole rows of d bytes; swizzled over the row (an MMA operand), or as they lie (V that the kernel converts)
  const bool fp8 = kv->kv_format == LOSA_KV_FP8_E4M3;
  const cuuint64_t es = fp8 ? 1 : 2;
  const cuuint64_t strides[3] = {static_cast<cuuint64_t>(kv->stride_tok) * es, static_cast<cuuint64_t>(kv->stride_head) * es,
                                 static_cast<cuuint64_t>(kv->stride_page) * es};
  const cuuint32_t box[4] = {fp8 ? static_cast<cuuint32_t>(sh.head_dim) : 64u, static_cast<cuuint32_t>(sh.page_size), 1, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = reinterpret_cast<EncodeTiledFn>(c->encode_fn)(
      reinterpret_cast<CUtensorMap*>(blob), fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4,
      const_cast<void*>(pool), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
      fp8 && plain ? CU_TENSOR_MAP_SWIZZLE_NONE : (fp8 && sh.head_dim == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B),
      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    c->last_cuda_error = static_cast<int32_t>(r);
    return LOSA_ERR_CUDA;
  }
  return LOSA_OK;
}

int32_t ensure_tensor_maps(losa_ctx* c, const losa_kv_t* kv) {
  const bool same = c->tmap_key_k == kv->k_pages && c->tmap_key_v == kv->v_pages &&
                    c->tmap_strides[0] == kv->stride_page && c->tmap_strides[1] == kv->stride_head &&
                    c->tmap_strides[2] == kv->stride_tok && c->tmap_n_phys == kv->n_phys_pages &&
                    c->tmap_format == kv->kv_format;
  if (same) return LOSA_OK;
  // (taken over together: a map of a new pool must not stay beside an old key when a later one cannot be encoded)
  alignas(64) unsigned char k[128], v[128], vs[128];
  const bool with_vs = kv->kv_format == LOSA_KV_FP8_E4M3 && c->shape.head_dim == 128;      // the kernel that has the narrow path
  int32_t rc = encode_pool_map(c, k, kv->k_pages, kv, false);
  if (rc == LOSA_OK) rc = encode_pool_map(c, v, kv->v_pages, kv, true);
  if (rc == LOSA_OK && with_vs) rc = encode_pool_map(c, vs, kv->v_pages, kv, false);
  if (rc != LOSA_OK) return rc;
  memcpy(c->tmap_k, k, sizeof(k));
  memcpy(c->tmap_v, v, sizeof(v));
  if (with_vs) memcpy(c->tmap_vs, vs, sizeof(vs));
  c->tmap_key_k = kv->k_pages;
  c->tmap_key_v = kv->v_pages;
  c->tmap_strides[0] = kv->stride_page;
  c->tmap_strides[1] = kv->stride_head;
  c->tmap_strides[2] = kv->stride_tok;
  c->tmap_n_phys = kv->n_phys_pages;
  c->tmap_format = kv->kv_format;
  return LOSA_OK;
}

// f(head dimension, page size) as compile-time numbers
template <typename F>
int32_t with_page_shape(const losa_shape_t& sh, F&& f) {
  auto page = [&](auto d) {
    switch (sh.page_size) {
      case 16: return f(d, std::integral_constant<int, 16>{});
      case 32: return f(d, std::integral_constant<int, 32>{});
      default: return f(d, std::integral_constant<int, 64>{});
    }
  };
  return sh.head_dim == 128 ? page(std::integral_constant<int, 128>{}) : page(std::integral_constant<int, 64>{});
}

template <int D, int GP, bool FP8>
int32_t prepare_tc5(losa_ctx* c) {
  constexpr int smem = tc5_smem_bytes<D, GP, FP8>();
  static_assert(smem <= kSmemBudget, "shared memory of the stage-4 kernel");
  constexpr int bit = FP8 ? 2 : 1;  // a context has one shape on one device: one instantiation per cache format
  if (c->attn_attr_set & bit) return LOSA_OK;
  auto set = [&](auto kernel) -> int32_t {
    LOSA_CUDA_TRY(c, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    // the kernel moves registers between its warps: a build that is launched with fewer than it deals out would wait for ever
    cudaFuncAttributes fa;
    LOSA_CUDA_TRY(c, cudaFuncGetAttributes(&fa, kernel));
    return fa.numRegs < (FP8 ? kTc5LaunchRegs8 : kTc5LaunchRegs) ? LOSA_ERR_UNSUPPORTED : LOSA_OK;
  };
  int32_t rc = set(attn_tc5_kernel<D, GP, FP8, false>);
  if constexpr (FP8 && D == 128)
    if (rc == LOSA_OK) rc = set(attn_tc5_kernel<D, GP, FP8, true>);
  if (rc != LOSA_OK) return rc;
  c->attn_attr_set |= bit;
  return LOSA_OK;
}

template <int D, int GP>
int32_t prepare_f32(losa_ctx* c) {
  constexpr int smem = sizeof(F32Smem<D>);
  static_assert(smem <= kSmemBudget, "shared memory of the fp32 stage-4 kernel");
  if (c->attn_attr_set & 1) return LOSA_OK;
  LOSA_CUDA_TRY(c, cudaFuncSetAttribute(attn_f32_kernel<D, GP, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  LOSA_CUDA_TRY(c, cudaFuncSetAttribute(attn_f32_kernel<D, GP, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  c->attn_attr_set |= 1;
  return LOSA_OK;
}

template <int D, int GP, bool FP8>
int32_t launch_tc5(losa_ctx* c, const AttnParams& ap, cudaStream_t st, bool with_combine) {
  if (c->profile) LOSA_CUDA_TRY(c, cudaEventRecord(c->ev_begin, st));
  auto launch = [&](auto kernel, const auto& maps) { launch_k(kernel, ap.n_ctas, tc5_threads<FP8>(), tc5_smem_bytes<D, GP, FP8>(), st, maps, ap); };
  auto map_of = [](const unsigned char* blob) {
    CUtensorMap m;
    memcpy(&m, blob, sizeof(m));
    return m;
  };
  const CUtensorMap mk = map_of(c->tmap_k), mv = map_of(c->tmap_v);
  // With the narrow path from 32 groups of 128 tokens per CTA in the whole table on.  How much of it the prompts fill, and whether a
  // step has few rows, is known on the device only: in the kernel that has both paths a step that takes the other one is 0.5 us
  // longer, in a large cache 1 % and less (64 segments, shares of 2 / 8 / 32 groups 18.0 / 27.6 / 55.9 us, 18.6 / 28.1 / 56.3).
  bool both = false;
  if constexpr (FP8 && D == 128) {
    both = static_cast<int64_t>(ap.n_sk) * ap.Pmax * GP >= static_cast<int64_t>(ap.n_ctas) * 32 * kTc5Tok;
    if (both) launch(attn_tc5_kernel<D, GP, FP8, true>, Tc5Maps<true>{mk, mv, map_of(c->tmap_vs)});
  }
  if (!both) launch(attn_tc5_kernel<D, GP, FP8, false>, Tc5Maps<false>{mk, mv});
  if (c->profile) LOSA_CUDA_TRY(c, cudaEventRecord(c->ev_end, st));
  int32_t rc = after_launch(c);
  if (rc != LOSA_OK || !with_combine) return rc;
  launch_k(attn_combine_kernel<D, true>, dim3(ap.n_seg, kCombineTiles), kCombineThreads, 0, st, ap);
  return after_launch(c);
}

template <int D, int GP>
int32_t launch_f32(losa_ctx* c, const AttnParams& ap, cudaStream_t st, bool with_combine) {
  if (c->profile) LOSA_CUDA_TRY(c, cudaEventRecord(c->ev_begin, st));
  launch_k(ap.union_bits ? attn_f32_kernel<D, GP, true> : attn_f32_kernel<D, GP, false>, ap.n_ctas, kF32Threads, sizeof(F32Smem<D>), st, ap);
  if (c->profile) LOSA_CUDA_TRY(c, cudaEventRecord(c->ev_end, st));
  int32_t rc = after_launch(c);
  if (rc != LOSA_OK || !with_combine) return rc;
  launch_k(attn_combine_kernel<D, false>, dim3(ap.n_seg, kCombineTiles), kCombineThreads, 0, st, ap);
  return after_launch(c);
}

}  // namespace


int32_t prepare_sparse_prefix_attn(losa_ctx* c, const losa_kv_t* kv) {
  const bool bf = c->shape.dtype == LOSA_BF16, fp8 = kv->kv_format == LOSA_KV_FP8_E4M3;     // (FP8 pages: bf16 contexts only)
  const int32_t rc = bf ? ensure_tensor_maps(c, kv) : LOSA_OK;
  if (rc != LOSA_OK) return rc;
  return with_page_shape(c->shape, [&](auto d, auto gp) {
    constexpr int D = decltype(d)::value, GP = decltype(gp)::value;
    return fp8 ? prepare_tc5<D, GP, true>(c) : bf ? prepare_tc5<D, GP, false>(c) : prepare_f32<D, GP>(c);
  });
}

int32_t launch_sparse_prefix_attn(losa_ctx* c, const void* q, const losa_kv_t* kv,
                                  const int32_t* active_idx, const int32_t* n_active,
                                  const int32_t* union_pages, const int32_t* union_count,
                                  losa_state_t* state, cudaStream_t st, bool defer_combine, bool from_bits) {
  const losa_shape_t& sh = c->shape;
  const int32_t rc = prepare_sparse_prefix_attn(c, kv);
  if (rc != LOSA_OK) return rc;
  AttnParams ap;
  ap.q = q;
  ap.k_pages = kv->k_pages;
  ap.v_pages = kv->v_pages;
  ap.stride_page = kv->stride_page;
  ap.stride_head = kv->stride_head;
  ap.stride_tok = kv->stride_tok;
  ap.page_table = kv->page_table;
  ap.kv_len = kv->kv_len;
  ap.active_idx = active_idx;
  ap.n_active = n_active;
  ap.union_pages = union_pages;
  ap.union_count = union_count;
  ap.union_bits = from_bits ? reinterpret_cast<const uint32_t*>(c->ws + c->lay.union_bits) : nullptr;
  ap.union_pages_out = from_bits ? const_cast<int32_t*>(union_pages) : nullptr;
  ap.union_count_out = from_bits ? const_cast<int32_t*>(union_count) : nullptr;
  ap.W = union_words(c);
  ap.partials = reinterpret_cast<float*>(c->ws + c->lay.partials);
  ap.seg_records = reinterpret_cast<int2*>(c->ws + c->lay.seg_records);
  ap.o_p = state->o_p;
  ap.o_p_bf16 = state->o_p_format == LOSA_STATE_BF16 ? 1 : 0;
  ap.lse_p = state->lse_p;
  ap.status = status_ptr(c);
  const bool fp8 = kv->kv_format == LOSA_KV_FP8_E4M3;
  ap.k_scale = fp8 ? kv->k_scale : nullptr;
  ap.v_scale = fp8 ? kv->v_scale : nullptr;
  ap.N = sh.batch;
  ap.B = sh.block_size;
  ap.Hq = sh.n_q_heads;
  ap.Hkv = sh.n_kv_heads;
  ap.G = sh.n_q_heads / sh.n_kv_heads;
  ap.Pmax = sh.max_pages_per_seq;
  ap.n_phys = kv->n_phys_pages;
  ap.n_rg = c->lay.n_row_groups;
  ap.n_seg = c->lay.n_segments;
  ap.n_sk = sh.batch * sh.n_kv_heads;
  ap.n_ctas = c->lay.n_ctas;
  ap.sm_scale = sh.sm_scale;
  ap.early = defer_combine ? 1 : 0;
  ap.wait_cycles = c->wait_cycles > 0 ? c->wait_cycles : kWaitCycles;
  const bool bf = sh.dtype == LOSA_BF16, with_combine = !defer_combine;
  return with_page_shape(sh, [&](auto d, auto gp) {
    constexpr int D = decltype(d)::value, GP = decltype(gp)::value;
    return fp8 ? launch_tc5<D, GP, true>(c, ap, st, with_combine)
               : bf ? launch_tc5<D, GP, false>(c, ap, st, with_combine) : launch_f32<D, GP>(c, ap, st, with_combine);
  });
}

int32_t launch_attn_finish(losa_ctx* c, const void* q, const int32_t* slot_map, losa_state_t* state, void* out,
                           float* lse_out_opt, cudaStream_t st) {
  const losa_shape_t& sh = c->shape;
  AttnParams ap = {};                       // (what the merge reads of it)
  ap.partials = reinterpret_cast<float*>(c->ws + c->lay.partials);
  ap.seg_records = reinterpret_cast<int2*>(c->ws + c->lay.seg_records);
  ap.o_p = state->o_p;
  ap.o_p_bf16 = state->o_p_format == LOSA_STATE_BF16 ? 1 : 0;
  ap.lse_p = state->lse_p;
  ap.N = sh.batch;
  ap.B = sh.block_size;
  ap.Hq = sh.n_q_heads;
  ap.Hkv = sh.n_kv_heads;
  ap.G = sh.n_q_heads / sh.n_kv_heads;
  ap.n_sk = sh.batch * sh.n_kv_heads;
  FinishParams fp;
  fp.q = q;
  fp.slot_map = slot_map;
  fp.q_prev = state->q_prev;
  fp.o_b = reinterpret_cast<const float*>(c->ws + c->lay.block_o);
  fp.lse_b = reinterpret_cast<const float*>(c->ws + c->lay.block_lse);
  fp.out = out;
  fp.lse_out = lse_out_opt;
  fp.step = state->step;
  fp.n_rows = static_cast<size_t>(sh.batch) * sh.block_size * sh.n_q_heads;
  const int blocks = static_cast<int>((fp.n_rows + kFinishThreads / 32 - 1) / (kFinishThreads / 32));
  if (sh.dtype == LOSA_BF16) {
    if (sh.head_dim == 128) launch_k(attn_finish_kernel<__nv_bfloat16, 128>, blocks, kFinishThreads, 0, st, ap, fp);
    else launch_k(attn_finish_kernel<__nv_bfloat16, 64>, blocks, kFinishThreads, 0, st, ap, fp);
  } else {
    if (sh.head_dim == 128) launch_k(attn_finish_kernel<float, 128>, blocks, kFinishThreads, 0, st, ap, fp);
    else launch_k(attn_finish_kernel<float, 64>, blocks, kFinishThreads, 0, st, ap, fp);
  }
  return after_launch(c);
}

}  // namespace losa
