// Stages 2 and 3 — QUEST page scores, top-k per active query, union per KV head
// (Section 2.3, Section 4.2, Section 4.4).
//
//   (the page scores themselves are computed by the kernel in page_scores.cu)
//   topk_select_kernel : one 128-thread CTA per (sequence, active token, head); threshold search over
//                        64-bit keys (order-preserving score bits, inverted page id), see below.
//   topk_kernel        : budgets above 512 pages: one CTA per query sorts all keys with a
//                        shared-memory bitonic network.
//   topk_refine_kernel : bf16, k <= 512 (the default): candidates from tensor-core bounds, exact scores
//                        for those only; in the whole-step call it also writes stage 3's union.
//   union_kernel       : one CTA per (sequence, KV head) ORs the selected ids into a bitmap and
//                        emits the set bits in ascending order with a popcount scan.
#include <algorithm>

#include "block_attn_mma.cuh"
#include "kernels.h"

namespace losa {
namespace {

constexpr int kThreads = 256;

// One score row, or (pooled selector) the element-wise maximum of the `g` consecutive rows of a KV
// head's query heads.
template <bool POOLED>
struct RowView {
  const float* base;
  int g, stride;
  __device__ __forceinline__ float operator[](int p) const {
    float v = base[p];
    if (POOLED)
      for (int gi = 1; gi < g; ++gi) v = fmaxf(v, base[static_cast<size_t>(gi) * stride + p]);
    return v;
  }
};

__device__ __forceinline__ uint32_t order_bits(float x) {
  const uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float unorder_bits(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

__global__ void __launch_bounds__(kThreads)
topk_kernel(const float* __restrict__ scores, const int32_t* __restrict__ kv_len,
            const int32_t* __restrict__ active_idx, const int32_t* __restrict__ n_active,
            const int32_t* __restrict__ step, int32_t* __restrict__ topk_pages,
            float* __restrict__ topk_scores, int B, int Hq, int g, int k, int Pmax, int score_stride, int pool,
            int32_t* __restrict__ status) {
  grid_dep_wait();
  extern __shared__ __align__(16) unsigned long long keys[];
  const int h = blockIdx.x * pool, a = blockIdx.y, s = blockIdx.z;   // pooled: first head of the KV head
  if (step && step[s] == 0) return;
  int na = n_active[s];
  na = na > B ? B : na;
  if (a >= na) return;
  int tok = active_idx[s * B + a];
  if (tok < 0 || tok >= B) { set_status(status, LOSA_ERR_BOUNDS); return; }
  int P = pages_of(kv_len[s], g);
  if (P > Pmax) { set_status(status, LOSA_ERR_BOUNDS); P = Pmax; }
  const int tid = threadIdx.x;
  int n = 2;
  while (n < P) n <<= 1;
  const RowView<true> sc{scores + ((static_cast<size_t>(s) * B + a) * Hq + h) * score_stride, pool, score_stride};
  for (int p = tid; p < n; p += kThreads)
    keys[p] = (p < P) ? ((static_cast<unsigned long long>(order_bits(sc[p])) << 32) |
                         static_cast<unsigned long long>(0xffffffffu - static_cast<uint32_t>(p)))
                      : 0ull;
  __syncthreads();
  // bitonic network, descending
  for (int k2 = 2; k2 <= n; k2 <<= 1) {
    for (int j = k2 >> 1; j > 0; j >>= 1) {
      for (int t = tid; t < (n >> 1); t += kThreads) {
        const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1));
        const int x = i | j;
        const unsigned long long ka = keys[i], kb = keys[x];
        const bool desc = (i & k2) == 0;
        if ((ka < kb) == desc) { keys[i] = kb; keys[x] = ka; }
      }
      __syncthreads();
    }
  }
  for (int gi = 0; gi < pool; ++gi) {                 // pooled: every head of the group gets the list
    const size_t o = ((static_cast<size_t>(s) * B + tok) * Hq + h + gi) * k;
    for (int j = tid; j < k; j += kThreads) {
      if (j < P) {
        const unsigned long long key = keys[j];
        topk_pages[o + j] = static_cast<int32_t>(0xffffffffu - static_cast<uint32_t>(key));
        if (topk_scores) topk_scores[o + j] = unorder_bits(static_cast<uint32_t>(key >> 32));
      } else {
        topk_pages[o + j] = -1;
      }
    }
  }
}

// ---- top-k by threshold search: one small CTA per query, O(P) work ---------------------------
// Keys are (order-preserving score bits, inverted page id), all distinct, so "the k largest keys"
// is the required answer with ties already broken.  The CTA histograms the score bits of the
// still-undecided range into 256 equal-width bins, finds the bin holding the k-th largest, takes
// every key above that bin, and either finishes by sorting "taken + threshold bin" (a few dozen
// keys) or narrows the range to the threshold bin and repeats.  A range of one value means the
// remaining candidates tie on the score: the lowest page ids win, taken in page order.
constexpr int kSelCap = kListCap;   // candidate keys a CTA can sort; also the largest k of this path
constexpr int kSelBins = 256;

__device__ __forceinline__ unsigned long long make_key(uint32_t ob, int p) {
  return (static_cast<unsigned long long>(ob) << 32) |
         static_cast<unsigned long long>(0xffffffffu - static_cast<uint32_t>(p));
}

// One CTA of kSelThreads per query.  Thread t owns keys p = t + kSelThreads * i; with CACHED
// (P <= kSelThreads * kSelPerThread) their order bits stay in registers for the whole selection.
constexpr int kSelThreads = 128;
constexpr int kSelPerThread = 8;
constexpr int kCrowd = 32;          // lists whose candidates crowd more than that into one bin take exact scores for all of them
constexpr int kSelSlots = 8;        // CTAs per (sequence, head), at most: active slots are dealt out round-robin

template <bool CACHED, typename Row, typename F>
__device__ __forceinline__ void for_each_key(const uint32_t (&cache)[kSelPerThread], const Row& row,
                                             int P, int tid, F&& f) {
  if (CACHED) {
#pragma unroll
    for (int i = 0; i < kSelPerThread; ++i) {
      const int p = tid + kSelThreads * i;
      if (p < P) f(cache[i], p);
    }
  } else {
    for (int p = tid; p < P; p += kSelThreads) f(order_bits(row[p]), p);
  }
}

// bits: page bitmap that the chosen pages are ORed into, or null.
template <bool CACHED, typename Row>
__device__ __forceinline__ void topk_select_body(const Row& row, int P, int kk, int k,
                                                 int32_t* out_pages, float* out_scores, int n_out, uint32_t* bits) {
  __shared__ __align__(16) unsigned long long cand[kSelCap];
  __shared__ int hist[kSelBins];
  __shared__ uint32_t s_red[2][kSelThreads / 32];
  __shared__ int s_ncand, s_bstar, s_above, s_thr;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t cache[kSelPerThread];
  if (CACHED) {
#pragma unroll
    for (int i = 0; i < kSelPerThread; ++i) {
      const int p = tid + kSelThreads * i;
      cache[i] = p < P ? order_bits(row[p]) : 0u;
    }
  }
  uint32_t lo = 0xffffffffu, hi = 0u;
  for_each_key<CACHED, Row>(cache, row, P, tid, [&](uint32_t ob, int) { lo = min(lo, ob); hi = max(hi, ob); });
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) { s_red[0][warp] = lo; s_red[1][warp] = hi; }
  if (tid == 0) s_ncand = 0;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kSelThreads / 32; ++w) { lo = min(lo, s_red[0][w]); hi = max(hi, s_red[1][w]); }
  int need = kk;
  while (need > 0) {
    if (lo == hi) {
      // every remaining candidate has the same score: lowest pages first, in page order (rare;
      // one warp walks the pages so that the order is kept)
      if (warp == 0) {
        int ncand = s_ncand;
        const unsigned below = (1u << lane) - 1u;
        for (int base = 0; base < P && need > 0; base += 32) {
          const int p = base + lane;
          const bool hit = p < P && order_bits(row[p]) == lo;
          const unsigned bal = __ballot_sync(0xffffffffu, hit);
          const int rank = __popc(bal & below);
          if (hit && rank < need) cand[ncand + rank] = make_key(lo, p);
          const int taken = min(need, __popc(bal));
          ncand += taken;
          need -= taken;
        }
        if (lane == 0) s_ncand = ncand;
      }
      break;
    }
    const int width = 32 - __clz(hi - lo);           // bits needed for hi - lo  (>= 1)
    const int shift = width > 8 ? width - 8 : 0;      // (ob - lo) >> shift is in [0, 255]
    for (int b = tid; b < kSelBins; b += kSelThreads) hist[b] = 0;
    __syncthreads();
    for_each_key<CACHED, Row>(cache, row, P, tid, [&](uint32_t ob, int) {
      if (ob >= lo && ob <= hi) atomicAdd(&hist[(ob - lo) >> shift], 1);
    });
    __syncthreads();
    if (warp == 0) {
      // lane owns bins [8*lane, 8*lane+8); suffix sums over lanes locate the threshold bin
      int c[8], tot = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) { c[e] = hist[8 * lane + e]; tot += c[e]; }
      int suf = tot;                                   // inclusive suffix: lanes >= this one
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_down_sync(0xffffffffu, suf, o);
        if (lane + o < 32) suf += t;
      }
      const int above_lanes = suf - tot;
      if (above_lanes < need && need <= suf) {
        int run = above_lanes;
#pragma unroll
        for (int e = 7; e >= 0; --e) {
          if (run < need && need <= run + c[e]) { s_bstar = 8 * lane + e; s_above = run; s_thr = c[e]; }
          run += c[e];
        }
      }
    }
    __syncthreads();
    const int bstar = s_bstar, cnt_above = s_above, cnt_thr = s_thr;
    const bool finish = s_ncand + cnt_above + cnt_thr <= kSelCap;
    __syncthreads();                                   // everyone has read s_ncand before it moves
    // take the keys above the threshold bin (and, when finishing, the threshold bin itself); the
    // order inside cand does not matter: it is sorted below
    for_each_key<CACHED, Row>(cache, row, P, tid, [&](uint32_t ob, int p) {
      if (ob >= lo && ob <= hi) {
        const int bin = static_cast<int>((ob - lo) >> shift);
        if (bin > bstar || (finish && bin == bstar)) cand[atomicAdd(&s_ncand, 1)] = make_key(ob, p);
      }
    });
    if (finish) break;
    need -= cnt_above;
    const uint32_t nlo = lo + (static_cast<uint32_t>(bstar) << shift);
    const unsigned long long top = static_cast<unsigned long long>(nlo) + ((1ull << shift) - 1ull);
    hi = top < hi ? static_cast<uint32_t>(top) : hi;
    lo = nlo;
    __syncthreads();
  }
  __syncthreads();
  // order the candidates (descending) and emit the first kk
  const int ncand = s_ncand;
  auto emit = [&](int rank, unsigned long long key) {
    const int pg = static_cast<int32_t>(0xffffffffu - static_cast<uint32_t>(key));
    for (int gi = 0; gi < n_out; ++gi) {               // pooled: the list goes to every head of the group
      out_pages[gi * k + rank] = pg;
      if (out_scores) out_scores[gi * k + rank] = unorder_bits(static_cast<uint32_t>(key >> 32));
    }
    if (bits) atomicOr(&bits[pg >> 5], 1u << (pg & 31));
  };
  if (ncand <= kSelThreads) {                          // few: a candidate's position is the number of larger keys (all differ)
    if ((tid & ~31) < ncand) {
      const unsigned long long mine = tid < ncand ? cand[tid] : ~0ull;
      int rank = 0;
      for (int i = 0; i < ncand; ++i) rank += cand[i] > mine ? 1 : 0;
      if (tid < ncand && rank < kk) emit(rank, mine);
    }
  } else {
    int n2 = 2;
    while (n2 < ncand) n2 <<= 1;
    for (int i = ncand + tid; i < n2; i += kSelThreads) cand[i] = 0ull;
    __syncthreads();
    for (int k2 = 2; k2 <= n2; k2 <<= 1) {
      for (int j = k2 >> 1; j > 0; j >>= 1) {
        for (int t = tid; t < (n2 >> 1); t += kSelThreads) {
          const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1));
          const int x = i | j;
          const unsigned long long ka = cand[i], kb = cand[x];
          if ((ka < kb) == ((i & k2) == 0)) { cand[i] = kb; cand[x] = ka; }
        }
        __syncthreads();
      }
    }
    for (int j = tid; j < kk; j += kSelThreads) emit(j, cand[j]);
  }
  for (int gi = 0; gi < n_out; ++gi)
    for (int j = kk + tid; j < k; j += kSelThreads) out_pages[gi * k + j] = -1;
}


// ---- bf16 fast path: candidates from tensor-core bounds, exact scores for the candidates only ----
// The page score in the order the interface fixes, by four lanes (u = lane % 4; qs: [q+ (D) | q- (D)]
// fp32 in shared memory): lane u runs the chains of runs u, u + 4(, u + 8, u + 12) - 16 fused
// multiply-adds per run of 8 dimensions - and the butterfly c[i] += c[i ^ off], off = D/16 .. 1, is
// taken inside the lane while off >= 4 and with two shuffles below that.  All four lanes return it.
template <int D> struct SummaryRuns { uint4 lo[D / 32], hi[D / 32]; };      // a lane's runs of one page's kmin and kmax
template <int D>
__device__ __forceinline__ SummaryRuns<D> load_summary(const __nv_bfloat16* __restrict__ lo_p, const __nv_bfloat16* __restrict__ hi_p, int u) {
  SummaryRuns<D> r;                // requested together, converted run by run
#pragma unroll
  for (int w = 0; w < D / 32; ++w) {
    r.lo[w] = __ldg(reinterpret_cast<const uint4*>(lo_p + 8 * (u + 4 * w)));
    r.hi[w] = __ldg(reinterpret_cast<const uint4*>(hi_p + 8 * (u + 4 * w)));
  }
  return r;
}
template <int D>
__device__ __forceinline__ float exact_score4(const float* __restrict__ qs, const SummaryRuns<D>& r, int u) {
  constexpr int RPL = D / 32;      // runs per lane
  float c[RPL];
#pragma unroll
  for (int w = 0; w < RPL; ++w) {
    const int t = u + 4 * w;
    const uint32_t lw[4] = {r.lo[w].x, r.lo[w].y, r.lo[w].z, r.lo[w].w};
    const uint32_t hw[4] = {r.hi[w].x, r.hi[w].y, r.hi[w].z, r.hi[w].w};
    float acc = 0.f;
#pragma unroll
    for (int j4 = 0; j4 < 2; ++j4) {
      const float4 qp = *reinterpret_cast<const float4*>(qs + 8 * t + 4 * j4);
      const float4 qn = *reinterpret_cast<const float4*>(qs + D + 8 * t + 4 * j4);
      acc = __fmaf_rn(qp.x, __uint_as_float(hw[2 * j4] << 16), acc);
      acc = __fmaf_rn(qn.x, __uint_as_float(lw[2 * j4] << 16), acc);
      acc = __fmaf_rn(qp.y, __uint_as_float(hw[2 * j4] & 0xffff0000u), acc);
      acc = __fmaf_rn(qn.y, __uint_as_float(lw[2 * j4] & 0xffff0000u), acc);
      acc = __fmaf_rn(qp.z, __uint_as_float(hw[2 * j4 + 1] << 16), acc);
      acc = __fmaf_rn(qn.z, __uint_as_float(lw[2 * j4 + 1] << 16), acc);
      acc = __fmaf_rn(qp.w, __uint_as_float(hw[2 * j4 + 1] & 0xffff0000u), acc);
      acc = __fmaf_rn(qn.w, __uint_as_float(lw[2 * j4 + 1] & 0xffff0000u), acc);
    }
    c[w] = acc;
  }
  float v;
  if constexpr (RPL == 4) v = __fadd_rn(__fadd_rn(c[0], c[2]), __fadd_rn(c[1], c[3]));   // off = 8, then off = 4
  else v = __fadd_rn(c[0], c[1]);                                                         // off = 4
  v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 2));
  v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return __fadd_rn(v, 0.0f);
}

struct RefineParams {
  float2* bounds;                 // (A - delta, A + delta) per (row, page); reused as fp32 score rows by the fallback
  const __nv_bfloat16* q;
  const __nv_bfloat16* kmin;
  const __nv_bfloat16* kmax;
  const int32_t* page_table;
  const int32_t* kv_len;
  const int32_t* active_idx;
  const int32_t* n_active;
  const int32_t* step;
  int32_t* topk_pages;
  float* topk_scores;
  int32_t* status;
  int N, B, Hq, Hkv, g, k, score_stride, Pmax, n_phys;
  // stage 3 inside this kernel (whole-step call): the lists are ORed into one bitmap per (sequence, KV
  // head) as they are emitted, and the last CTA of a (sequence, KV head) to finish writes the union.
  // union_bits == nullptr: lists only.
  uint32_t* union_bits;           // [N][Hkv][W] words, all zero between launches
  unsigned int* union_tickets;    // [N][Hkv] arrival counters, self-resetting
  int32_t* union_pages;
  int32_t* union_count;
  int W;                          // words per bitmap, ceil(Pmax / 32) <= kSelBins
  int bound_rows;                 // pooled: rows of bounds per list: the heads' own, or 1 where the bounds kernel has pooled them
  int slots;                      // CTAs per (sequence, head or KV head): active slots are dealt out round-robin
  int blk_tiles;                  // row tiles of the in-block attention per (sequence, KV head)
};

// The set bits of a bitmap in shared memory, ascending, then -1 up to Pmax; the count.  All NT threads
// of the CTA call it; s_warp: NT / 32 ints of shared memory.
template <int NT>
__device__ __forceinline__ void union_emit(const uint32_t* bitmap, int W, int Pmax, int32_t* __restrict__ out,
                                           int32_t* __restrict__ count, int* s_warp) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // each thread owns a contiguous run of words; exclusive scan of the per-thread popcounts
  const int per = (W + NT - 1) / NT;
  const int w0 = tid * per, w1 = min(W, w0 + per);
  int cnt = 0;
  for (int w = w0; w < w1; ++w) cnt += __popc(bitmap[w]);
  int inc = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  int base = 0, total = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    if (w < warp) base += s_warp[w];
    total += s_warp[w];
  }
  int pos = base + inc - cnt;
  for (int w = w0; w < w1; ++w) {
    uint32_t v = bitmap[w];
    while (v) {
      const int b = __ffs(v) - 1;
      v &= v - 1;
      out[pos++] = w * 32 + b;
    }
  }
  for (int t = total + tid; t < Pmax; t += NT) out[t] = -1;
  if (tid == 0) *count = total;
}

__device__ __forceinline__ uint32_t prefix_word(int w, int P) {   // word w of the bitmap "pages 0 .. P-1"
  const int lo = w * 32;
  return (P >= lo + 32) ? 0xffffffffu : (P > lo ? ((1u << (P - lo)) - 1u) : 0u);
}

// How many of n keys (all different) are larger than `mine`: read as broadcasts, four at a time.
__device__ __forceinline__ int larger_keys(const unsigned long long* keys, int n, unsigned long long mine) {
  int rank = 0;
  const int n4 = n & ~3;
  for (int i = 0; i < n4; i += 4) {
    const ulonglong2 k01 = *reinterpret_cast<const ulonglong2*>(&keys[i]);
    const ulonglong2 k23 = *reinterpret_cast<const ulonglong2*>(&keys[i + 2]);
    rank += (k01.x > mine ? 1 : 0) + (k01.y > mine ? 1 : 0) + (k23.x > mine ? 1 : 0) + (k23.y > mine ? 1 : 0);
  }
  for (int i = n4; i < n; ++i) rank += keys[i] > mine ? 1 : 0;
  return rank;
}

// One CTA of kSelThreads per (sequence, head, share of the active slots).  Per query: tau = lower edge
// of the histogram bin that holds the k-th largest LOWER bound; every page whose UPPER bound reaches
// tau is a candidate (a superset of the exact top-k, ties included: the exact score lies between the
// bounds); the candidates by descending lower bound; exact scores in the fixed order (four lanes each) only
// for those that lie so close to a neighbour that the bounds leave their order open; emit.  More
// than kSelCap candidates (possible only when most pages nearly tie): exact scores for every page
// into the score row, then the plain threshold search.
// POOLED (one list per KV head, Section 4.2's selector with the group's maximum as the page score):
// a CTA serves the G heads of a KV head at once.  max over the heads of the lower (upper) bounds is
// a lower (upper) bound of the pooled score, so the same search applies to those; a candidate's
// exact score is the largest of its G exact scores; the list goes to every head of the group.
constexpr int kMaxPool = 16;     // heads per KV head the interface admits

template <int D, bool POOLED>
struct RefineSmem {
  float qs[(POOLED ? kMaxPool : 1) * 2 * D];
  unsigned long long ckey[kSelCap];              // candidates: exact score and page (RUNS: first, as found, lower bound and page)
  union {
    struct { int cpage[kSelCap], cphys[kSelCap]; };
    unsigned long long skey[kSelCap];            // RUNS: by descending lower bound
  };
  union { alignas(8) int hist[kSelBins]; uint16_t close[kSelCap]; };   // (close: once tau is known)
  uint32_t run[kSelCap / 32];                    // bit r: a run of close candidates starts at position r
  uint32_t red[2][kSelThreads / 32];
  uint32_t width;                                // the widest pair of bounds, rounded up: the bits of a float
  int ncand, nclose, bstar;
};
static_assert(kSelBins * sizeof(int) >= kSelCap * sizeof(uint16_t) && kSelBins == 2 * kSelThreads, "positions; two bins per thread");

// In a whole step the grid ends with the row tiles of the in-block attention (BK: its padded key
// count).  It needs only the step's inputs, and these CTAs fill the gaps of a kernel that is bound by
// latency.  On a second stream it was hidden as well, but the join in front of the step's last kernel
// cost that kernel its early launch (4 us of idle GPU per step); in stage 1's launch it delayed stage
// 2 (eight sequences: bounds from 12 us on instead of 7).
template <int D, bool POOLED, int BK, bool RUNS>
__global__ void __launch_bounds__(kSelThreads, POOLED ? 4 : 6)
topk_refine_kernel(RefineParams p, BlockAttnParams bp) {
  static_assert(kSelThreads == kMmaThreads, "one CTA size");
  __shared__ __align__(16) union { RefineSmem<D, POOLED> r; BlockAttnSmem<D, BK> b; } sm;
  const int qid = blockIdx.x, n_refine = p.N * (POOLED ? p.Hkv : p.Hq) * p.slots;
  if (qid >= n_refine) {
    const int t = qid - n_refine, sk = t / p.blk_tiles;
    if (!(p.step && __ldcg(p.step + sk / p.Hkv) == 0)) grid_dep_trigger();      // (as below)
    grid_dep_wait();
    block_attn_mma_cta<D, BK, false, 64>(bp, sm.b, t % p.blk_tiles, sk % p.Hkv, sk / p.Hkv);
    return;
  }
  const int pool = POOLED ? p.Hq / p.Hkv : 1, Hl = p.Hq / pool;
  const int h = (qid % Hl) * pool, s = (qid / Hl) % p.N, j0 = qid / (Hl * p.N);   // pooled: h = the group's first head
  // With stage 3 inside (whole-step call) the next kernel is stage 4, and the chain of launches
  // guarantees that the step counters are final before any CTA of this kernel runs.  On a first step
  // stage 4 is not released early: its CTAs then take the SMs in launch order once this grid has
  // drained, which its dense pass is measurably faster with (one sequence: 38 against 46 us).
  bool first_step;
  if (p.union_bits) {
    first_step = p.step && __ldcg(p.step + s) == 0;
    if (!first_step) grid_dep_trigger();
  } else {
    grid_dep_trigger();
  }
  grid_dep_wait();
  if (!p.union_bits) first_step = p.step && p.step[s] == 0;
  float* qs = sm.r.qs;
  unsigned long long* ckey = sm.r.ckey;
  int* cpage = sm.r.cpage;
  int* hist = sm.r.hist;
  uint32_t (&s_red)[2][kSelThreads / 32] = sm.r.red;
  int& s_ncand = sm.r.ncand;
  int& s_bstar = sm.r.bstar;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int kh = h / (p.Hq / p.Hkv);
  int na = first_step ? 0 : p.n_active[s];
  na = na > p.B ? p.B : na;
  if (na <= 0) {
    // no lists for this sequence: on the first step of a block the union is the whole prefix, with
    // no active token it is empty; written by the first CTA of the (sequence, KV head)
    if (!p.union_bits || j0 != 0 || h != kh * (p.Hq / p.Hkv)) return;
    const int P0 = first_step ? min(pages_of(p.kv_len[s], p.g), p.Pmax) : 0;
    uint32_t* bm = reinterpret_cast<uint32_t*>(hist);
    for (int w = tid; w < p.W; w += kSelThreads) bm[w] = prefix_word(w, P0);
    __syncthreads();
    union_emit<kSelThreads>(bm, p.W, p.Pmax, p.union_pages + (static_cast<size_t>(s) * p.Hkv + kh) * p.Pmax,
                            p.union_count + s * p.Hkv + kh, reinterpret_cast<int*>(s_red[0]));
    return;
  }
  if (j0 >= na) return;                                  // no slot for this CTA
  int P = pages_of(p.kv_len[s], p.g);
  if (P > p.Pmax) { if (tid == 0) set_status(p.status, LOSA_ERR_BOUNDS); P = p.Pmax; }
  const int kk = min(p.k, P);
  uint32_t* bits = p.union_bits ? p.union_bits + (static_cast<size_t>(s) * p.Hkv + kh) * p.W : nullptr;
  auto mark = [&](int pg) { if (bits) atomicOr(&bits[pg >> 5], 1u << (pg & 31)); };
  const __nv_bfloat16* lo_base = p.kmin + static_cast<size_t>(kh) * D;
  const __nv_bfloat16* hi_base = p.kmax + static_cast<size_t>(kh) * D;
  const int u = lane & 3;
  for (int a = j0; a < na; a += p.slots) {
    const int tok = p.active_idx[s * p.B + a];
    if (tok < 0 || tok >= p.B) { if (tid == 0) set_status(p.status, LOSA_ERR_BOUNDS); continue; }
    float2* row2 = p.bounds + ((static_cast<size_t>(s) * p.B + a) * p.Hq + h) * p.score_stride;
    const size_t o = ((static_cast<size_t>(s) * p.B + tok) * p.Hq + h) * p.k;
    int32_t* out_pages = p.topk_pages + o;
    float* out_scores = p.topk_scores ? p.topk_scores + o : nullptr;
    // the bounds of this thread's pages: one round trip, kept in registers when the prefix has at
    // most kSelThreads * kSelPerThread pages
    const bool cached = P <= kSelThreads * kSelPerThread;
    if constexpr (POOLED) {
      if (!cached && p.bound_rows > 1) {
        // the passes below read the row several times: pool once, into the group's first row (the
        // rows are scratch, this CTA is their only reader, and a thread reads back only what it wrote)
        constexpr int U = 4;                                   // pages per thread whose loads are in flight together
        for (int p0 = tid; p0 < P; p0 += kSelThreads * U) {
          float2 v[U];
#pragma unroll
          for (int e = 0; e < U; ++e) v[e] = p0 + e * kSelThreads < P ? row2[p0 + e * kSelThreads] : make_float2(0.f, 0.f);
          for (int gi = 1; gi < p.bound_rows; ++gi) {
            float2 w[U];
#pragma unroll
            for (int e = 0; e < U; ++e)
              w[e] = p0 + e * kSelThreads < P ? row2[static_cast<size_t>(gi) * p.score_stride + p0 + e * kSelThreads]
                                              : make_float2(0.f, 0.f);
#pragma unroll
            for (int e = 0; e < U; ++e) { v[e].x = fmaxf(v[e].x, w[e].x); v[e].y = fmaxf(v[e].y, w[e].y); }
          }
#pragma unroll
          for (int e = 0; e < U; ++e)
            if (p0 + e * kSelThreads < P) row2[p0 + e * kSelThreads] = v[e];
        }
      }
    }
    uint32_t lbc[kSelPerThread], ubc[kSelPerThread];
    float width = 0.f;                                     // of the widest pair of bounds, rounded up
    if (cached) {
      float2 bv[kSelPerThread];
#pragma unroll
      for (int i = 0; i < kSelPerThread; ++i) {
        const int pg = tid + kSelThreads * i;
        bv[i] = pg < P ? row2[pg] : make_float2(0.f, 0.f);
      }
      if constexpr (POOLED) {
        for (int gi = 1; gi < p.bound_rows; ++gi) {
          float2 bg[kSelPerThread];
#pragma unroll
          for (int i = 0; i < kSelPerThread; ++i) {
            const int pg = tid + kSelThreads * i;
            bg[i] = pg < P ? row2[static_cast<size_t>(gi) * p.score_stride + pg] : make_float2(0.f, 0.f);
          }
#pragma unroll
          for (int i = 0; i < kSelPerThread; ++i) {
            bv[i].x = fmaxf(bv[i].x, bg[i].x);
            bv[i].y = fmaxf(bv[i].y, bg[i].y);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < kSelPerThread; ++i) {
        if (RUNS) width = fmaxf(width, __fsub_ru(bv[i].y, bv[i].x));
        lbc[i] = order_bits(bv[i].x);
        ubc[i] = order_bits(bv[i].y);
      }
    }
    auto for_each_page = [&](auto&& f) {        // f(lower bits, upper bits, page)
      if (cached) {
#pragma unroll
        for (int i = 0; i < kSelPerThread; ++i) {
          const int pg = tid + kSelThreads * i;
          if (pg < P) f(lbc[i], ubc[i], pg);
        }
      } else {
        for (int pg = tid; pg < P; pg += kSelThreads) {
          const float2 bv = row2[pg];                  // pooled: already the group's maximum
          f(order_bits(bv.x), order_bits(bv.y), pg);
        }
      }
    };
    // the query, split into its positive and negative parts
    for (int j = tid; j < pool * D; j += kSelThreads) {       // the group's heads are consecutive in q
      const float v = __bfloat162float(p.q[((static_cast<size_t>(s) * p.B + tok) * p.Hq + h) * D + j]);
      const int gi = j / D, d = j % D;
      qs[gi * 2 * D + d] = fmaxf(v, 0.f);
      qs[gi * 2 * D + D + d] = fminf(v, 0.f);
    }
    if (tid == 0) { s_ncand = 0; sm.r.nclose = 0; sm.r.width = 0u; }
    for (int b = tid; b < kSelBins; b += kSelThreads) hist[b] = 0;
    // ---- tau
    uint32_t tau = 0u;
    bool crowded = false;                          // RUNS: all bounds the same, or more than kCrowd pages in one of this thread's bins that reach the list
    if (kk < P) {
      uint32_t lo = 0xffffffffu, hi = 0u;
      for_each_page([&](uint32_t lb, uint32_t, int) { lo = min(lo, lb); hi = max(hi, lb); });
      lo = __reduce_min_sync(0xffffffffu, lo);
      hi = __reduce_max_sync(0xffffffffu, hi);
      if (lane == 0) { s_red[0][warp] = lo; s_red[1][warp] = hi; }
      __syncthreads();
#pragma unroll
      for (int w = 0; w < kSelThreads / 32; ++w) { lo = min(lo, s_red[0][w]); hi = max(hi, s_red[1][w]); }
      if (lo < hi) {
        const int bits_of = 32 - __clz(hi - lo);
        const int shift = bits_of > 8 ? bits_of - 8 : 0;
        for_each_page([&](uint32_t lb, uint32_t, int) { atomicAdd(&hist[(lb - lo) >> shift], 1); });
        __syncthreads();
        if (warp == 0) {
          int c[8], tot = 0;
#pragma unroll
          for (int e = 0; e < 8; ++e) { c[e] = hist[8 * lane + e]; tot += c[e]; }
          int suf = tot;
#pragma unroll
          for (int off = 1; off < 32; off <<= 1) {
            const int t = __shfl_down_sync(0xffffffffu, suf, off);
            if (lane + off < 32) suf += t;
          }
          const int above_lanes = suf - tot;
          if (above_lanes < kk && kk <= suf) {
            int run = above_lanes;
#pragma unroll
            for (int e = 7; e >= 0; --e) {
              if (run < kk && kk <= run + c[e]) s_bstar = 8 * lane + e;
              run += c[e];
            }
          }
        }
        __syncthreads();
        const int bstar = s_bstar;
        tau = lo + (static_cast<uint32_t>(bstar) << shift);
        if (RUNS) {
          const int2 c = *reinterpret_cast<const int2*>(&hist[2 * tid]);
          crowded = (2 * tid >= bstar && c.x > kCrowd) || (2 * tid + 1 >= bstar && c.y > kCrowd);
        }
      } else {
        tau = lo;
        crowded = true;
      }
    } else {
      __syncthreads();
    }
    // ---- candidates: pages whose upper bound reaches tau
    // (one ticket per warp for all of its pages: a ticket per page is a chain of eight shared-memory round trips, which
    // five CTAs per SM share; eight 32K prompts 4,200 cycles, 1,200 now)
    if (cached) {
      uint32_t hit[kSelPerThread];
      int total = 0;
#pragma unroll
      for (int i = 0; i < kSelPerThread; ++i) {
        hit[i] = __ballot_sync(0xffffffffu, tid + kSelThreads * i < P && ubc[i] >= tau);
        total += __popc(hit[i]);
      }
      int at = 0;
      if (lane == 0 && total > 0) at = atomicAdd(&s_ncand, total);
      at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
      for (int i = 0; i < kSelPerThread; ++i) {
        const int mine = at + __popc(hit[i] & ((1u << lane) - 1u));
        if (((hit[i] >> lane) & 1u) && mine < kSelCap) {
          if (RUNS) ckey[mine] = make_key(lbc[i], tid + kSelThreads * i);
          else cpage[mine] = tid + kSelThreads * i;
        }
        at += __popc(hit[i]);
      }
    } else {
      for_each_page([&](uint32_t lb, uint32_t ub, int pg) {
        if (ub >= tau) {
          const int i = atomicAdd(&s_ncand, 1);
          if (i < kSelCap) {
            if (RUNS) ckey[i] = make_key(lb, pg);
            else cpage[i] = pg;
          }
          if (RUNS) width = fmaxf(width, __fsub_ru(unorder_bits(ub), unorder_bits(lb)));
        }
      });
    }
    if constexpr (RUNS) crowded = __syncthreads_or(crowded) != 0;
    else __syncthreads();
    const int ncand = s_ncand;
    auto phys_of = [&](int pg) {
      int ph = __ldg(p.page_table + static_cast<size_t>(s) * p.Pmax + pg);
      if (ph < 0 || ph >= p.n_phys) { set_status(p.status, LOSA_ERR_BOUNDS); ph = 0; }
      return ph;
    };
    auto exact_at = [&](int ph) {                 // called by the four lanes of a group with the same page
      const size_t so = static_cast<size_t>(ph) * p.Hkv * D;
      const SummaryRuns<D> sr = load_summary<D>(lo_base + so, hi_base + so, u);
      float e = exact_score4<D>(qs, sr, u);
      if constexpr (POOLED) {                      // the summary serves all heads of the group
#pragma unroll 1
        for (int gi = 1; gi < pool; ++gi) e = fmaxf(e, exact_score4<D>(qs + gi * 2 * D, sr, u));
      }
      return e;
    };
    auto emit = [&](int rank, unsigned long long key) {      // entry `rank` of the list
      const int pg = static_cast<int32_t>(0xffffffffu - static_cast<uint32_t>(key));
      for (int gi = 0; gi < pool; ++gi) {
        out_pages[gi * p.k + rank] = pg;
        if (out_scores) out_scores[gi * p.k + rank] = unorder_bits(static_cast<uint32_t>(key >> 32));
      }
      mark(pg);
    };
    if (ncand > kSelCap) {
      float* row = reinterpret_cast<float*>(row2);             // the bounds are not needed any more
      for (int p0 = 0; p0 < P; p0 += kSelThreads / 4) {          // whole warps: the shuffles need all lanes
        const int pg = min(p0 + tid / 4, P - 1);
        const float e = exact_at(phys_of(pg));
        if (u == 0 && p0 + tid / 4 < P) row[pg] = e;
      }
      __syncthreads();
      const RowView<false> rv{row, 1, p.score_stride};
      topk_select_body<false>(rv, P, kk, p.k, out_pages, out_scores, pool, bits);
      __syncthreads();
      continue;
    }
    // RUNS: every candidate takes its exact score where one round of scores is enough for all, and where the pages crowd (most are close
    // then: 300 pages of one score, 256 lists, bounds included, 72 us by bounds, 55 so); a list per head stays in the same code (beside
    // the other way's it takes 1.1 us longer in a step with 256 lists), a pooled one, whose scores take longer, takes the other way's.
    const bool all_exact = !RUNS || ncand <= kSelThreads / 4 || crowded;
    if (RUNS && (!POOLED || !all_exact)) {
      // The candidates in descending order of their lower bounds.  No pair of bounds is wider than `width`: where a lower bound
      // lies more than that below the one before it, everything from there on scores below everything before.  Only within a run
      // of closer ones does the order need exact scores: 20 of 67 candidates at 64 pages per list (see refine_runs).
      constexpr int kPer = kSelThreads / 4;
      const bool every = !POOLED && all_exact;
      const unsigned long long* by_bound = every ? ckey : sm.r.skey;
      unsigned long long* exact = every ? sm.r.skey : ckey;
      int nclose = ncand;
      if (!every) {
        const uint32_t wide = __reduce_max_sync(0xffffffffu, __float_as_uint(width));        // (not negative: ordered like its bits)
        if (lane == 0) atomicMax(&sm.r.width, wide);
#pragma unroll 1
        for (int i = tid; (i & ~31) < ncand; i += kSelThreads) {    // (whole warps without a candidate skip the count)
          const unsigned long long mine = i < ncand ? ckey[i] : ~0ull;
          const int rank = larger_keys(ckey, ncand, mine);
          if (i < ncand) sm.r.skey[rank] = mine;
        }
        __syncthreads();
        width = __uint_as_float(sm.r.width);
        for (int r0 = warp * 32; r0 < ncand; r0 += kSelThreads) {
          const int r = r0 + lane;
          auto lower = [&](int i) { return unorder_bits(static_cast<uint32_t>(by_bound[i] >> 32)); };
          auto starts = [&](int i) { return i == 0 || lower(i - 1) > __fadd_ru(lower(i), width); };
          const bool in = r < ncand, first = in && starts(r), last = in && (r + 1 == ncand || starts(r + 1));
          const bool open = in && !(first && last);
          const uint32_t runs = __ballot_sync(0xffffffffu, first), opens = __ballot_sync(0xffffffffu, open);
          int at = 0;
          if (lane == 0) {
            sm.r.run[r0 / 32] = runs;
            if (opens) at = atomicAdd(&sm.r.nclose, __popc(opens));
          }
          at = __shfl_sync(0xffffffffu, at, 0) + __popc(opens & ((1u << lane) - 1u));
          if (open) sm.r.close[at] = static_cast<uint16_t>(r);
        }
        __syncthreads();
        nclose = sm.r.nclose;
      }
      auto position = [&](int i) { return every ? i : static_cast<int>(sm.r.close[i]); };
      auto page_at = [&](int r) { return static_cast<int>(~reinterpret_cast<const uint32_t*>(by_bound)[2 * r]); };     // (a key's low word)
      int r_next = 0, pg_next = 0, ph_next = 0;
      if (nclose > 0) {
        r_next = position(min(tid / 4, nclose - 1));
        pg_next = page_at(r_next);
        ph_next = phys_of(pg_next);
      }
#pragma unroll 1
      for (int i = tid / 4; i - tid / 4 < nclose; i += kPer) {      // uniform over the CTA
        const int r = r_next, pg = pg_next, ph = ph_next;
        if (i - tid / 4 + kPer < nclose) {                  // (the next round's pages are looked up beside this one's scores)
          r_next = position(min(i + kPer, nclose - 1));
          pg_next = page_at(r_next);
          ph_next = phys_of(pg_next);
        }
        const float e = exact_at(ph);
        if (u == 0 && i < nclose) exact[r] = make_key(order_bits(e), pg);
      }
      __syncthreads();
      // ---- a candidate's position: its run's, and the number of larger keys in the run (all differ); emit the first kk
      for (int r = tid; r < ncand; r += kSelThreads) {
        unsigned long long mine;
        int rank;
        if (every) {
          mine = exact[r];
          rank = larger_keys(exact, ncand, mine);
        } else {
          int w = r >> 5, end = ncand;
          uint32_t b = sm.r.run[w] & (0xffffffffu >> (31 - (r & 31)));
          while (b == 0u) b = sm.r.run[--w];
          const int start = w * 32 + 31 - __clz(b);
          if (start >= kk) continue;
          w = r >> 5;
          b = sm.r.run[w] & (0xfffffffeu << (r & 31));
          const int nw = (ncand + 31) >> 5;
          while (b == 0u && ++w < nw) b = sm.r.run[w];
          if (b) end = w * 32 + __ffs(b) - 1;
          mine = by_bound[r];
          rank = start;
          if (end - start > 1) {
            mine = exact[r];
            for (int i = start; i < end; ++i) rank += exact[i] > mine ? 1 : 0;
          }
        }
        if (rank < kk) emit(rank, mine);
      }
      for (int gi = 0; gi < pool; ++gi)
        for (int j = kk + tid; j < p.k; j += kSelThreads) out_pages[gi * p.k + j] = -1;
    } else {
      // a group of four lanes per candidate, 32 candidates per round, all physical page ids in one round trip
      // (through shared memory: with four rounds' ids in registers the loop was unrolled, spilled, and a whole step
      // took 1 us longer with one 8K sequence, 2 us with eight of 32K)
      int* cphys = sm.r.cphys;
      for (int i = tid; i < ncand; i += kSelThreads) {
        if (RUNS) cpage[i] = static_cast<int>(~static_cast<uint32_t>(ckey[i]));
        cphys[i] = phys_of(cpage[i]);
      }
      __syncthreads();
      constexpr int kPer = kSelThreads / 4;
#pragma unroll 1
      for (int i0 = 0; i0 < ncand; i0 += kPer) {           // uniform over the CTA
        const int i = i0 + tid / 4, ic = min(i, ncand - 1);
        const float e = exact_at(cphys[ic]);
        if (u == 0 && i < ncand) ckey[i] = make_key(order_bits(e), cpage[i]);
      }
      // ---- order the candidates (descending) and emit the first kk
      __syncthreads();
      if (ncand <= kSelThreads) {
        // few candidates (the usual case): a candidate's position is the number of larger keys
        if ((tid & ~31) < ncand) {                       // whole warps without a candidate skip the count
          const unsigned long long mine = tid < ncand ? ckey[tid] : ~0ull;
          const int rank = larger_keys(ckey, ncand, mine);
          if (tid < ncand && rank < kk) emit(rank, mine);
        }
        for (int gi = 0; gi < pool; ++gi)
          for (int j = kk + tid; j < p.k; j += kSelThreads) out_pages[gi * p.k + j] = -1;
      } else {
        int n2 = 2;
        while (n2 < ncand) n2 <<= 1;
        for (int i = ncand + tid; i < n2; i += kSelThreads) ckey[i] = 0ull;
        __syncthreads();
        for (int k2 = 2; k2 <= n2; k2 <<= 1) {
          for (int j = k2 >> 1; j > 0; j >>= 1) {
            for (int t = tid; t < (n2 >> 1); t += kSelThreads) {
              const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1));
              const int x = i | j;
              const unsigned long long ka = ckey[i], kb = ckey[x];
              if ((ka < kb) == ((i & k2) == 0)) { ckey[i] = kb; ckey[x] = ka; }
            }
            __syncthreads();
          }
        }
        for (int gi = 0; gi < pool; ++gi) {
          for (int j = tid; j < p.k; j += kSelThreads) {
            if (j < kk) {
              const unsigned long long key = ckey[j];
              out_pages[gi * p.k + j] = static_cast<int32_t>(0xffffffffu - static_cast<uint32_t>(key));
              if (out_scores) out_scores[gi * p.k + j] = unorder_bits(static_cast<uint32_t>(key >> 32));
              if (gi == 0) mark(static_cast<int32_t>(0xffffffffu - static_cast<uint32_t>(key)));
            } else {
              out_pages[gi * p.k + j] = -1;
            }
          }
        }
      }
    }
    __syncthreads();                               // the shared state is reused by the next slot
  }
  if (!bits) return;
  // ---- stage 3: the last CTA of this (sequence, KV head) writes the union
  __syncthreads();                                 // every thread's marks precede ...
  if (tid == 0) {                                  // ... this thread's ticket, a release of all of them (cumulative)
    // CTAs of this (sequence, KV head) that hold a slot: all of them arrive here
    const unsigned int n_grp = static_cast<unsigned int>((p.Hq / p.Hkv / pool) * min(na, p.slots));
    s_bstar = atomic_inc_acq_rel(&p.union_tickets[s * p.Hkv + kh], n_grp - 1) == n_grp - 1 ? 1 : 0;
  }
  __syncthreads();
  if (!s_bstar) return;
  uint32_t* bm = reinterpret_cast<uint32_t*>(hist);
  for (int w = tid; w < p.W; w += kSelThreads) {
    bm[w] = atomicExch(bits + w, 0u);              // the marks were made in L2; all zero again for the next launch
  }
  __syncthreads();
  union_emit<kSelThreads>(bm, p.W, p.Pmax, p.union_pages + (static_cast<size_t>(s) * p.Hkv + kh) * p.Pmax,
                          p.union_count + s * p.Hkv + kh, reinterpret_cast<int*>(s_red[0]));
}

template <bool POOLED>
__global__ void __launch_bounds__(kSelThreads)
topk_select_kernel(float* __restrict__ scores, const int32_t* __restrict__ kv_len,
                   const int32_t* __restrict__ active_idx, const int32_t* __restrict__ n_active,
                   const int32_t* __restrict__ step, int32_t* __restrict__ topk_pages,
                   float* __restrict__ topk_scores, int N, int B, int Hq, int g, int k, int Pmax, int score_stride, int pool,
                   uint32_t* __restrict__ union_bits, int G, int W, int32_t* __restrict__ status) {
  grid_dep_trigger();
  grid_dep_wait();
  // A CTA serves the active slots a = j, j + kSelSlots, ... of one (sequence, head): launching a CTA
  // costs about as much as an idle CTA's whole life, and most of the B slots are idle on most steps.
  // pool > 1 (pooled selector): one list per KV head from the maximum of its `pool` heads' rows
  const int qid = blockIdx.x, Hl = Hq / pool;
  const int h = (qid % Hl) * pool, s = (qid / Hl) % N, j = qid / (Hl * N);
  // fp32 whole step: the chosen pages go into the bitmap of the KV head's list, from which stage 4 takes the union (all
  // zero at the start; on the first step of a block the whole prefix)
  uint32_t* bits = union_bits ? union_bits + (static_cast<size_t>(s) * (Hq / G) + h / G) * W : nullptr;
  if (step && step[s] == 0) {
    if (bits && j == 0 && h % G == 0) {
      const int P0 = min(pages_of(kv_len[s], g), Pmax);
      for (int w = threadIdx.x; w < W; w += kSelThreads) bits[w] = prefix_word(w, P0);
    }
    return;
  }
  int na = n_active[s];
  na = na > B ? B : na;
  int P = pages_of(kv_len[s], g);
  if (P > Pmax) { if (threadIdx.x == 0) set_status(status, LOSA_ERR_BOUNDS); P = Pmax; }
  const int kk = min(k, P);
  for (int a = j; a < na; a += kSelSlots) {
    const int tok = active_idx[s * B + a];
    if (tok < 0 || tok >= B) { if (threadIdx.x == 0) set_status(status, LOSA_ERR_BOUNDS); continue; }
    RowView<POOLED> row{scores + ((static_cast<size_t>(s) * B + a) * Hq + h) * score_stride, pool, score_stride};
    const size_t o = ((static_cast<size_t>(s) * B + tok) * Hq + h) * k;
    if (P <= kSelThreads * kSelPerThread) {
      topk_select_body<true>(row, P, kk, k, topk_pages + o, topk_scores ? topk_scores + o : nullptr, pool, bits);
    } else {
      if (POOLED && pool > 1) {
        // the selection reads the row several times: pool once, into the group's first row (the
        // score rows are scratch and this CTA is the only reader of these)
        float* first = scores + ((static_cast<size_t>(s) * B + a) * Hq + h) * score_stride;
        constexpr int U = 4;                                   // pages per thread whose loads are in flight together
        for (int p0 = threadIdx.x; p0 < P; p0 += kSelThreads * U) {
          float v[U];
#pragma unroll
          for (int u = 0; u < U; ++u) v[u] = p0 + u * kSelThreads < P ? row[p0 + u * kSelThreads] : 0.f;
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (p0 + u * kSelThreads < P) first[p0 + u * kSelThreads] = v[u];
        }
        __syncthreads();
        row.g = 1;
      }
      topk_select_body<false>(row, P, kk, k, topk_pages + o, topk_scores ? topk_scores + o : nullptr, pool, bits);
    }
    __syncthreads();                                 // the shared state is reused by the next slot
  }
}

__global__ void __launch_bounds__(kThreads)
union_kernel(const int32_t* __restrict__ topk_pages, const int32_t* __restrict__ active_idx,
             const int32_t* __restrict__ n_active, const int32_t* __restrict__ kv_len,
             const int32_t* __restrict__ step, int32_t* __restrict__ union_pages,
             int32_t* __restrict__ union_count, int B, int Hq, int Hkv, int g, int k, int Pmax,
             int32_t* __restrict__ status) {
  grid_dep_trigger();                              // the stage-4 kernel sets up its barriers and tensor memory meanwhile
  grid_dep_wait();
  extern __shared__ uint32_t bitmap[];
  __shared__ int s_warp[kThreads / 32];
  const int kh = blockIdx.x, s = blockIdx.y, tid = threadIdx.x;
  const int P = min(pages_of(kv_len[s], g), Pmax);
  const int W = (Pmax + 31) / 32;
  const int G = Hq / Hkv;
  const bool all = step && step[s] == 0;
  for (int w = tid; w < W; w += kThreads) {
    bitmap[w] = all ? prefix_word(w, P) : 0u;
  }
  __syncthreads();
  if (!all) {
    int na = n_active[s];
    na = na < 0 ? 0 : (na > B ? B : na);
    const int per_tok = G * k;
    // two dependent reads per entry (block position of the active slot, then the list entry): the
    // positions are staged once, and the list entries are requested four at a time
    __shared__ int s_tok[LOSA_MAX_BLOCK];
    for (int a = tid; a < na; a += kThreads) s_tok[a] = active_idx[s * B + a];
    __syncthreads();
    constexpr int U = 4;
    const int total = na * per_tok;
    for (int base = tid; base < total; base += kThreads * U) {
      int pv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int idx = base + u * kThreads;
        pv[u] = -1;
        if (idx < total) {
          const int a = idx / per_tok, rem = idx % per_tok, gi = rem / k, j = rem % k;
          const int tok = s_tok[a];
          if (tok < 0 || tok >= B) { set_status(status, LOSA_ERR_BOUNDS); continue; }
          pv[u] = topk_pages[((static_cast<size_t>(s) * B + tok) * Hq + kh * G + gi) * k + j];
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int p = pv[u];
        if (p < 0) continue;
        if (p >= P) { set_status(status, LOSA_ERR_BOUNDS); continue; }
        atomicOr(&bitmap[p >> 5], 1u << (p & 31));
      }
    }
    __syncthreads();
  }
  union_emit<kThreads>(bitmap, W, Pmax, union_pages + (static_cast<size_t>(s) * Hkv + kh) * Pmax,
                       union_count + s * Hkv + kh, s_warp);
}

int pow2_at_least(int x) {
  int n = 2;
  while (n < x) n <<= 1;
  return n;
}

}  // namespace

int32_t topk_max_sortable(const losa_ctx* c) {
  int n = 2;
  while (static_cast<size_t>(n) * 2 * sizeof(unsigned long long) <= static_cast<size_t>(c->max_smem_optin)) n <<= 1;
  return n;
}

// CTAs of the refinement per list, i.e. (sequence, head) or (sequence, KV head): the fewest from three up that
// fill at least five sixths of the waves they take, else eight; no more than block tokens.  Most slots are idle
// on most steps, and an idle CTA costs its dispatch; on steps with many active tokens a last wave that is
// nearly empty doubles the time.  Whole step, us, at 3 / 8 / 32 active tokens (888 resident CTAs):
//   256 lists (8 x 32K tokens)  3 CTAs 107 / 163 / 364, 4 CTAs (1.15 waves) 108 / 176 / 405, 8 CTAs 111 / 171 / 370
//   512 lists (16 x 8K)         3 CTAs 130 / 178 / 362, 2 CTAs (1.15 waves) 128 / 190 / 416, 8 CTAs 134 / 182 / 353
//   128 lists (4 x 24K)         6 CTAs 63 / 87 / 172, 7 CTAs (1.01 waves) 64 / 92 / 184, 3 CTAs 64 / 94 / 198
int refine_slots(int lists, int resident, int block_size) {
  int slots = kSelSlots;
  for (int n = kSelSlots - 1; n >= 3; --n) {
    const int ctas = n * lists, waves = (ctas + resident - 1) / resident;
    if (6 * ctas >= 5 * waves * resident) slots = n;
  }
  return std::min(slots, block_size);
}

// Exact scores only where the bounds leave the order open (RUNS), or for every candidate.  The former saves two rounds of
// gathers out of three at 64 pages per list (eight 32K prompts: 29 MB of summaries out of L2, 4.6 us of a list's 11.7; 20 of 67
// candidates are close) and costs a sort on the bounds.  It pays where many lists share L2's bandwidth, or a score is the largest of a
// group's and more than two rounds of scores are saved.  Not where the scores are asked for: all candidates need them then.
// Whole step, us, without and with it, at 48 / 64 / 100 / 128 pages per list:
//   256 lists (8 x 32K tokens)             95.1 / 106.1 / 125.8 / 143.1,  93.5 / 103.2 / 122.9 / 137.7
//   128 lists (4 x 24K)                    58.0 / 62.3 / 71.1 / 79.9,  57.5 / 61.5 / 69.8 / 76.9
//   128 lists (4 x 64K)                    70.1 / 76.8 / 92.2 / 103.9,  70.0 / 76.4 / 91.2 / 101.0
//   96 lists (3 x 32K)                     52.3 / 56.3 / 64.1 / 71.8,  51.8 / 55.2 / 63.8 / 69.8
//   32 lists (1 x 32K)                     37.5 / 39.0 / 42.5 / 47.1,  38.8 / 39.9 / 43.2 / 46.4
//   8 pooled lists (8K)                    36.0 / 37.6 / 40.3 / 45.6,  36.4 / 36.4 / 39.6 / 41.4
//   8 pooled lists (64K)                   42.9 / 45.5 / 48.7 / 55.4,  43.2 / 45.5 / 49.0 / 53.2
//   64 pooled lists (8 x 16K, 8 active)    87.2 / 96.1 / 110.0 / 123.0,  85.7 / 92.1 / 105.5 / 114.6
bool refine_runs(int lists, int pool, int k) { return pool > 1 ? k >= 60 : k >= 48 && lists >= 128; }

bool selects_by_refinement(const losa_ctx* c, int32_t k, int selector) {
  return c->shape.dtype == LOSA_BF16 && (selector == kSelectorExact || selector == kSelectorPooled) && k <= kSelCap &&
         c->shape.max_pages_per_seq > 0;
}

int32_t launch_page_scores_topk(losa_ctx* c, const void* q, const losa_kv_t* kv,
                                const int32_t* active_idx, const int32_t* n_active,
                                const int32_t* step, int32_t k, int32_t* topk_pages,
                                float* topk_scores_opt, cudaStream_t st, int selector, bool after_stage1,
                                int32_t* union_pages, int32_t* union_count, bool* union_done, const BlockInputs* blk) {
  if (union_done) *union_done = false;
  const losa_shape_t& sh = c->shape;
  if (sh.max_pages_per_seq == 0) return LOSA_OK;
  const bool pooled = selector == kSelectorPooled;
  const int pool = pooled ? sh.n_q_heads / sh.n_kv_heads : 1;
  if (selects_by_refinement(c, k, selector)) {
    // bf16, exact lists (per query head, or per KV head from the group's maximum): bounds from the
    // tensor cores, exact scores for the candidates only
    const bool pool_bounds = pooled && bounds_can_pool(c);
    int32_t rc = launch_page_bounds(c, q, kv, active_idx, n_active, step, st, false, after_stage1, pool_bounds);
    if (rc != LOSA_OK) return rc;
    RefineParams rp;
    rp.bounds = reinterpret_cast<float2*>(c->ws + c->lay.scores);
    rp.q = static_cast<const __nv_bfloat16*>(q);
    rp.kmin = static_cast<const __nv_bfloat16*>(kv->kmin);
    rp.kmax = static_cast<const __nv_bfloat16*>(kv->kmax);
    rp.page_table = kv->page_table;
    rp.kv_len = kv->kv_len;
    rp.active_idx = active_idx;
    rp.n_active = n_active;
    rp.step = step;
    rp.topk_pages = topk_pages;
    rp.topk_scores = topk_scores_opt;
    rp.status = status_ptr(c);
    rp.N = sh.batch; rp.B = sh.block_size; rp.Hq = sh.n_q_heads; rp.Hkv = sh.n_kv_heads; rp.g = sh.page_size;
    rp.k = k; rp.score_stride = c->lay.score_stride; rp.Pmax = sh.max_pages_per_seq; rp.n_phys = kv->n_phys_pages;
    rp.W = (sh.max_pages_per_seq + 31) / 32;
    const bool with_union = union_pages && union_count && union_done && rp.W <= kSelBins;
    rp.union_bits = with_union ? reinterpret_cast<uint32_t*>(c->ws + c->lay.union_bits) : nullptr;
    rp.bound_rows = pool_bounds ? 1 : pool;
    rp.union_tickets = reinterpret_cast<unsigned int*>(c->ws + c->lay.union_tickets);
    rp.union_pages = union_pages;
    rp.union_count = union_count;
    if (with_union) *union_done = true;
    const int lists = sh.batch * (sh.n_q_heads / pool);
    // As a call of its own (six-call path) the kernel has nothing beside or behind it: eight CTAs per list, and the
    // driver's shared-memory / L1 split, under which the summaries that a list's queries share are found in
    // L1 (eight 32K prompts, 32 active tokens: 188 us with bounds, 200 with a step's CTAs and split; three: 28.4 and 29.2).
    const bool in_step = blk != nullptr;
    rp.slots = in_step ? refine_slots(lists, c->n_sms * (pool > 1 ? 4 : 6), sh.block_size) : std::min(kSelSlots, sh.block_size);
    rp.blk_tiles = block_attn_tiles(sh);
    const bool with_block = blk && blk->q;
    const BlockAttnParams bp = with_block ? block_attn_params(c, blk->q, blk->k_blk, blk->v_blk) : BlockAttnParams{};
    const int grid = lists * rp.slots + (with_block ? rp.blk_tiles * sh.n_kv_heads * sh.batch : 0);
    with_block_attn_shape(sh, [&](auto d, auto bk) {
      constexpr int D = decltype(d)::value, BK = decltype(bk)::value;
      const int split = in_step ? cudaSharedmemCarveoutMaxShared : cudaSharedmemCarveoutDefault;
      auto launch = [&](auto kernel) { launch_split(split, kernel, grid, kSelThreads, 0, st, rp, bp); };
      const bool runs = refine_runs(lists, pool, k) && !topk_scores_opt;
      if (pool > 1) launch(runs ? topk_refine_kernel<D, true, BK, true> : topk_refine_kernel<D, true, BK, false>);
      else launch(runs ? topk_refine_kernel<D, false, BK, true> : topk_refine_kernel<D, false, BK, false>);
    });
    return after_launch(c);
  }
  int32_t rc = selector == kSelectorMma ? launch_page_bounds(c, q, kv, active_idx, n_active, step, st, true, after_stage1)
                                        : launch_page_scores(c, q, kv, active_idx, n_active, step, st, after_stage1);
  if (rc != LOSA_OK) return rc;

  float* sc = reinterpret_cast<float*>(c->ws + c->lay.scores);
  if (k <= kSelCap) {
    uint32_t* bits = union_pages && union_done && union_from_bits(c, k) ? reinterpret_cast<uint32_t*>(c->ws + c->lay.union_bits) : nullptr;
    const int G = sh.n_q_heads / sh.n_kv_heads;
    if (bits) *union_done = true;
    const int queries = sh.batch * std::min<int>(sh.block_size, kSelSlots) * (sh.n_q_heads / pool);
    if (pool > 1)
      launch_k(topk_select_kernel<true>, queries, kSelThreads, 0, st,
          sc, kv->kv_len, active_idx, n_active, step, topk_pages, topk_scores_opt, sh.batch, sh.block_size,
          sh.n_q_heads, sh.page_size, k, sh.max_pages_per_seq, c->lay.score_stride, pool, bits, G, union_words(c), status_ptr(c));
    else
      launch_k(topk_select_kernel<false>, queries, kSelThreads, 0, st,
          sc, kv->kv_len, active_idx, n_active, step, topk_pages, topk_scores_opt, sh.batch, sh.block_size,
          sh.n_q_heads, sh.page_size, k, sh.max_pages_per_seq, c->lay.score_stride, 1, bits, G, union_words(c), status_ptr(c));
    return after_launch(c);
  }
  // budgets beyond what one warp can sort: whole-list bitonic sort, one CTA per query
  const size_t smem = static_cast<size_t>(pow2_at_least(sh.max_pages_per_seq)) * sizeof(unsigned long long);
  if (smem > 48 * 1024)               // (the most that any context asks for: the attribute is shared by all of them)
    LOSA_CUDA_TRY(c, cudaFuncSetAttribute(topk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          topk_max_sortable(c) * static_cast<int>(sizeof(unsigned long long))));
  dim3 grid(sh.n_q_heads / pool, sh.block_size, sh.batch);
  launch_k(topk_kernel, grid, kThreads, smem, st, sc, kv->kv_len, active_idx, n_active, step, topk_pages,
                                            topk_scores_opt, sh.block_size, sh.n_q_heads, sh.page_size,
                                            k, sh.max_pages_per_seq, c->lay.score_stride, pool, status_ptr(c));
  return after_launch(c);
}

int32_t launch_page_union(losa_ctx* c, const int32_t* topk_pages, const int32_t* active_idx,
                          const int32_t* n_active, int32_t k, const int32_t* kv_len,
                          const int32_t* step, int32_t* union_pages, int32_t* union_count,
                          cudaStream_t st) {
  const losa_shape_t& sh = c->shape;
  const size_t smem = static_cast<size_t>((sh.max_pages_per_seq + 31) / 32 + 1) * sizeof(uint32_t);
  dim3 grid(sh.n_kv_heads, sh.batch);
  launch_k(union_kernel, grid, kThreads, smem, st, topk_pages, active_idx, n_active, kv_len, step, union_pages,
                                             union_count, sh.block_size, sh.n_q_heads, sh.n_kv_heads,
                                             sh.page_size, k, sh.max_pages_per_seq, status_ptr(c));
  return after_launch(c);
}

}  // namespace losa
