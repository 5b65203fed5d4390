// Stage 4, bf16, 5th-generation tensor cores: included by sparse_prefix_attn.cu (same namespace;
// the flat work decomposition, the partial-record format and the combine kernel are described there).
//
// A CTA owns up to 128 GQA-grouped query rows of one (sequence, KV head) at a time: the M = 128 rows
// of every MMA, one row per tensor-memory lane.  Pages are taken in groups of 128 tokens (PG pages):
//   S[128 x 128]  = Q . K^T      A = Q from tensor memory (bf16, written there once per piece),
//                                B = the group's K tiles, K-major in shared memory (128-byte swizzle,
//                                as TMA wrote them); D / 16 instructions
//   softmax       eight warps, thread = (query row, half of the columns): the row's scores are read
//                 from tensor memory once, the maximum is exchanged with the partner thread, then
//                 P = 2^(s - m); the reference maximum m only moves when it would grow by more than
//                 2^8 (then O is rescaled in place); P is rounded to bf16 and written over the
//                 scores it came from
//   O[128 x D]   += P . V        A = P from tensor memory, B = the group's V tiles as they lie in
//                                memory (tokens x d: MN-major); 8 instructions
// Issuing one tcgen05.mma costs the issuing thread ~120 cycles whatever its shape (measured), so the
// shapes are as large as the layout allows and the two products have an issuing thread each.
// K and V have a ring of group-sized slots each, filled by one producer warp each (lane = page:
// 32 pages' copies are issued by one instruction); a K slot is free again as soon as its Q K^T has
// run, a V slot after its P V.  S is double-buffered.  Completion is tracked with tcgen05.commit on
// mbarriers; every wait is bounded; tensor memory is returned on every path.
#pragma once

constexpr int kTc5SoftmaxWarps = 8;              // two sets of four: set h takes columns 64h .. 64h+63 of every group
constexpr int kTc5QkWarp = 8, kTc5PvWarp = 9, kTc5KWarp = 10, kTc5VWarp = 11;
constexpr int kTc5CvtWarp = 12;                  // FP8 pages: four converting warps, two for K and two for V
template <bool FP8> constexpr int tc5_threads() { return FP8 ? 512 : 384; }
constexpr int kTc5Tok = 128;                     // tokens per group = N of Q K^T = columns of one S buffer
constexpr float kTc5Tau = 8.0f;                  // reference maximum moves only when it would grow by more than this (log2 units)
constexpr int kTc5XchgBytes = (2 * 2 + 1) * kRowsPerGroup * 4;   // row maxima [group parity][set][row], row sums [row]
// FP8 pages: binary places by which P is held above the reference maximum.  P stays below 2^(8 + 7) < 65504.
constexpr float kTc5Fp8Lift = 7.0f;
constexpr int kTc5StgMax = 20;                   // FP8 pages: staging slots per tensor, one page each, at most
// FP8: value pages whose multiplier is kept.  Page x + 32 is issued once page x + 32 - 20 or a later one has
// been converted, and with it the whole group of page x (at most 8 pages).
constexpr int kTc5VmulRing = 32;
// Groups whose per-page data (token counts; FP8: scales) is kept.  The K producer writes a page's entry
// when it issues the page's copy, so the ring must be longer than its lead over the softmax warps.  A
// group never spans two segments, so in a run of one-page segments every page in flight is a group of
// its own.  The first page of group g is issued once its slot is free:
//   bf16  Q K^T of group g - NR has run, hence P V of group g - NR - 2: group g - NR - 1 may still be
//         read, a lead of NR + 1;
//   FP8   page, and so at worst group, g - NSP has been converted (NSP staging slots), hence Q K^T of
//         group g - NSP - NR has run: a lead of NSP + NR + 1.
// Small pages have up to 20 staging slots, a lead of 23; the others at most 10.
template <int D, int GP, bool FP8> constexpr int tc5_meta_ring() { return FP8 && GP * D <= 2048 ? 32 : 16; }
// Barriers, the segment prefix and index cache, the exchange arrays, the charged prefix, the staging
// barriers (landed, emptied; K and V) and the value pages' multipliers, two words per page of the meta ring
template <int D, int GP, bool FP8> constexpr int tc5_tail_bytes() {
  return kTailBytes + kTc5XchgBytes + (kMaxSegments + 2) * 4 + kTc5StgMax * 2 * (8 + 8) + kTc5VmulRing * 4 + tc5_meta_ring<D, GP, FP8>() * (kTc5Tok / GP) * 8;
}

template <int D> constexpr int tc5_slot_bytes() { return kTc5Tok * D * 2; }
template <int D, int GP, bool FP8> constexpr int tc5_ring_slots() {     // per ring (K and V have one each)
  if (FP8) return 2;                                            // the staging slots take the rest
  const int n = (kSmemBudget - 1024 - tc5_tail_bytes<D, GP, FP8>()) / tc5_slot_bytes<D>() / 2;
  return n > 6 ? 6 : n;
}
// FP8: pages per staging ring (one for K, one for V): what the ring slots leave, up to five groups
template <int D, int GP> constexpr int tc5_stg_slots() {
  const int fit = (kSmemBudget - 1024 - tc5_tail_bytes<D, GP, true>() - 4 * tc5_slot_bytes<D>()) / 2 / (GP * D), five = 5 * (kTc5Tok / GP);
  const int n = fit < five ? fit : five;
  return n < kTc5StgMax ? n : kTc5StgMax;
}
template <int D, int GP, bool FP8> constexpr int tc5_smem_bytes() {
  return 1024 + 2 * tc5_ring_slots<D, GP, FP8>() * tc5_slot_bytes<D>() + (FP8 ? 2 * tc5_stg_slots<D, GP>() * GP * D : 0) + tc5_tail_bytes<D, GP, FP8>();
}

// Shared-memory matrix descriptor: 128-byte swizzle, 8-row groups 1024 bytes apart; lbo = distance
// between 64-element blocks along the MN dimension of an MN-major operand.
__device__ __forceinline__ uint64_t tc5_desc(uint32_t saddr, uint32_t lbo) {
  return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16) |
         (static_cast<uint64_t>(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// Instruction descriptor, kind::f16: fp32 accumulate, A and B both bf16 (fmt 1) or both fp16 (fmt 0),
// M x N tile, B optionally MN-major.
__device__ __forceinline__ uint32_t tc5_idesc(int M, int N, int b_mn_major, uint32_t fmt = 1u) {
  return (1u << 4) | (fmt << 7) | (fmt << 10) | (static_cast<uint32_t>(b_mn_major) << 16) |
         (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}
// D[tmem] (+)= A[tmem] . B[smem descriptor]
__device__ __forceinline__ void tc5_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc5_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc5_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc5_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// tcgen05.ld of 32 consecutive 32-bit columns of this thread's lane; the wait is part of the same
// statement so that no use of the registers can be scheduled ahead of it.
__device__ __forceinline__ void tc5_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// The same load without the wait: several can be in flight; tc5_wait_ld() then tc5_pin32() on each
// destination before any use (the empty statement ties the registers to a point after the wait).
__device__ __forceinline__ void tc5_ld32_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc5_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc5_pin32(uint32_t* r) {
#pragma unroll
  for (int i = 0; i < 32; ++i) asm volatile("" : "+r"(r[i]) :: "memory");
}
__device__ __forceinline__ void tc5_st16(uint32_t taddr, const uint32_t* w) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(taddr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]), "r"(w[8]),
        "r"(w[9]), "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]), "r"(w[15])
      : "memory");
}
__device__ __forceinline__ void tc5_st32(uint32_t taddr, const uint32_t* w) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]), "r"(w[8]),
        "r"(w[9]), "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]), "r"(w[15]), "r"(w[16]), "r"(w[17]),
        "r"(w[18]), "r"(w[19]), "r"(w[20]), "r"(w[21]), "r"(w[22]), "r"(w[23]), "r"(w[24]), "r"(w[25]), "r"(w[26]),
        "r"(w[27]), "r"(w[28]), "r"(w[29]), "r"(w[30]), "r"(w[31])
      : "memory");
}
__device__ __forceinline__ void tc5_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// byte offset of 16-byte chunk c (0..7) of row t in a [rows][128 B] tile with the 128-byte swizzle
__device__ __forceinline__ uint32_t tc5_sw(int t, int c) { return static_cast<uint32_t>(t * 128 + ((c ^ (t & 7)) << 4)); }

// FP8: the K / V pools hold E4M3 bytes with one power-of-two scale per (page, KV head).  The page
// copies land in staging rings as they lie in memory (half the bytes); four converting warps, one
// per scheduler, turn a landed page's codes into fp16 (exact) in the group's ring slot, in the layout
// the tensor maps of the bf16 path produce, and every MMA runs on fp16 operands (Q and P are
// converted to fp16 instead of bf16).  The scales stay out of the conversion, which is bound by its
// instruction count: the key scale joins the softmax scale of the page's columns, and the value
// scale 2^e is added to their exponent, so that P' = p 2^e multiplies the codes of V and the row sum
// takes its columns back by 2^-e.  P' is rounded to fp16 relative to the largest p 2^e, so a page whose
// scale lies below another's would lose that many places of fp16's range.  Two things keep every
// weight at least as precise as an unscaled one: only the scales' part from 2^-6 to 2^0 goes into the
// exponent (pages of values up to 448; once a share has met a larger one, the converters go over each
// group of V a second time and multiply by the rest, exactly), and the reference lies 2^7 below the maximum.  A weight is then subnormal only 2^-15 or more
// below its row's largest, 2^-14 without scales.  A group is 2 x 16 KiB of codes:
// one warp needs about 3.8 us for 16 KiB, and while the two producing warps did this work it set the
// pace (eight 32K prompts: dense step 372 us, sparse step at three active tokens 120 us).  Now 224 and
// 81 us (scaling in the converters: 245 and 87; bit moves instead of the conversion instruction: 306
// and 105; no conversion at all: 207 and 77).  Staging slots are single pages, so that one is refilled
// while its neighbours are converted.  The
// CTA's 512 threads start with 128 registers each; the softmax warps take 168 and the other eight
// give theirs up to 88 (2 x 128 x 168 + 2 x 128 x 88 = 512 x 128).
template <int D, int GP, bool FP8>
__global__ void __launch_bounds__(tc5_threads<FP8>(), 1)
attn_tc5_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, AttnParams p) {
  constexpr int NR = tc5_ring_slots<D, GP, FP8>();  // slots per ring
  constexpr int NSP = FP8 ? tc5_stg_slots<D, GP>() : 1, STG = GP * D;   // FP8: staging slots per tensor, bytes of a slot (one page of codes)
  constexpr int NT = tc5_threads<FP8>();
  constexpr uint32_t FMT = FP8 ? 0u : 1u;       // operand format of the MMAs: fp16 / bf16
  constexpr int SLOT = tc5_slot_bytes<D>();
  constexpr int PG = kTc5Tok / GP;              // pages per group
  constexpr int MR = tc5_meta_ring<D, GP, FP8>();   // groups of the meta ring
  constexpr int HALVES = D / 64;                // 64-column (128-byte) blocks of a K or V row
  constexpr int HS = kTc5Tok * 128;             // bytes of one such block of a whole group
  constexpr int PAGE_BYTES = GP * D * 2;        // of K, and of V
  constexpr uint32_t COL_O = 0, COL_S = 128, COL_Q = 384;   // tensor-memory columns: O[D], S0[128], S1[128], Q[D/2]
  constexpr int TMEM_COLS = 512;
  static_assert(D == 64 || D == 128, "head dimensions of the tensor-core path");
  static_assert(GP == 16 || GP == 32 || GP == 64, "page sizes of the tensor-core path");
  static_assert(NR >= 2, "ring too shallow");
  static_assert(!FP8 || (NSP >= PG && NSP <= kTc5StgMax), "staging ring");
  static_assert((FP8 ? NSP : 0) + NR + 1 < MR, "the producer's lead fits the meta ring");
  static_assert(8 * (4 * 6 + 14) + 16 <= 512, "tail layout");

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - raw);
  const uint32_t kring = base, vring = base + NR * SLOT;
  constexpr int STG_ALL = FP8 ? 2 * NSP * STG : 0;
  const uint32_t kstg = base + 2 * NR * SLOT, vstg = kstg + NSP * STG;          // FP8 only
  uint8_t* tail = gen + 2 * NR * SLOT + STG_ALL;
  const uint32_t tail_s = base + 2 * NR * SLOT + STG_ALL;
  const uint32_t kfull = tail_s, kfree = kfull + 8 * NR, vfull = kfree + 8 * NR, vfree = vfull + 8 * NR;
  const uint32_t s_full = vfree + 8 * NR, s_free = s_full + 16, p_full = s_free + 16, q_full = p_full + 16, q_free = q_full + 8, xbar = q_free + 8;
  const uint32_t drain_bar = xbar + 32;            // two barriers: the issuing threads' last commit when the CTA gives up
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 8 * (4 * 6 + 14));
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(const_cast<int*>(abort_flag) + 1);
  int* pre = reinterpret_cast<int*>(tail + 512);
  int* tok_s = pre + kMaxSegments + 2;
  int* na_s = tok_s + kStageIdx;
  int* len_s = na_s + kStageSeq;
  float* xmax = reinterpret_cast<float*>(len_s + kStageSeq);   // [2][2][128]
  float* xsum = xmax + 4 * kRowsPerGroup;                        // [128]
  int* vpre = reinterpret_cast<int*>(xsum + kRowsPerGroup);      // prefix of the charged segment lengths (pages + pad)
  // FP8: per tensor, a staging slot's page has landed / has been converted
  const uint32_t stg_bars = smem_u32(vpre + kMaxSegments + 1) + 4;   // (kMaxSegments + 1 is odd)
  const uint32_t kstg_full = stg_bars, vstg_full = kstg_full + 8 * kTc5StgMax, kstg_free = vstg_full + 8 * kTc5StgMax, vstg_free = kstg_free + 8 * kTc5StgMax;
  // FP8: multipliers of the newest value pages' codes, as two fp16; whether any was other than one
  volatile uint32_t* vmul = reinterpret_cast<volatile uint32_t*>(vpre + kMaxSegments + 2 + 8 * kTc5StgMax);
  volatile int* vmul_used = abort_flag + 2;
  // per page of the groups in flight, [MR][PG]: valid tokens (FP8: and the exponent field of the value scale's part in P << 8), FP8: key scale
  volatile int* meta = vpre + kMaxSegments + 2 + 8 * kTc5StgMax + kTc5VmulRing;
  volatile float* kscale_meta = reinterpret_cast<volatile float*>(const_cast<int*>(meta) + MR * PG);
  const bool staged = p.N * p.B <= kStageIdx && p.N <= kStageSeq;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    for (int i = 0; i < NR; ++i) {
      mbar_init(kfull + 8 * i, FP8 ? 2 : 1);         // the copies' bytes / the two converting warps
      mbar_init(kfree + 8 * i, 1);
      mbar_init(vfull + 8 * i, FP8 ? 2 : 1);
      mbar_init(vfree + 8 * i, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(s_full + 8 * b, 1);                  // tcgen05.commit after Q K^T
      mbar_init(s_free + 8 * b, 1);                  // tcgen05.commit after P V: the S buffer is free and O holds the group
      mbar_init(p_full + 8 * b, kTc5SoftmaxWarps);
    }
    mbar_init(q_full, kTc5SoftmaxWarps);
    mbar_init(q_free, 1);
    for (int i = 0; i < 4; ++i) mbar_init(xbar + 8 * i, 2);      // the two softmax warps of a scheduler meet here
    mbar_init(drain_bar, 1);
    mbar_init(drain_bar + 8, 1);
    if (FP8)
      for (int i = 0; i < NSP; ++i) {
        mbar_init(kstg_full + 8 * i, 1);
        mbar_init(vstg_full + 8 * i, 1);
        mbar_init(kstg_free + 8 * i, 2);
        mbar_init(vstg_free + 8 * i, 2);
      }
    *abort_flag = 0;
    *vmul_used = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {                                 // tensor memory: taken while the previous kernel drains
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "n"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  grid_dep_trigger();
  grid_dep_wait();                                 // nothing above touches global memory
  if (warp == 0) {
    segment_prefix(pre, p.n_seg, p.n_rg, p.Hkv, p.G, p.n_active, [&](int sk) { return p.union_count[sk]; }, p.B, lane, vpre);
  } else if (staged) {
    for (int i = tid - 32; i < p.N * p.B; i += NT - 32) tok_s[i] = p.active_idx[i];
    for (int i = tid - 32; i < p.N; i += NT - 32) {
      na_s[i] = clamp_active(p.n_active[i], p.B);
      len_s[i] = p.kv_len[i];
    }
  }
  tc5_fence_before();
  __syncthreads();
  tc5_fence_after();
  const uint32_t tmem = *tmem_slot;
  // this CTA's share of the charged list, mapped back to pages: the first page at or after a charged position
  // (no share is empty: a segment's records are consecutive; rounding short shares up to whole groups of 128
  // tokens instead took 1.5 % off one case, 131,072 tokens, nothing off shorter lists, and P rounded relative to
  // a longer share's maximum was up to 1.8 % further from float64)
  const int V_all = vpre[p.n_seg], n_share = min(V_all, p.n_ctas);
  if (warp == kTc5PvWarp)                          // (this warp is needed last) for the merging kernels
    for (int seg = blockIdx.x * 32 + lane; seg < p.n_seg; seg += gridDim.x * 32) {
      const int n_pages = pre[seg + 1] - pre[seg], end = vpre[seg + 1];
      p.seg_records[seg] = segment_records(V_all, n_share, end - n_pages, end);
    }
  int lo = pre[p.n_seg], hi = lo, sg0 = 0;         // sg0: the segment of the share's first page, or one before it
  if (static_cast<int>(blockIdx.x) < n_share) {
    const int v_lo = cta_lo(V_all, blockIdx.x, n_share), v_hi = cta_lo(V_all, blockIdx.x + 1, n_share);
    int a = 0, b = p.n_seg, c = 0, d = p.n_seg;    // vpre[a] <= v_lo < vpre[b], vpre[c] <= v_hi (< vpre[d]): two searches side by side
    while (b - a > 1 || d - c > 1) {
      const int m0 = (a + b) >> 1, m1 = (c + d) >> 1;
      const int x0 = vpre[m0], x1 = vpre[m1];
      if (b - a > 1) { if (x0 <= v_lo) a = m0; else b = m0; }
      if (d - c > 1) { if (x1 <= v_hi) c = m1; else d = m1; }
    }
    auto page_at = [&](int a, int v) {             // the pages of a segment lie at the end of its charged run
      return pre[a] + max(0, v - vpre[a + 1] + (pre[a + 1] - pre[a]));
    };
    if (v_lo < V_all) { sg0 = a; lo = page_at(a, v_lo); }
    if (v_hi < V_all) hi = page_at(c, v_hi);
  }
  if (lo >= hi) {                                  // nothing to do: give the tensor memory back
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(TMEM_COLS) : "memory");
    return;
  }
  while (pre[sg0 + 1] <= lo) ++sg0;
  auto n_active_of = [&](int s) { return staged ? na_s[s] : clamp_active(p.n_active[s], p.B); };
  auto kv_len_of = [&](int s) { return staged ? len_s[s] : p.kv_len[s]; };
  auto token_of = [&](int s, int a) { return staged ? tok_s[s * p.B + a] : p.active_idx[s * p.B + a]; };

  int issued = -1;                                   // producer warps: newest group (FP8: page) whose copies have been issued
  if (warp >= kTc5SoftmaxWarps) {
  if constexpr (FP8) asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");    // whole warpgroups
  if (warp == kTc5KWarp || warp == kTc5VWarp) {
    // ------------------------------------------------------------------ producer warps: one for K, one for V
    // Lane j of a batch of 32 consecutive items resolves item -> logical page -> physical page (a
    // three-stage pipeline over batches, the two dependent loads of different batches in flight
    // together) and later issues that page's copies itself.  A piece's items are cut into groups of
    // PG pages; the first lane of a group's run waits for the group's ring slot and announces the
    // group's bytes, then every lane of the run issues its page.
    const bool is_v = warp == kTc5VWarp;
    const unsigned long long policy = l2_evict_first_policy();
    const CUtensorMap* map = is_v ? &tmV : &tmK;
    const uint32_t ring = is_v ? vring : kring, full0 = is_v ? vfull : kfull, free0 = is_v ? vfree : kfree;
    const uint32_t stg = is_v ? vstg : kstg, landed = is_v ? vstg_full : kstg_full, emptied = is_v ? vstg_free : kstg_free;
    int cursor = sg0, gbase = 0, pstart = lo;       // segment of the lane's newest item, groups before its piece, the piece's first item
    struct Item { int page, sk, grp, j, ng; };
    struct Ready { int phys, kh, valid, grp, j, ng; float ks, vs; };
    auto stage_a = [&](int i) {
      Item it{-1, 0, 0, 0, 0};
      if (i < hi) {
        while (pre[cursor + 1] <= i) {
          gbase += (pre[cursor + 1] - pstart + PG - 1) / PG;
          ++cursor;
          pstart = pre[cursor];
        }
        const int q = i - pstart, seg_end = min(hi, pre[cursor + 1]);
        it.sk = cursor;
        while (it.sk >= p.n_sk) it.sk -= p.n_sk;
        it.grp = gbase + q / PG;
        it.j = q % PG;
        it.ng = min(PG, seg_end - (i - it.j));
        it.page = ld_nc_s32(p.union_pages + static_cast<size_t>(it.sk) * p.Pmax + (i - pre[cursor]));
      }
      return it;
    };
    auto stage_b = [&](int i, const Item& it) {
      Ready r{0, 0, 0, it.grp, it.j, it.ng, 1.f, 1.f};
      if (i < hi) {
        const int s = it.sk / p.Hkv;
        r.kh = it.sk % p.Hkv;
        const bool ok = it.page >= 0 && it.page < p.Pmax;
        r.phys = ok ? ld_nc_s32(p.page_table + static_cast<size_t>(s) * p.Pmax + it.page) : -1;
        r.valid = ok ? min(GP, kv_len_of(s) - it.page * GP) : 0;
      }
      return r;
    };
    auto stage_c = [&](int i, Ready& r) {             // bounds; FP8: the page's scales (their address needs the physical page)
      if (i < hi) {
        if (r.phys < 0 || r.phys >= p.n_phys || r.valid <= 0) {
          set_status(p.status, LOSA_ERR_BOUNDS);
          r.phys = 0;
          r.valid = 0;
        }
        if (FP8) {
          if (!is_v) r.ks = __ldg(p.k_scale + static_cast<size_t>(r.phys) * p.Hkv + r.kh);
          r.vs = __ldg(p.v_scale + static_cast<size_t>(r.phys) * p.Hkv + r.kh);
        }
      }
    };
    // copies of the batch of items b0 .. b0 + 31 (one per lane); false when a wait has run out
    auto issue = [&](int b0, const Ready& b) {
      const int nb = min(32, hi - b0);
      if constexpr (FP8) {                            // page by page: every lane handles its own staging slot
        // the value scale: 2^-6 .. 2^0 of it go into P (as an exponent field), the rest onto the codes (also
        // what a caller's own scale has beside its power of two)
        const int e = (__float_as_int(b.vs) >> 23) & 0xff, in_p = min(max(e, 127 - 6), 127);
        const __half2 in_v = __float2half2_rn(b.vs * __int_as_float((254 - in_p) << 23));
        for (int pos = 0; pos < nb; ++pos) {
          int ok = 1;
          if (lane == pos) {
            const int x = b0 + pos - lo, slot = x % NSP, round = x / NSP;
            if (round > 0) ok = mbar_wait(emptied + 8 * slot, (round - 1) & 1, abort_flag, p.status, p.wait_cycles);
            if (ok) {
              if (is_v) {
                const uint32_t m2 = *reinterpret_cast<const uint32_t*>(&in_v);
                vmul[x % kTc5VmulRing] = m2;
                if (m2 != 0x3c003c00u) *vmul_used = 1;
              } else {
                const int at = (b.grp % MR) * PG + b.j;
                meta[at] = b.valid | in_p << 8;
                kscale_meta[at] = b.ks;
              }
              mbar_expect_tx(landed + 8 * slot, STG);
              tma_load_4d(stg + slot * STG, map, landed + 8 * slot, 0, 0, b.kh, b.phys, policy);
            }
          }
          if (__shfl_sync(0xffffffffu, ok, pos) == 0) return false;
          issued = b0 + pos - lo;
        }
        return true;
      }
      int pos = 0;
      while (pos < nb) {
        const int grp = __shfl_sync(0xffffffffu, b.grp, pos), j0 = __shfl_sync(0xffffffffu, b.j, pos);
        const int ng = __shfl_sync(0xffffffffu, b.ng, pos);
        const int cnt = min(ng - j0, nb - pos);
        const int slot = grp % NR, round = grp / NR;
        if (j0 == 0) {
          int ok = 1;
          if (lane == 0 && round > 0) ok = mbar_wait(free0 + 8 * slot, (round - 1) & 1, abort_flag, p.status, p.wait_cycles);
          if (__shfl_sync(0xffffffffu, ok, 0) == 0) return false;
        }
        const bool mine = lane >= pos && lane < pos + cnt;
        if (!is_v && mine) meta[(grp % MR) * PG + b.j] = b.valid;
        __syncwarp();
        if (j0 == 0 && lane == 0) mbar_expect_tx(full0 + 8 * slot, ng * PAGE_BYTES);
        __syncwarp();
        if (mine) {
          const uint32_t dst = ring + slot * SLOT + b.j * (GP * 128);
#pragma unroll
          for (int hf = 0; hf < HALVES; ++hf) tma_load_4d(dst + hf * HS, map, full0 + 8 * slot, hf * 64, 0, b.kh, b.phys, policy);
        }
        issued = grp;
        pos += cnt;
      }
      return true;
    };
    const Item a0 = stage_a(lo + lane);
    Item a = stage_a(lo + lane + 32);                 // requested beside the first batch: the first copies wait for two loads, not three
    Ready b = stage_b(lo + lane, a0);
    if constexpr (FP8) {                              // one stage deeper: the scales of a batch are requested a batch ahead
      stage_c(lo + lane, b);
      Ready b1 = stage_b(lo + lane + 32, a);
      a = stage_a(lo + lane + 64);
      bool go = true;
      for (int b0 = lo; b0 < hi && go; b0 += 32) {
        const Item a_next = stage_a(b0 + lane + 96);
        const Ready b2 = stage_b(b0 + lane + 64, a);
        stage_c(b0 + lane + 32, b1);
        go = issue(b0, b);
        a = a_next;
        b = b1;
        b1 = b2;
      }
    } else {
      bool go = true;
      for (int b0 = lo; b0 < hi && go; b0 += 32) {
        const Item a_next = stage_a(b0 + lane + 64);
        const Ready b_next = stage_b(b0 + lane + 32, a);
        stage_c(b0 + lane, b);
        go = issue(b0, b);
        a = a_next;
        b = b_next;
      }
    }
  } else if (FP8 && warp >= kTc5CvtWarp) {
    // ------------------------------------------------------------------ converting warps (FP8 pages)
    // Two warps per tensor, each half of every page's tokens.  A lane takes eight codes at a time (one
    // 16-byte chunk of fp16): 8-byte reads of consecutive codes and 16-byte stores of consecutive
    // swizzled chunks, both without bank conflicts; up to eight are requested before any is converted.
    const bool is_v = warp >= kTc5CvtWarp + 2;
    const int half = warp & 1;
    const uint8_t* stg_gen = gen + ((is_v ? vstg : kstg) - base);
    uint8_t* ring_gen = gen + ((is_v ? vring : kring) - base);
    const uint32_t landed = is_v ? vstg_full : kstg_full, emptied = is_v ? vstg_free : kstg_free;
    const uint32_t full0 = is_v ? vfull : kfull, free0 = is_v ? vfree : kfree;
    constexpr int CPR = D / 8, TPI = 32 / CPR;        // chunks of a row, tokens per warp access
    constexpr int NU = GP / 2 / TPI, U = NU < 8 ? NU : 8;   // accesses per page and warp, in flight
    const int tl = half * (GP / 2) + lane / CPR, c = lane % CPR;
    auto wait = [&](uint32_t bar, uint32_t parity) {
      int ok = 1;
      if (lane == 0) ok = mbar_wait(bar, parity, abort_flag, p.status, p.wait_cycles);
      ok = __shfl_sync(0xffffffffu, ok, 0);
      return ok != 0 && mbar_try_wait(bar, parity);   // (every lane observes the phase it was told of)
    };
    int sg = sg0, item = lo, g = 0;
    bool ok = true;
    while (item < hi && ok) {
      const int seg_end = min(hi, pre[sg + 1]);
      for (int first = item; first < seg_end && ok; first += PG, ++g) {
        const int ng = min(PG, seg_end - first), sr = g % NR;
        if (g >= NR) ok = wait(free0 + 8 * sr, (g / NR - 1) & 1);
        for (int pg = 0; pg < ng; ++pg) {
          const int x = first + pg - lo, ss = x % NSP;
          ok = ok && wait(landed + 8 * ss, (x / NSP) & 1);
          if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
          const uint8_t* src = stg_gen + ss * STG + tl * D + c * 8;
          uint8_t* dst = ring_gen + sr * SLOT + (c >> 3) * HS;
#pragma unroll
          for (int u0 = 0; u0 < NU; u0 += U) {
            uint2 w[U];
#pragma unroll
            for (int u = 0; u < U; ++u) w[u] = *reinterpret_cast<const uint2*>(src + (u0 + u) * TPI * D);
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const uint32_t x4[4] = {w[u].x & 0xffffu, w[u].x >> 16, w[u].y & 0xffffu, w[u].y >> 16};
              uint32_t h[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const __half2_raw v = __nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(x4[e]), __NV_E4M3);
                h[e] = *reinterpret_cast<const uint32_t*>(&v);
              }
              *reinterpret_cast<uint4*>(dst + tc5_sw(pg * GP + tl + (u0 + u) * TPI, c & 7)) = make_uint4(h[0], h[1], h[2], h[3]);
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(emptied + 8 * ss, 1);
        }
        if (!ok) break;
        if (is_v && *vmul_used) {                     // this lane's chunks once more, times what of the scales is not in P
#pragma unroll 1
          for (int i = 0; i < ng * NU; ++i) {
            const int pg = i / NU, u = i % NU;
            const uint32_t mul = vmul[(first + pg - lo) % kTc5VmulRing];
            const __half2 m2 = *reinterpret_cast<const __half2*>(&mul);
            uint4* at = reinterpret_cast<uint4*>(ring_gen + sr * SLOT + (c >> 3) * HS + tc5_sw(pg * GP + tl + u * TPI, c & 7));
            uint4 x = *at;
            auto scale = [&](uint32_t& y) {
              const __half2 v = __hmul2(*reinterpret_cast<const __half2*>(&y), m2);
              y = *reinterpret_cast<const uint32_t*>(&v);
            };
            scale(x.x); scale(x.y); scale(x.z); scale(x.w);
            *at = x;
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read the slot through the async proxy
        __syncwarp();
        if (lane == 0) mbar_arrive(full0 + 8 * sr, 1);
      }
      item = seg_end;
      ++sg;
      while (item < hi && pre[sg + 1] <= item) ++sg;
    }
  } else if (warp == kTc5QkWarp) {
    // ------------------------------------------------------------------ Q K^T issuer (one thread)
    if (lane == 0) {
      int sg = sg0, item = lo, piece = 0, g = 0;
      bool ok = true;
      while (item < hi && ok) {
        const int seg_end = min(hi, pre[sg + 1]);
        ok = mbar_wait(q_full, piece & 1, abort_flag, p.status, p.wait_cycles);
        for (int first = item; first < seg_end && ok; first += PG, ++g) {
          const int ng = min(PG, seg_end - first), b = g & 1, use = g >> 1, slot = g % NR;
          ok = mbar_wait(kfull + 8 * slot, (g / NR) & 1, abort_flag, p.status, p.wait_cycles);
          ok = ok && (use == 0 || mbar_wait(s_free + 8 * b, (use - 1) & 1, abort_flag, p.status, p.wait_cycles));
          if (!ok) break;
          tc5_fence_after();
          const uint32_t idesc = tc5_idesc(kRowsPerGroup, ng * GP, 0, FMT), kt = kring + slot * SLOT;
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks)
            tc5_mma_ts(tmem + COL_S + b * kTc5Tok, tmem + COL_Q + ks * 8, tc5_desc(kt + (ks >> 2) * HS + (ks & 3) * 32, 16),
                       idesc, ks > 0 ? 1u : 0u);
          tc5_commit(s_full + 8 * b);
          tc5_commit(kfree + 8 * slot);
          if (first + PG >= seg_end) tc5_commit(q_free);        // Q may be replaced once the piece's last product has run
        }
        item = seg_end;
        ++sg;
        ++piece;
        while (item < hi && pre[sg + 1] <= item) ++sg;
      }
    }
  } else if (warp == kTc5PvWarp) {
    // ------------------------------------------------------------------ P V issuer (one thread)
    if (lane == 0) {
      const uint32_t idesc = tc5_idesc(kRowsPerGroup, D, 1, FMT);
      int sg = sg0, item = lo, g = 0;
      bool ok = true;
      while (item < hi && ok) {
        const int seg_end = min(hi, pre[sg + 1]);
        for (int first = item; first < seg_end && ok; first += PG, ++g) {
          const int ng = min(PG, seg_end - first), b = g & 1, use = g >> 1, slot = g % NR;
          ok = mbar_wait(vfull + 8 * slot, (g / NR) & 1, abort_flag, p.status, p.wait_cycles);
          ok = ok && mbar_wait(p_full + 8 * b, use & 1, abort_flag, p.status, p.wait_cycles);
          if (!ok) break;
          tc5_fence_after();
          const uint32_t vt = vring + slot * SLOT;
          for (int ks = 0; ks < ng * GP / 16; ++ks)
            tc5_mma_ts(tmem + COL_O, tmem + COL_S + b * kTc5Tok + ks * 8, tc5_desc(vt + ks * 2048, HS), idesc,
                       (first == item && ks == 0) ? 0u : 1u);
          tc5_commit(vfree + 8 * slot);
          tc5_commit(s_free + 8 * b);
        }
        item = seg_end;
        ++sg;
        while (item < hi && pre[sg + 1] <= item) ++sg;
      }
    }
  }
  } else {
    // ------------------------------------------------------------------ softmax / epilogue warps
    if constexpr (FP8) asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
    // Thread = query row (tensor-memory lane 32 * (warp % 4) + lane) and one half of the columns:
    // set h = warp / 4 takes columns 64h .. 64h+63 of every group (and half of Q, of O when it is
    // rescaled or read out).  The exponentials are the bottleneck of this path (one special-function
    // unit per scheduler); two warps per scheduler keep that unit busy while the partner loads,
    // packs and stores.  The pair meets once per group (named barrier) to exchange the row maxima.
    const __nv_bfloat16* q = static_cast<const __nv_bfloat16*>(p.q);
    const int quarter = warp & 3, h = warp >> 2;
    const int r = quarter * 32 + lane;                         // row of the tile = tensor-memory lane
    const uint32_t lane_addr = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
    const float scale2 = p.sm_scale * kLog2e;
    constexpr int QW = D / 4;                                  // 32-bit words of Q per thread (half a row)
    constexpr int OC = D / 2;                                  // columns of O per thread
    // every wait of these warps ends with one answer for the whole warp: the tensor-memory
    // instructions that follow need all 32 lanes
    auto warp_wait = [&](uint32_t bar, uint32_t parity) {
      return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, p.status, p.wait_cycles)) != 0;
    };
    int n_meet = 0;
    auto pair_sync = [&]() {                                    // bounded like every other wait
      __syncwarp();
      if (lane == 0) mbar_arrive(xbar + 8 * quarter, 1);
      const bool met = warp_wait(xbar + 8 * quarter, n_meet & 1);
      ++n_meet;
      return met;
    };
    int sg = sg0, item = lo, piece = 0, g = 0;
    bool ok = true;
    while (item < hi && ok) {
      const int seg_end = min(hi, pre[sg + 1]);
      const int rg = sg / p.n_sk, sk = sg % p.n_sk, s = sk / p.Hkv, kh = sk % p.Hkv;
      const int rows = rows_in_group(n_active_of(s), p.G, rg);
      const bool warp_has_rows = quarter * 32 < rows;          // the same for both warps of a pair
      // ---- the piece's Q tile: this thread's half row, two bf16 per tensor-memory column
      {
        uint32_t qw[QW];
        const uint4* src = nullptr;
        if (r < rows) {
          const int row = rg * kRowsPerGroup + r, a = row / p.G, gi = row % p.G;
          int tok = token_of(s, a);
          if (tok < 0 || tok >= p.B) { set_status(p.status, LOSA_ERR_BOUNDS); tok = 0; }
          src = reinterpret_cast<const uint4*>(q + ((static_cast<size_t>(s) * p.B + tok) * p.Hq + kh * p.G + gi) * D) + h * (QW / 4);
        }
#pragma unroll
        for (int c = 0; c < QW / 4; ++c) {
          const uint4 v = src ? __ldg(src + c) : make_uint4(0u, 0u, 0u, 0u);
          qw[4 * c] = v.x; qw[4 * c + 1] = v.y; qw[4 * c + 2] = v.z; qw[4 * c + 3] = v.w;
        }
        if constexpr (FP8) {                        // the MMAs of this variant take fp16 operands
#pragma unroll
          for (int c = 0; c < QW; ++c) {
            const __half2 hq = __floats2half2_rn(__uint_as_float(qw[c] << 16), __uint_as_float(qw[c] & 0xffff0000u));
            qw[c] = *reinterpret_cast<const uint32_t*>(&hq);
          }
        }
        if (piece > 0) ok = warp_wait(q_free, (piece - 1) & 1);
        if (!ok) break;
        tc5_fence_after();
        if constexpr (QW == 32) tc5_st32(lane_addr + COL_Q + h * QW, qw);
        else tc5_st16(lane_addr + COL_Q + h * QW, qw);
        tc5_wait_st();
        tc5_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(q_full, 1);
      }
      float m_ref = -INFINITY, l = 0.f;                         // l: this thread's columns only
      bool o_valid = false;                                     // O holds at least one group of this piece
      for (int first = item; first < seg_end && ok; first += PG, ++g) {
        const int ng = min(PG, seg_end - first), ncol = ng * GP, b = g & 1, use = g >> 1;
        const uint32_t s_addr = lane_addr + COL_S + b * kTc5Tok;
        volatile int* gmeta = meta + (g % MR) * PG;
        auto valid_of = [&](int j) { return FP8 ? gmeta[j] & 0xff : gmeta[j]; };     // tokens of the group's page j
        ok = warp_wait(s_full + 8 * b, use & 1);
        if (!ok) break;
        tc5_fence_after();
        // pages with fewer than GP tokens (the last page of a prefix), or a group that ends inside a
        // 32-column chunk, need per-column masks; everything else takes the plain path
        bool ragged = (ncol & 31) != 0;
        for (int j = 0; j < ng; ++j) ragged |= valid_of(j) < GP;
        auto masked = [&](int col) {
          const int j = col / GP, t = col % GP;
          return j >= ng || t >= valid_of(j);
        };
        const int col0 = 64 * h;                                // this thread's columns: col0 .. col0+63, below ncol
        if (warp_has_rows) {
          // ---- the row's scores: one read of tensor memory into registers, both loads in flight together
          uint32_t sraw[64];
#pragma unroll
          for (int c = 0; c < 2; ++c)
            if (col0 + c * 32 < ncol) tc5_ld32_nowait(s_addr + col0 + 32 * c, sraw + 32 * c);
          tc5_wait_ld();
#pragma unroll
          for (int c = 0; c < 2; ++c)
            if (col0 + c * 32 < ncol) tc5_pin32(sraw + 32 * c);
          if (ragged) {
#pragma unroll
            for (int c = 0; c < 2; ++c)
              if (col0 + c * 32 < ncol) {
#pragma unroll
                for (int e = 0; e < 32; ++e) if (masked(col0 + 32 * c + e)) sraw[32 * c + e] = 0xff800000u;   // -inf
              }
          }
          // ---- pass 1: the row's maximum over the group (own columns, then the partner's)
          // (FP8: of the shifted exponents; NP page runs of PW columns per 32, each with its scales)
          constexpr int PW = (FP8 && GP == 16) ? 16 : 32, NP = 32 / PW;
          float kmul[2 * NP], vexp[2 * NP];
          if constexpr (FP8) {
#pragma unroll
            for (int x = 0; x < 2 * NP; ++x) {
              const int j = (col0 + x * PW) / GP;
              kmul[x] = j < ng ? scale2 * kscale_meta[(g % MR) * PG + j] : 1.f;
              vexp[x] = j < ng ? static_cast<float>((gmeta[j] >> 8) - 127) : 0.f;
            }
          }
          float mx_own = -INFINITY;
          float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int c = 0; c < 2; ++c)
            if (col0 + c * 32 < ncol) {
#pragma unroll
              for (int e = 0; e < 32; ++e) {
                mx[e & 3] = fmaxf(mx[e & 3], __uint_as_float(sraw[32 * c + e]));
                if (FP8 && (e + 1) % PW == 0) {
                  const int x = c * NP + e / PW;
                  mx_own = fmaxf(mx_own, fmaf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])), kmul[x], vexp[x]));
                  mx[0] = mx[1] = mx[2] = mx[3] = -INFINITY;
                }
              }
            }
          if (!FP8) mx_own = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
          xmax[(b * 2 + h) * kRowsPerGroup + r] = mx_own;
          ok = pair_sync();
          const float m_new = fmaxf(mx_own, xmax[(b * 2 + (h ^ 1)) * kRowsPerGroup + r]) * (FP8 ? 1.f : scale2);
          float corr = 1.f;
          constexpr float LIFT = FP8 ? kTc5Fp8Lift : 0.f;
          if (m_new > m_ref + (kTc5Tau + LIFT) || (m_ref == -INFINITY && m_new > -INFINITY)) {
            corr = (m_ref == -INFINITY) ? 0.f : ex2(m_ref - (m_new - LIFT));
            m_ref = m_new - LIFT;
            l *= corr;
          }
          // ---- rescale O (rare): the previous group's P V must have run; all lanes of the warp take
          //      part, each set on its half of the columns
          if (__any_sync(0xffffffffu, o_valid && corr != 1.f)) {
            ok = ok && warp_wait(s_free + 8 * ((g - 1) & 1), ((g - 1) >> 1) & 1);
            if (ok) {
              tc5_fence_after();
#pragma unroll
              for (int c0 = 0; c0 < OC; c0 += 32) {
                float t[32];
                uint32_t w[32];
                tc5_ld32(lane_addr + COL_O + h * OC + c0, t);
#pragma unroll
                for (int e = 0; e < 32; ++e) w[e] = __float_as_uint(t[e] * corr);
                tc5_st32(lane_addr + COL_O + h * OC + c0, w);
              }
              tc5_wait_st();
            }
          }
          // ---- pass 2: P = 2^(s - m) as bf16, written over the scores (column c of P takes the
          //      place of columns 2c, 2c+1 of S; every score of the group is in registers by now,
          //      the partner's too: it has passed the pair barrier)
          if (ok) {
            const float ms = (m_ref == -INFINITY) ? 0.f : m_ref;
            float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              if (col0 + c * 32 < ncol) {
                uint32_t w[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                  const int x = c * NP + 2 * e / PW;
                  const float mul = FP8 ? kmul[x] : scale2, add = FP8 ? vexp[x] - ms : -ms;
                  const float p0 = ex2(fmaf(__uint_as_float(sraw[32 * c + 2 * e]), mul, add));
                  const float p1 = ex2(fmaf(__uint_as_float(sraw[32 * c + 2 * e + 1]), mul, add));
                  sum[e & 3] += p0 + p1;
                  w[e] = FP8 ? pack_f16(p0, p1) : pack_bf16(p0, p1);
                  if (FP8 && (2 * e + 2) % PW == 0) {     // the page run's sum, without the value scale
                    l = fmaf((sum[0] + sum[1]) + (sum[2] + sum[3]), __int_as_float((127 - static_cast<int>(vexp[x])) << 23), l);
                    sum[0] = sum[1] = sum[2] = sum[3] = 0.f;
                  }
                }
                tc5_st16(s_addr + col0 / 2 + 16 * c, w);
              }
            }
            tc5_wait_st();
            if (!FP8) l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
          }
        }
        if (!ok) break;
        if (ragged) {
          // rows of V past the end of the prefix may hold anything (even NaN): clear them once the
          // tile has landed (all softmax warps, whether or not they own rows)
          bool any_short = false;
          for (int j = 0; j < ng; ++j) any_short |= valid_of(j) < GP;
          if (any_short) {
            const int slot = g % NR;
            ok = warp_wait(vfull + 8 * slot, (g / NR) & 1);
            if (!ok) break;
            uint8_t* vg = gen + (NR + slot) * SLOT;
            for (int j = 0; j < ng; ++j) {
              const int valid = valid_of(j);
              for (int idx = tid; idx < (GP - valid) * (D / 8); idx += kTc5SoftmaxWarps * 32) {
                const int t = j * GP + valid + idx / (D / 8), ch = idx % (D / 8);
                *reinterpret_cast<uint4*>(vg + (ch >> 3) * HS + tc5_sw(t, ch & 7)) = make_uint4(0u, 0u, 0u, 0u);
              }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          }
        }
        tc5_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(p_full + 8 * b, 1);
        o_valid = true;
      }
      if (!ok) break;
      // ---- the piece's record: one 16-row tile record per 16 rows, reference maximum in base-2
      //      units; each set writes its half of the columns, set 0 the row's maximum and sum
      ok = warp_wait(s_free + 8 * ((g - 1) & 1), ((g - 1) >> 1) & 1);
      if (!ok) break;
      tc5_fence_after();
      if (warp_has_rows) {
        if (h == 1) xsum[r] = l;
        ok = pair_sync();
        if (!ok) break;
        float* rec = record_base(p.partials, blockIdx.x + sg, r / kTileRows, D);
        const int rr = r % kTileRows;
#pragma unroll
        for (int c0 = 0; c0 < OC; c0 += 32) {
          float t[32];
          tc5_ld32(lane_addr + COL_O + h * OC + c0, t);
          if (r < rows) {
#pragma unroll
            for (int e = 0; e < 32; e += 4)
              *reinterpret_cast<float4*>(rec + 2 * kTileRows + rr * D + h * OC + c0 + e) = make_float4(t[e], t[e + 1], t[e + 2], t[e + 3]);
          }
        }
        if (h == 0 && r < rows) { rec[rr] = m_ref; rec[kTileRows + rr] = l + xsum[r]; }
      }
      tc5_fence_before();
      item = seg_end;
      ++sg;
      ++piece;
      while (item < hi && pre[sg + 1] <= item) ++sg;
    }
  }
  // ---- every thread that passed the allocation meets here; tensor memory is returned on all paths
  tc5_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // The CTA has given up (a wait ran out).  Its shared and tensor memory must not be handed on
    // while work it started is still in flight: the producers wait, within a bound, for the newest
    // round of copies of every ring slot (a group that was begun has had all its copies issued: the
    // producer loop only stops between groups), the issuing threads for the products they issued.
    if ((warp == kTc5KWarp || warp == kTc5VWarp) && lane == 0) {
      // (FP8 pages: the copies land in the staging slots)
      const uint32_t full0 = FP8 ? (warp == kTc5VWarp ? vstg_full : kstg_full) : (warp == kTc5VWarp ? vfull : kfull);
      constexpr int NSL = FP8 ? NSP : NR;
      for (int sl = 0; sl < NSL; ++sl) {
        if (issued < sl) continue;
        const int gl = issued - (issued - sl) % NSL;
        mbar_drain(full0 + 8 * sl, (gl / NSL) & 1);
      }
    }
    if ((warp == kTc5QkWarp || warp == kTc5PvWarp) && lane == 0) {
      const uint32_t bar = drain_bar + (warp == kTc5PvWarp ? 8 : 0);
      tc5_commit(bar);
      mbar_drain(bar, 0);
    }
    __syncthreads();
  }
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(TMEM_COLS) : "memory");
}
