// Stage 4, bf16, 5th-generation tensor cores: included by sparse_prefix_attn.cu (same namespace;
// the flat work decomposition, the partial-record format and the combine kernel are described there).
//
// A CTA owns up to 128 GQA-grouped query rows of one (sequence, KV head) at a time: the M = 128 rows
// of every MMA, one row per tensor-memory lane.  Pages are taken in groups of 128 tokens (PG pages):
//   S[128 x 128]  = Q . K^T      A = Q from shared memory (written there once per piece),
//                                B = the group's K tiles, K-major in shared memory (128-byte swizzle,
//                                as TMA wrote them); D / 16 instructions
//   softmax       three sets of four warps, thread = query row; the sets take every third group: the row's
//                 maximum in one pass, P = 2^(s - m) in a second, rounded to bf16 and written over the scores;
//                 the reference maximum m passes from group to group and only moves when it would grow by
//                 more than 2^8 (then O is rescaled in place)
//   O[128 x D]   += P . V        A = P from tensor memory, B = the group's V tiles as they lie in
//                                memory (tokens x d: MN-major); 8 instructions
// An instruction of either product takes the pipe 64 cycles (128 x 128 x 16); each product has an issuing
// warp of its own (one elected lane).  K and V have a ring of group-sized slots each, filled by one producer warp each
// (lane = page: 32 pages' copies are issued by one instruction); a K slot is free again as soon as its
// Q K^T has run, a V slot after its P V.  There is an S buffer per set (tensor memory: O 128 + 3 x 128
// columns; Q therefore lies in shared memory).  Completion is tracked with tcgen05.commit on mbarriers; every wait is
// bounded; tensor memory is returned on every path.
#pragma once

constexpr int kTc5Sets = 3, kTc5SetWarps = 4;    // sets of softmax warps: set h takes every third group, thread = one query row
constexpr int kTc5SoftmaxWarps = kTc5Sets * kTc5SetWarps;
constexpr int kTc5ScaleWarps = 2 * kTc5SetWarps; // FP8: softmax warps that look at the value scales before a share begins
constexpr int kTc5QkWarp = 12, kTc5PvWarp = 13, kTc5KWarp = 14, kTc5VWarp = 15;
constexpr int kTc5CvtWarp = 16, kTc5CvtWarps = 4; // FP8 pages: four warps that convert V
template <bool FP8> constexpr int tc5_threads() { return FP8 ? 640 : 512; }
// Registers per thread at the launch, and as they are dealt out to the softmax warps and the others:
// 12 x 32 x 136 + 4 x 32 x 104 = 512 x 128; FP8 12 x 32 x 112 + 8 x 32 x 72 = 640 x 96;
// with the narrow path in the kernel, whose producers would spill at 72 and are then late with every copy, 104 and 80 (one deal for
// both paths: with two in a kernel the compiler spills everywhere).
constexpr int kTc5LaunchRegs = 128, kTc5SoftmaxRegs = 136, kTc5OtherRegs = 104;
constexpr int kTc5LaunchRegs8 = 96, kTc5SoftmaxRegs8 = 112, kTc5OtherRegs8 = 72, kTc5nSoftmaxRegs = 104, kTc5nOtherRegs = 80;
static_assert(kTc5SoftmaxWarps * kTc5SoftmaxRegs + 4 * kTc5OtherRegs <= 16 * kTc5LaunchRegs, "registers");
static_assert(kTc5SoftmaxWarps * kTc5SoftmaxRegs8 + 8 * kTc5OtherRegs8 <= 20 * kTc5LaunchRegs8, "registers, FP8");
static_assert(kTc5SoftmaxWarps * kTc5nSoftmaxRegs + 8 * kTc5nOtherRegs <= 20 * kTc5LaunchRegs8, "registers, FP8 with the narrow path");
constexpr int kTc5Tok = 128;                     // tokens per group = N of Q K^T = columns of one S buffer
constexpr float kTc5Tau = 8.0f;                  // reference maximum moves only when it would grow by more than this (log2 units)
// Reference maxima [set][row]; row sums and the references they are relative to [piece parity][set][row]
constexpr int kTc5Xchg = 5 * kTc5Sets * kRowsPerGroup;
template <bool FP8> constexpr int tc5_xchg_bytes() { return (kTc5Xchg + (FP8 ? 512 : 0)) * 4; }     // (FP8: the narrow path's need more)
// FP8 pages: binary places by which P is held above the reference maximum.  P stays below 2^(8 + 7) < 65504.
constexpr float kTc5Fp8Lift = 7.0f;
constexpr int kTc5StgMax = 20;                   // FP8 pages: staging slots of V, one page each, at most
// FP8: value pages whose multiplier is kept.  Page x + 64 is issued once page x + 64 - 20 or a later one has been
// converted.  That is at least five groups (of at most 8 pages) after page x's, and a converting warp is less than
// two groups ahead of the others: it refills a V slot after the slot's P V, which waits for all of them.
constexpr int kTc5VmulRing = 64;
// Groups whose per-page data (token counts; FP8: scales) is kept.  The K producer writes a page's entry
// when it issues the page's copy, so the ring must be longer than its lead over the softmax warps.  A
// group never spans two segments, so in a run of one-page segments every page in flight is a group of
// its own.  The first page of group g is issued once its K slot is free: Q K^T of group g - NRK has run,
// hence P V of group g - NRK - 3 has released its S buffer: group g - NRK - 2 may still be read.
constexpr int kTc5MetaRing = 16;
// Barriers, the segment prefix and index cache, the exchange arrays, the charged prefix, the staging
// barriers (landed, emptied) and the value pages' multipliers, two words per page of the meta ring (FP8: three)
template <int GP, bool FP8> constexpr int tc5_tail_bytes() {
  return kTailBytes + tc5_xchg_bytes<FP8>() + (kMaxSegments + 2) * 4 + kTc5StgMax * (8 + 8) + kTc5VmulRing * 4 + kTc5MetaRing * (kTc5Tok / GP) * (FP8 ? 12 : 8) + (FP8 ? 2 * kTc5ScaleWarps * 4 : 0);
}

// Shared memory: the Q tile (FP8: one tile of codes per term), a ring of group-sized slots for K and one for V, FP8: a
// ring of page-sized slots where the codes of V land.
template <int D> constexpr int tc5_slot_bytes() { return kTc5Tok * D * 2; }                              // V, and bf16 K
template <int D, bool FP8> constexpr int tc5_kslot_bytes() { return kTc5Tok * D * (FP8 ? 1 : 2); }
constexpr int kTc5QTerms = 3;                    // FP8: E5M2 terms of a query
constexpr int kTc5nRows = 16;                    // FP8: most query rows of a segment on the narrow path (sparse_prefix_attn_tc5n.cuh)
constexpr int kTc5nLanes = 32;                   // entries of its per-row arrays, one per lane
constexpr int kTc5nP = kTc5Tok * 16;             // bytes of one term of 16 rows of its P'
constexpr int kTc5PTerms = 3;                    // E5M2 terms of P'
constexpr float kTc5nTermStep = 0.0625f;         // a term's unit is this much of the one before's
constexpr float kTc5nLift = 11.0f, kTc5nTop = 15.0f;   // binary places by which P' is held above the reference, and by which it may outgrow it
constexpr int tc5n_p_bytes() { return kTc5PTerms * kTc5nP; }
template <int D> constexpr int tc5n_q_bytes() { return kTc5nRows * D * kTc5QTerms; }
// The Q tile; narrow: in its place a smaller one and a set of P' terms for each set of softmax warps
template <int D, bool FP8> constexpr int tc5_q_bytes() {
  if (!FP8) return kRowsPerGroup * D * 2;
  static_assert(D == 64 || kRowsPerGroup * D * kTc5QTerms >= tc5n_q_bytes<D>() + kTc5Sets * tc5n_p_bytes(), "the narrow path's tiles (d = 128) fit");
  return kRowsPerGroup * D * kTc5QTerms;
}
template <int D, int GP, bool FP8> constexpr int tc5_ring_slots(bool v) {
  if (FP8) return v ? 2 : (D == 128 ? 3 : 6);                   // the staging slots take the rest
  const int n = (kSmemBudget - 1024 - tc5_tail_bytes<GP, FP8>() - tc5_q_bytes<D, false>()) / tc5_slot_bytes<D>();
  const int own = v ? n / 2 : (n + 1) / 2;                      // K is ahead of V by the S buffers
  return own > 6 ? 6 : own;
}
// FP8: pages of the staging ring of V: what the ring slots leave, up to five groups
template <int D, int GP> constexpr int tc5_stg_slots() {
  const int fit = (kSmemBudget - 1024 - tc5_tail_bytes<GP, true>() - tc5_q_bytes<D, true>() - tc5_ring_slots<D, GP, true>(false) * tc5_kslot_bytes<D, true>() -
                   tc5_ring_slots<D, GP, true>(true) * tc5_slot_bytes<D>()) / (GP * D), five = 5 * (kTc5Tok / GP);
  const int n = fit < five ? fit : five;
  return n < kTc5StgMax ? n : kTc5StgMax;
}
// FP8, narrow: the same memory as slots of a group's codes, half of them for K and half for V
template <int D, int GP> constexpr int tc5n_slots() {
  const int n = (tc5_ring_slots<D, GP, true>(false) * tc5_kslot_bytes<D, true>() + tc5_ring_slots<D, GP, true>(true) * tc5_slot_bytes<D>() +
                 tc5_stg_slots<D, GP>() * GP * D) / (2 * tc5_kslot_bytes<D, true>());
  return n < 6 ? n : 6;
}
template <int D, int GP, bool FP8> constexpr int tc5_smem_bytes() {
  return 1024 + tc5_q_bytes<D, FP8>() + tc5_ring_slots<D, GP, FP8>(false) * tc5_kslot_bytes<D, FP8>() + tc5_ring_slots<D, GP, FP8>(true) * tc5_slot_bytes<D>() +
         (FP8 ? tc5_stg_slots<D, GP>() * GP * D : 0) + tc5_tail_bytes<GP, FP8>();
}

// Shared-memory matrix descriptor: 128-byte swizzle, 8-row groups 1024 bytes apart; lbo = distance
// between 64-element blocks along the MN dimension of an MN-major operand.
__device__ __forceinline__ uint64_t tc5_desc(uint32_t saddr, uint32_t lbo) {
  return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16) |
         (static_cast<uint64_t>(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// K-major tile of 8-bit codes, rows of D bytes: the 128-byte swizzle for D = 128, the 64-byte one (8-row groups 512
// bytes apart) for D = 64.
template <int D> __device__ __forceinline__ uint64_t tc5_desc8(uint32_t saddr) {
  return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) | (1ull << 16) | (static_cast<uint64_t>((8 * D) >> 4) << 32) | (1ull << 46) |
         (static_cast<uint64_t>(D == 128 ? 2 : 4) << 61);
}
// byte offset of 16-byte chunk c of row t of such a tile
template <int D> __device__ __forceinline__ uint32_t tc5_sw8(int t, int c) {
  return static_cast<uint32_t>(t * D + ((D == 128 ? c ^ (t & 7) : c ^ ((t >> 1) & 3)) << 4));
}
// Instruction descriptor: fp32 accumulate, M x N tile, B optionally MN-major; kind::f16: A and B both bf16
// (format 1) or both fp16 (0); kind::f8f6f4: each E4M3 (0) or E5M2 (1).
__device__ __forceinline__ uint32_t tc5_idesc(int M, int N, int b_mn_major, uint32_t fmt_a, uint32_t fmt_b) {
  return (1u << 4) | (fmt_a << 7) | (fmt_b << 10) | (static_cast<uint32_t>(b_mn_major) << 16) |
         (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}
// D[tmem] (+)= A[tmem] . B[smem descriptor]
__device__ __forceinline__ void tc5_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// D[tmem] (+)= A[smem descriptor] . B[smem descriptor], bf16 operands, or 8-bit ones
__device__ __forceinline__ void tc5_mma_ss(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc5_mma_ss8(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// A warp's value that is the same in all lanes, in a form the compiler knows to be so, and the lane that issues for its warp.
// With `lane == 0` around the products and operands from ordinary registers an issuing warp took 75 to 100 cycles per
// instruction, whatever its shape (eight of them 600 to 820); chosen by elect.sync, 17 (eight 134), and the pipe's 64 count.
template <typename T> __device__ __forceinline__ T warp_uniform(T v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ bool elect_one() {
  uint32_t one;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(one) :: "memory");
  return one != 0;
}
// one answer for the whole warp
__device__ __forceinline__ bool warp_mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status, long long limit) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, status, limit)) != 0;
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
__device__ __forceinline__ void tc5_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
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
__device__ __forceinline__ void tc5_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// byte offset of 16-byte chunk c (0..7) of row t in a [rows][128 B] tile with the 128-byte swizzle
__device__ __forceinline__ uint32_t tc5_sw(int t, int c) { return static_cast<uint32_t>(t * 128 + ((c ^ (t & 7)) << 4)); }

#include "sparse_prefix_attn_tc5n.cuh"

// FP8: the K / V pools hold E4M3 bytes with one power-of-two scale per (page, KV head).  K is an operand as
// it lies: Q goes to shared memory as three E5M2 tiles whose sum is the bf16 query under a power of two of the row, and each is
// multiplied with the codes by kind::f8f6f4, at twice the 16-bit rate and with fp32 sums.  A term takes three significant bits and
// leaves at most half a unit of them, so three terms hold the eight of a bf16 value; with the row's largest element at
// 2^15 .. 2^16 that is exact down to 2^-9, 2^-24 of the largest, and below to within 2^-17, 2^-32 of it - more than the fp16
// value of an element keeps in a row below 256.  (Two E4M3 terms lose an element's low bits from 2^-9 of the row's largest
// on: with them the block of eight 32K prompts takes 954 us, 976 with three.  That is the third product; the slot of K's ring that its
// tile takes at d = 128 costs nothing: four slots and fewer staging pages are no faster.)  V is one on the narrow path only (P costs three terms there as well).  Here
// its codes land in a staging ring as they lie in memory; four converting warps, one per scheduler, turn a
// landed page into fp16 (exact) in the group's ring slot, in the layout the tensor maps of the bf16 path
// produce, and P is fp16.  The scales stay out of the conversion, which is bound by its instruction count: the
// key scale joins the softmax scale of the page's columns, and the value scale 2^e is added to their
// exponent, so that P' = p 2^e multiplies the codes of V and the row sum takes its columns back by 2^-e.  P'
// is rounded to fp16 relative to the largest p 2^e, so a page whose scale lies below another's would lose that
// many places of fp16's range.  Two things keep every weight at least as precise as an unscaled one: only the
// scales' part from 2^-6 to 2^0 goes into the exponent (pages of values up to 448; once a share has met a
// larger one, the converters go over each group of V a second time and multiply by the rest, exactly), and
// the reference lies 2^7 below the maximum.  A weight is then subnormal only 2^-15 or more below its row's
// largest, 2^-14 without scales.  Staging slots are single pages, so that one is refilled while its
// neighbours are converted.
// BOTH: with the narrow path (chosen by launch_tc5 on the size of the cache).
template <bool BOTH> struct Tc5Maps { CUtensorMap k, v; };
template <> struct Tc5Maps<true> { CUtensorMap k, v, vs; };      // vs: V once more, swizzled like K
template <int D, int GP, bool FP8, bool BOTH>
__global__ void __launch_bounds__(tc5_threads<FP8>(), 1)
attn_tc5_kernel(const __grid_constant__ Tc5Maps<BOTH> maps, AttnParams p) {
  static_assert(!BOTH || (FP8 && D == 128), "the narrow path");   // (d = 64: a group's bytes are HBM's 675 cycles, less than that path's own)
  constexpr int NRK = tc5_ring_slots<D, GP, FP8>(false), NRV = tc5_ring_slots<D, GP, FP8>(true);   // slots per ring
  constexpr int NSP = FP8 ? tc5_stg_slots<D, GP>() : 1, STG = GP * D;   // FP8: staging slots of V, bytes of a slot (one page of codes)
  constexpr int NT = tc5_threads<FP8>();
  constexpr int NN = BOTH ? tc5n_slots<D, GP>() : 1;   // narrow: slots of K, and of V
  constexpr int KSLOT = tc5_kslot_bytes<D, FP8>(), SLOT = tc5_slot_bytes<D>(), QB = tc5_q_bytes<D, FP8>();
  constexpr int PG = kTc5Tok / GP;              // pages per group
  constexpr int MR = kTc5MetaRing;              // groups of the meta ring
  constexpr int HALVES = D / 64;                // 64-column (128-byte) blocks of a 16-bit K or V row
  constexpr int HS = kTc5Tok * 128;             // bytes of one such block of a whole group
  constexpr int PAGE_BYTES = GP * D * 2;        // of a 16-bit page of K, and of V
  constexpr int UT = GP < 32 ? GP : 32, UPP = GP / UT;   // FP8: tokens that a converting warp takes at a time, such runs per page
  constexpr int SB = kTc5Sets;                  // S buffers, one per set
  constexpr uint32_t COL_O = 0, COL_S = 128;    // tensor-memory columns: O[D], S0[128], S1[128], S2[128]
  constexpr int TMEM_COLS = 512;
  static_assert(D == 64 || D == 128, "head dimensions of the tensor-core path");
  static_assert(GP == 16 || GP == 32 || GP == 64, "page sizes of the tensor-core path");
  static_assert(NRK >= 2 && NRV >= 2 && NRK <= 6 && NRV <= 6, "ring depth");
  // A converting warp waits on the parity of a staging slot whose page before, NSP pages back, another warp may have taken: that page
  // has to lie two groups back at least, where all four warps have finished (less than two groups lie between them).
  static_assert(!FP8 || (NSP >= 2 * PG && NSP <= kTc5StgMax), "staging ring");
  static_assert(NRK + 2 < MR && NN + 3 < MR, "the producer's lead fits the meta ring");   // (narrow: a set reads the ring until it leaves P')
  static_assert(!BOTH || (NN >= 2 && NN * 2 * KSLOT <= NRK * KSLOT + NRV * SLOT + NSP * STG), "narrow: slots");
  constexpr int kBars = 4 * 6 + 3 * SB + 3 + 4 + 4 * SB + 2 + 2 * SB + 2;
  static_assert(8 * kBars + 16 <= 512, "tail layout");

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - raw);
  const uint32_t qtile = base, kring = base + QB, vring = kring + NRK * KSLOT, vstg = vring + NRV * SLOT;   // vstg: FP8 only
  constexpr int TAIL = QB + NRK * KSLOT + NRV * SLOT + (FP8 ? NSP * STG : 0);
  uint8_t* tail = gen + TAIL;
  const uint32_t tail_s = base + TAIL;
  const uint32_t kfull = tail_s, kfree = kfull + 8 * 6, vfull = kfree + 8 * 6, vfree = vfull + 8 * 6;     // (room for six slots each)
  const uint32_t s_full = vfree + 8 * 6, s_free = s_full + 8 * SB, p_full = s_free + 8 * SB, q_full = p_full + 8 * SB, q_free = q_full + 8, o_free = q_free + 8;
  const uint32_t xbar = o_free + 8, mbar = xbar + 32;     // per lane quarter: the sets meet; [set][quarter]: a group's reference is published
  const uint32_t drain_bar = mbar + 32 * SB;            // two barriers: the issuing threads' last commit when the CTA gives up
  const uint32_t s_read = drain_bar + 16, meet = s_read + 8 * SB, piece_meet = meet + 8 * SB, path_bar = piece_meet + 8;   // FP8, narrow path
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 8 * kBars);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(const_cast<int*>(abort_flag) + 1);
  int* pre = reinterpret_cast<int*>(tail + 512);
  int* tok_s = pre + kMaxSegments + 2;
  int* na_s = tok_s + kStageIdx;
  int* len_s = na_s + kStageSeq;
  float* mref = reinterpret_cast<float*>(len_s + kStageSeq);   // [set][128]
  float* xsum = mref + SB * kRowsPerGroup;                       // [piece parity][set][128]: row sums of a piece ...
  float* xref = xsum + 2 * SB * kRowsPerGroup;                   // ... and the references they are relative to
  int* vpre = reinterpret_cast<int*>(mref + tc5_xchg_bytes<FP8>() / 4);  // prefix of the charged segment lengths (pages + pad)
  // FP8: a staging slot's page has landed / has been converted
  const uint32_t vstg_full = smem_u32(vpre + kMaxSegments + 1) + 4;   // (kMaxSegments + 1 is odd)
  const uint32_t vstg_free = vstg_full + 8 * kTc5StgMax;
  // FP8: multipliers of the newest value pages' codes, as two fp16; whether any was other than one
  volatile uint32_t* vmul = reinterpret_cast<volatile uint32_t*>(vpre + kMaxSegments + 2 + 4 * kTc5StgMax);
  volatile int* vmul_used = abort_flag + 2;
  // per page of the groups in flight, [MR][PG]: valid tokens (FP8: and the exponent field of the value scale's part in P << 8), FP8: key scale
  volatile int* meta = vpre + kMaxSegments + 2 + 4 * kTc5StgMax + kTc5VmulRing;
  volatile float* kscale_meta = reinterpret_cast<volatile float*>(const_cast<int*>(meta) + MR * PG);
  volatile float* vlog_meta = kscale_meta + MR * PG;           // narrow: the value scale's logarithm
  const bool staged = p.N * p.B <= kStageIdx && p.N <= kStageSeq;

  const int tid = threadIdx.x, lane = tid & 31, warp = warp_uniform(tid >> 5);
  if (tid == 0) {
    for (int i = 0; i < (NRK > NN ? NRK : NN); ++i) {
      mbar_init(kfull + 8 * i, 1);
      mbar_init(kfree + 8 * i, 1);
    }
    for (int i = 0; i < (NRV > NN ? NRV : NN); ++i) {
      mbar_init(vfull + 8 * i, FP8 ? kTc5CvtWarps : 1);   // the converting warps (narrow: as many arrivals by the producer) / the copies' bytes
      mbar_init(vfree + 8 * i, 1);
    }
    for (int b = 0; b < SB; ++b) {
      mbar_init(s_full + 8 * b, 1);                  // tcgen05.commit after Q K^T
      mbar_init(s_free + 8 * b, 1);                  // tcgen05.commit after P V: the S buffer is free and O holds the group
      mbar_init(p_full + 8 * b, kTc5SetWarps);
    }
    mbar_init(q_full, kTc5SoftmaxWarps);
    mbar_init(q_free, 1);
    mbar_init(o_free, kTc5SoftmaxWarps);
    for (int i = 0; i < 4; ++i) mbar_init(xbar + 8 * i, kTc5Sets);
    for (int i = 0; i < 4 * SB; ++i) mbar_init(mbar + 8 * i, 1);
    if (BOTH) {
      for (int b = 0; b < SB; ++b) {
        mbar_init(s_read + 8 * b, kTc5SetWarps);       // the set's scores have been read
        mbar_init(meet + 8 * b, kTc5SetWarps);         // the set's warps meet
      }
      mbar_init(piece_meet, kTc5SoftmaxWarps);         // all of them, at the end of a piece
      mbar_init(path_bar, kTc5ScaleWarps);           // the share's value scales have been looked at
    }
    mbar_init(drain_bar, 1);
    mbar_init(drain_bar + 8, 1);
    if (FP8)
      for (int i = 0; i < NSP; ++i) {
        mbar_init(vstg_full + 8 * i, 1);
        mbar_init(vstg_free + 8 * i, UPP);
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
  // behind the selection of the same step the lengths are final (stage 1 has waited for everything before the step)
  if (p.early && staged)
    for (int i = tid; i < p.N; i += NT) len_s[i] = p.kv_len[i];
  grid_dep_trigger();
  grid_dep_wait();                                 // nothing above reads what the kernels of this step write
  if (warp == 0) {
    segment_prefix(pre, p.n_seg, p.n_rg, p.Hkv, p.G, p.n_active, [&](int sk) { return p.union_count[sk]; }, p.B, lane, vpre);
  } else if (staged) {
    for (int i = tid - 32; i < p.N * p.B; i += NT - 32) tok_s[i] = p.active_idx[i];
    for (int i = tid - 32; i < p.N; i += NT - 32) {
      na_s[i] = clamp_active(p.n_active[i], p.B);
      if (!p.early) len_s[i] = p.kv_len[i];
    }
  }
  bool many_rows = false;                          // for the narrow path, in any sequence
  if (BOTH && warp > 0)
    for (int i = tid - 32; i < p.N; i += NT - 32) many_rows |= clamp_active(p.n_active[i], p.B) * p.G > kTc5nRows;
  tc5_fence_before();
  if constexpr (BOTH) many_rows = __syncthreads_or(many_rows) != 0;
  else __syncthreads();
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
  auto kv_len_of = [&](int s) { return staged ? len_s[s] : p.kv_len[s]; };

  Tc5Cta cta;
  cta.gen = gen; cta.base = base; cta.kring = kring; cta.vring = kring + NN * KSLOT;
  cta.kfull = kfull; cta.kfree = kfree; cta.vfull = vfull; cta.vfree = vfree; cta.s_full = s_full; cta.s_free = s_free; cta.p_full = p_full;
  cta.q_full = q_full; cta.q_free = q_free; cta.o_free = o_free; cta.s_read = s_read; cta.meet = meet; cta.piece_meet = piece_meet;
  cta.abort_flag = abort_flag; cta.pre = pre; cta.tok_s = tok_s; cta.na_s = na_s; cta.staged = staged;
  cta.scratch = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(mref) + 15) & ~static_cast<uintptr_t>(15));
  cta.meta = meta; cta.kscale_meta = kscale_meta; cta.vlog_meta = vlog_meta; cta.tmem = tmem; cta.lo = lo; cta.hi = hi; cta.sg0 = sg0;
  // The roles, once with the narrow path and once without: wide code that asks which path it is on is a tenth slower (shares of 32
  // groups 55.9 us, 61.7).
  auto roles = [&](auto narrow_too) {
  constexpr bool NARROW = decltype(narrow_too)::value;
  // Narrow: the share's value scales have the last word.  They must be positive, and so close to one another that no weight keeps fewer
  // bits than on the other path: P' holds a page's whole scale here, under a reference 2^4 higher, the part from 2^-6 to 2^0
  // there.  (Values up to 448 have no larger scales, and always pass.  With a limit of four, a hundredth of the pages eight times the
  // others' scale sent half of the CTAs the other way: a step of eight 32K prompts 120 us, 108 with all of them on it, 83 so.)
  // They are the last of three dependent reads, for the softmax warps, which look at them all, as for the producers, whose copies
  // wait for the answer.
  bool narrow = NARROW;
  float* scale_lo = reinterpret_cast<float*>(const_cast<int*>(meta)) + 3 * MR * PG;      // [8] smallest and largest, per warp that looks
  float* scale_hi = scale_lo + kTc5ScaleWarps;
  auto choose_path = [&]() {                         // false: a wait has run out
    if (!NARROW) return true;
    if (!warp_mbar_wait(path_bar, 0, abort_flag, p.status, p.wait_cycles)) return false;
    float a = INFINITY, b = 0.f;
#pragma unroll
    for (int w = 0; w < kTc5ScaleWarps; ++w) { a = fminf(a, scale_lo[w]); b = fmaxf(b, scale_hi[w]); }
    auto in_p = [](float v) { return fminf(fmaxf(v, 0.015625f), 1.f); };
    narrow = warp_uniform(a > 1e-18f && b < 1e18f && b * in_p(a) <= 16.f * a * in_p(b) ? 1 : 0) != 0;
    return true;
  };

  int issued = -1;                                   // producer warps: newest group (FP8: page) whose copies have been issued
  if (warp >= kTc5SoftmaxWarps) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(BOTH ? kTc5nOtherRegs : FP8 ? kTc5OtherRegs8 : kTc5OtherRegs));   // whole warpgroups
  if (warp == kTc5KWarp || warp == kTc5VWarp) {
    // ------------------------------------------------------------------ producer warps: one for K, one for V
    // Lane j of a batch of 32 consecutive items resolves item -> logical page -> physical page (a
    // three-stage pipeline over batches, the two dependent loads of different batches in flight
    // together) and later issues that page's copies itself.  A piece's items are cut into groups of
    // PG pages; the first lane of a group's run waits for the group's ring slot and announces the
    // group's bytes, then every lane of the run issues its page.
    const bool is_v = warp == kTc5VWarp;
    const unsigned long long policy = l2_evict_first_policy();
    bool staging = false;                              // page by page, into the staging ring
    const CUtensorMap* map = nullptr;
    uint32_t ring = 0;
    const uint32_t full0 = is_v ? vfull : kfull, free0 = is_v ? vfree : kfree;
    auto start = [&]() {                               // before the first copies: which path, hence which slots
      const bool ok = choose_path();
      staging = FP8 && is_v && !narrow;
      map = is_v ? &maps.v : &maps.k;
      if constexpr (BOTH)
        if (is_v && narrow) map = &maps.vs;
      ring = is_v ? (NARROW && narrow ? cta.vring : vring) : kring;
      return ok;
    };
    auto slot_of = [&](int grp) { return NARROW && narrow ? grp % NN : is_v ? grp % NRV : grp % NRK; };
    auto round_of = [&](int grp) { return NARROW && narrow ? grp / NN : is_v ? grp / NRV : grp / NRK; };
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
    auto scale_in_p = [](float vs) { return min(max((__float_as_int(vs) >> 23) & 0xff, 127 - 6), 127); };
    // copies of the batch of items b0 .. b0 + 31 (one per lane); false when a wait has run out
    auto issue = [&](int b0, const Ready& b) {
      const int nb = min(32, hi - b0);
      if (FP8 && staging) {                           // page by page: every lane handles its own staging slot
        // the value scale: 2^-6 .. 2^0 of it go into P (as an exponent field), the rest onto the codes (also
        // what a caller's own scale has beside its power of two)
        const __half2 in_v = __float2half2_rn(b.vs * __int_as_float((254 - scale_in_p(b.vs)) << 23));
        for (int pos = 0; pos < nb; ++pos) {
          int ok = 1;
          if (lane == pos) {
            const int x = b0 + pos - lo, slot = x % NSP, round = x / NSP;
            if (round > 0) ok = mbar_wait(vstg_free + 8 * slot, (round - 1) & 1, abort_flag, p.status, p.wait_cycles);
            if (ok) {
              const uint32_t m2 = *reinterpret_cast<const uint32_t*>(&in_v);
              vmul[x % kTc5VmulRing] = m2;
              if (m2 != 0x3c003c00u) *vmul_used = 1;
              mbar_expect_tx(vstg_full + 8 * slot, STG);
              tma_load_4d(vstg + slot * STG, map, vstg_full + 8 * slot, 0, 0, b.kh, b.phys, policy);
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
        const int slot = slot_of(grp), round = round_of(grp);
        if (j0 == 0) {
          int ok = 1;
          if (lane == 0 && round > 0) ok = mbar_wait(free0 + 8 * slot, (round - 1) & 1, abort_flag, p.status, p.wait_cycles);
          if (__shfl_sync(0xffffffffu, ok, 0) == 0) return false;
        }
        const bool mine = lane >= pos && lane < pos + cnt;
        if (!is_v && mine) {
          const int at = (grp % MR) * PG + b.j;
          meta[at] = FP8 ? b.valid | scale_in_p(b.vs) << 8 : b.valid;
          if (FP8) {
            kscale_meta[at] = b.ks;
            if (NARROW && narrow) vlog_meta[at] = log2f(b.vs);
          }
        }
        __syncwarp();
        if (j0 == 0 && lane == 0) {
          if (FP8 && is_v) mbar_arrive(full0 + 8 * slot, kTc5CvtWarps - 1);
          mbar_expect_tx(full0 + 8 * slot, ng * (FP8 ? STG : PAGE_BYTES));
        }
        __syncwarp();
        if (mine) {
          if constexpr (FP8) {                        // K: a page of codes, swizzled by the copy, is an operand as it is
            tma_load_4d(ring + slot * KSLOT + b.j * STG, map, full0 + 8 * slot, 0, 0, b.kh, b.phys, policy);
          } else {
            const uint32_t dst = ring + slot * SLOT + b.j * (GP * 128);
#pragma unroll
            for (int hf = 0; hf < HALVES; ++hf) tma_load_4d(dst + hf * HS, map, full0 + 8 * slot, hf * 64, 0, b.kh, b.phys, policy);
          }
        }
        issued = grp;
        pos += cnt;
      }
      return true;
    };
    // One batch of items per trip, every stage of another one: a list entry is requested two (FP8: three) trips before
    // its page is copied.  The pipeline fills and drains inside the loop, so that its code is there, and fetched, once.
    constexpr int DEEP = FP8 ? 32 : 0;                // FP8: the scales of a batch are requested a batch ahead
    Item a{};
    Ready b{}, b1{};
    bool go = true;
#pragma unroll 1
    for (int b0 = lo - 64 - DEEP; b0 < hi && go; b0 += 32) {
      const Item a_next = stage_a(b0 + lane + 64 + DEEP);
      Ready b_next{};
      if (b0 >= lo - 32 - DEEP) b_next = stage_b(b0 + lane + 32 + DEEP, a);
      if constexpr (FP8) {
        if (b0 >= lo - 32) stage_c(b0 + lane + 32, b1);
        if (b0 == lo) go = start();
        if (b0 >= lo && go) go = issue(b0, b);
        b = b1;
        b1 = b_next;
      } else {
        if (b0 >= lo) {
          if (b0 == lo) start();
          stage_c(b0 + lane, b);
          go = issue(b0, b);
        }
        b = b_next;
      }
      a = a_next;
    }
  } else if (FP8 && warp >= kTc5CvtWarp) {
    if (choose_path() && !narrow) {
    // ------------------------------------------------------------------ converting warps (FP8 pages): V
    // A warp takes every fourth run of UT tokens (a page, or half a page of 64) of a group: one wait and one arrival for
    // up to 64 conversions (a quarter of every page per warp had four of each; a block of eight 32K prompts 1,032 us, 968 so).
    // A lane takes eight codes at a time (one 16-byte chunk of fp16): 8-byte reads of consecutive codes and 16-byte
    // stores of consecutive swizzled chunks, both without bank conflicts; up to eight are requested before any is converted.
    const uint8_t* stg_gen = gen + (vstg - base);
    uint8_t* ring_gen = gen + (vring - base);
    constexpr int CPR = D / 8, TPI = 32 / CPR;        // chunks of a row, tokens per warp access
    constexpr int NU = UT / TPI, U = NU < 8 ? NU : 8; // accesses per run, in flight
    static_assert(NU % U == 0 && NU * TPI == UT, "a run's tokens");
    const int tl = lane / CPR, c = lane % CPR;
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
        const int ng = min(PG, seg_end - first), sr = g % NRV;
        if (g >= NRV) ok = wait(vfree + 8 * sr, (g / NRV - 1) & 1);
        uint8_t* dst = ring_gen + sr * SLOT + (c >> 3) * HS;
        for (int u = warp - kTc5CvtWarp; u < ng * UPP; u += kTc5CvtWarps) {
          const int pg = u / UPP, x = first + pg - lo, ss = x % NSP, t0 = u % UPP * UT + tl;
          ok = ok && wait(vstg_full + 8 * ss, (x / NSP) & 1);
          if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
          const uint8_t* src = stg_gen + ss * STG + t0 * D + c * 8;
#pragma unroll 1
          for (int u0 = 0; u0 < NU; u0 += U) {
            uint2 w[U];
#pragma unroll
            for (int e = 0; e < U; ++e) w[e] = *reinterpret_cast<const uint2*>(src + (u0 + e) * TPI * D);
#pragma unroll
            for (int e = 0; e < U; ++e) {
              const uint32_t x4[4] = {w[e].x & 0xffffu, w[e].x >> 16, w[e].y & 0xffffu, w[e].y >> 16};
              uint32_t h[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const __half2_raw v = __nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(x4[k]), __NV_E4M3);
                h[k] = *reinterpret_cast<const uint32_t*>(&v);
              }
              *reinterpret_cast<uint4*>(dst + tc5_sw(pg * GP + t0 + (u0 + e) * TPI, c & 7)) = make_uint4(h[0], h[1], h[2], h[3]);
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(vstg_free + 8 * ss, 1);
        }
        if (!ok) break;
        if (*vmul_used) {                             // this lane's chunks once more, times what of the scales is not in P
          for (int u = warp - kTc5CvtWarp; u < ng * UPP; u += kTc5CvtWarps) {
            const int pg = u / UPP;
            const uint32_t mul = vmul[(first + pg - lo) % kTc5VmulRing];
            const __half2 m2 = *reinterpret_cast<const __half2*>(&mul);
#pragma unroll 1
            for (int i = 0; i < NU; ++i) {
              uint4* at = reinterpret_cast<uint4*>(dst + tc5_sw(pg * GP + u % UPP * UT + tl + i * TPI, c & 7));
              uint4 x = *at;
              auto scale = [&](uint32_t& y) {
                const __half2 v = __hmul2(*reinterpret_cast<const __half2*>(&y), m2);
                y = *reinterpret_cast<const uint32_t*>(&v);
              };
              scale(x.x); scale(x.y); scale(x.z); scale(x.w);
              *at = x;
            }
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read the slot through the async proxy
        __syncwarp();
        if (lane == 0) mbar_arrive(vfull + 8 * sr, 1);
      }
      item = seg_end;
      ++sg;
      while (item < hi && pre[sg + 1] <= item) ++sg;
    }
    }
  } else if (warp == kTc5QkWarp) {
    // ------------------------------------------------------------------ Q K^T issuer (a warp, one elected lane issues)
    if (!choose_path()) {
    } else if (narrow) {
      if constexpr (NARROW) tc5n_issue_qk<D, GP>(p, cta);
    } else {
      const uint32_t qt = warp_uniform(qtile), kr = warp_uniform(kring), s_col0 = warp_uniform(tmem) + COL_S;
      const int end = warp_uniform(hi);
      auto wait = [&](uint32_t bar, uint32_t parity) { return warp_mbar_wait(bar, parity, abort_flag, p.status, p.wait_cycles); };
      int sg = sg0, item = warp_uniform(lo), piece = 0, g = 0;
      bool ok = true;
      while (item < end && ok) {
        const int seg_end = warp_uniform(min(end, pre[sg + 1]));
        ok = wait(q_full, piece & 1);
        for (int first = item; first < seg_end && ok; first += PG, ++g) {
          const int ng = min(PG, seg_end - first), b = g % SB, use = g / SB, slot = g % NRK;
          ok = wait(kfull + 8 * slot, (g / NRK) & 1);
          ok = ok && (use == 0 || wait(s_free + 8 * b, (use - 1) & 1));
          if (!ok) break;
          tc5_fence_after();
          if (elect_one()) {
            const uint32_t kt = kr + slot * KSLOT, s_col = s_col0 + b * kTc5Tok;
            if constexpr (FP8) {                       // the terms of Q (E5M2) against the same codes (E4M3)
              const uint32_t idesc = tc5_idesc(kRowsPerGroup, ng * GP, 0, 1u, 0u);
              const uint64_t qd = tc5_desc8<D>(qt), kd = tc5_desc8<D>(kt);
#pragma unroll
              for (int ks = 0; ks < D / 32; ++ks)
#pragma unroll
                for (int t = 0; t < kTc5QTerms; ++t)
                  tc5_mma_ss8(s_col, qd + (t * (kRowsPerGroup * D) + ks * 32) / 16, kd + ks * 2, idesc, ks + t > 0 ? 1u : 0u);
            } else {
              const uint32_t idesc = tc5_idesc(kRowsPerGroup, ng * GP, 0, 1u, 1u);
              const uint64_t qd = tc5_desc(qt, 16), kd = tc5_desc(kt, 16);
#pragma unroll
              for (int ks = 0; ks < D / 16; ++ks) {
                const uint32_t at = ((ks >> 2) * HS + (ks & 3) * 32) / 16;
                tc5_mma_ss(s_col, qd + at, kd + at, idesc, ks > 0 ? 1u : 0u);
              }
            }
            tc5_commit(s_full + 8 * b);
            tc5_commit(kfree + 8 * slot);
            if (first + PG >= seg_end) tc5_commit(q_free);        // Q may be replaced once the piece's last product has run
          }
          __syncwarp();
        }
        item = seg_end;
        ++sg;
        ++piece;
        while (item < end && warp_uniform(pre[sg + 1]) <= item) ++sg;
      }
    }
  } else if (warp == kTc5PvWarp) {
    // ------------------------------------------------------------------ P V issuer (a warp, one elected lane issues)
    if (!choose_path()) {
    } else if (narrow) {
      if constexpr (NARROW) tc5n_issue_pv<D, GP>(p, cta);
    } else {
      const uint32_t idesc = tc5_idesc(kRowsPerGroup, D, 1, FP8 ? 0u : 1u, FP8 ? 0u : 1u);
      const uint32_t vr = warp_uniform(vring), tm = warp_uniform(tmem);
      const int end = warp_uniform(hi);
      auto wait = [&](uint32_t bar, uint32_t parity) { return warp_mbar_wait(bar, parity, abort_flag, p.status, p.wait_cycles); };
      int sg = sg0, item = warp_uniform(lo), piece = 0, g = 0;
      bool ok = true;
      while (item < end && ok) {
        const int seg_end = warp_uniform(min(end, pre[sg + 1]));
        for (int first = item; first < seg_end && ok; first += PG, ++g) {
          const int ng = min(PG, seg_end - first), b = g % SB, use = g / SB, slot = g % NRV;
          ok = wait(vfull + 8 * slot, (g / NRV) & 1);
          if (first == item && piece > 0) ok = ok && wait(o_free, (piece - 1) & 1);   // O has been read
          ok = ok && wait(p_full + 8 * b, use & 1);
          if (!ok) break;
          tc5_fence_after();
          if (elect_one()) {
            const uint64_t vd = tc5_desc(vr + slot * SLOT, HS);
            const uint32_t p_col = tm + COL_S + b * kTc5Tok, fresh = first == item ? 0u : 1u;
            if (ng == PG) {
#pragma unroll
              for (int ks = 0; ks < kTc5Tok / 16; ++ks) tc5_mma_ts(tm + COL_O, p_col + ks * 8, vd + ks * 128, idesc, ks == 0 ? fresh : 1u);
            } else {
              for (int ks = 0; ks < ng * GP / 16; ++ks) tc5_mma_ts(tm + COL_O, p_col + ks * 8, vd + ks * 128, idesc, ks == 0 ? fresh : 1u);
            }
            tc5_commit(vfree + 8 * slot);
            tc5_commit(s_free + 8 * b);
          }
          __syncwarp();
        }
        item = seg_end;
        ++sg;
        ++piece;
        while (item < end && warp_uniform(pre[sg + 1]) <= item) ++sg;
      }
    }
  }
  } else {
    // ------------------------------------------------------------------ softmax / epilogue warps
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(BOTH ? kTc5nSoftmaxRegs : FP8 ? kTc5SoftmaxRegs8 : kTc5SoftmaxRegs));
    if (NARROW && warp < kTc5ScaleWarps) {  // the share's value scales (the last set has its instructions to fetch)
      float a = INFINITY, b = 0.f;
      int sg = sg0;
      for (int i = lo + tid; i < hi; i += kTc5ScaleWarps * 32) {
        while (pre[sg + 1] <= i) ++sg;
        const int sk = sg % p.n_sk, page = ld_nc_s32(p.union_pages + static_cast<size_t>(sk) * p.Pmax + (i - pre[sg]));
        const int phys = page >= 0 && page < p.Pmax ? ld_nc_s32(p.page_table + static_cast<size_t>(sk / p.Hkv) * p.Pmax + page) : -1;
        const float v = phys >= 0 && phys < p.n_phys ? __ldg(p.v_scale + static_cast<size_t>(phys) * p.Hkv + sk % p.Hkv) : -1.f;
        a = fminf(a, v == v ? v : -1.f);             // (NaN: the wide path)
        b = fmaxf(b, v);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        a = fminf(a, __shfl_xor_sync(0xffffffffu, a, o));
        b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, o));
      }
      if (lane == 0) {
        scale_lo[warp] = a;
        scale_hi[warp] = b;
        mbar_arrive(path_bar, 1);
      }
    }
    if constexpr (NARROW) {
      tc5n_softmax<D, GP>(p, cta, [&]() { return choose_path() && narrow; });
    }
    if (!narrow) {                                     // (still set where a wait has run out)
    // Thread = query row (tensor-memory lane 32 * (warp % 4) + lane); set h = warp / 4 takes the groups
    // h, h + 3, ..., all columns, in S buffer h.  The three warps of a scheduler work on different groups, a
    // third of a period apart, so that one's exponentials (one special-function unit per scheduler) run while
    // the others load, take maxima, pack and store.  All sets add to the same O, under the same reference
    // maximum: a group's handler takes the reference over from the group before it, whose set publishes it
    // as soon as it has decided (before its exponentials).
    const __nv_bfloat16* q = static_cast<const __nv_bfloat16*>(p.q);
    const int quarter = warp & 3, h = warp >> 2, h_prev = h == 0 ? kTc5Sets - 1 : h - 1;
    const int r = quarter * 32 + lane;                         // row of the tile = tensor-memory lane
    const uint32_t lane_addr = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
    const uint32_t s_addr = lane_addr + COL_S + h * kTc5Tok;
    // every wait of these warps ends with one answer for the whole warp: the tensor-memory
    // instructions that follow need all 32 lanes
    auto warp_wait = [&](uint32_t bar, uint32_t parity) {
      return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, p.status, p.wait_cycles)) != 0;
    };
    int sg = sg0, item = lo, piece = 0, g = 0;
    int n_pub = 0;                                              // references the previous set's warp of this quarter has published, or will have
    bool ok = true;
    while (item < hi && ok) {
      const int seg_end = min(hi, pre[sg + 1]);
      const int rg = sg / p.n_sk, sk = sg % p.n_sk, s = sk / p.Hkv, kh = sk % p.Hkv;
      const int rows = rows_in_group(cta.n_active_of(p, s), p.G, rg);
      const bool warp_has_rows = quarter * 32 < rows;          // the same for the warps of a quarter
      float scale2 = p.sm_scale * kLog2e;
      // ---- the piece's Q tile: sets 0 and 1 write half a row per thread
      {
        const uint4* src = nullptr;
        if (r < rows) {
          const int row = rg * kRowsPerGroup + r, a = row / p.G, gi = row % p.G;
          int tok = cta.token_of(p, s, a);
          if (tok < 0 || tok >= p.B) { set_status(p.status, LOSA_ERR_BOUNDS); tok = 0; }
          src = reinterpret_cast<const uint4*>(q + ((static_cast<size_t>(s) * p.B + tok) * p.Hq + kh * p.G + gi) * D);
        }
        constexpr int NC = D / 16;                              // 16-byte chunks of half a row
        uint4 qv[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) qv[c] = src && h < 2 ? __ldg(src + h * NC + c) : make_uint4(0u, 0u, 0u, 0u);
        if constexpr (FP8) {
          // Q in three E5M2 terms, under the power of two that brings the row's largest element to 2^15 .. 2^16 (what of it
          // lies above 57344, the largest E5M2 value, is left to the second term).
          uint32_t top = 0;                                     // of the whole row
          if (src) {
#pragma unroll 4
            for (int c = 0; c < 2 * NC; ++c) {
              const uint4 v = __ldg(src + c);
              const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
              for (int e = 0; e < 4; ++e) top = max(top, max((w[e] << 16) & 0x7fffffffu, w[e] & 0x7fff0000u));
            }
          }
          // (exponent field e of the largest element: times 2^(142 - e) in two steps, each a normal number)
          const int e_top = max(static_cast<int>(top >> 23), 16), up = 142 - e_top, u0 = up / 2, u1 = up - u0;
          const float f0 = __int_as_float((127 + u0) << 23), f1 = __int_as_float((127 + u1) << 23);
          scale2 *= __int_as_float((127 - u0) << 23) * __int_as_float((127 - u1) << 23);
          if ((top >> 23) == 255) scale2 = __int_as_float(top);           // an infinity or NaN among them: in all the row's scores
          if (piece > 0) ok = warp_wait(q_free, (piece - 1) & 1);
          if (!ok) break;
          if (warp_has_rows && h < 2) {
#pragma unroll
            for (int c = 0; c < NC; c += 2) {                   // two chunks of bf16 make one of codes
              uint32_t w4[kTc5QTerms][4];
#pragma unroll
              for (int x = 0; x < 2; ++x) {
                const uint32_t w[4] = {qv[c + x].x, qv[c + x].y, qv[c + x].z, qv[c + x].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  float2 v = make_float2(__uint_as_float(w[e] << 16) * f0 * f1, __uint_as_float(w[e] & 0xffff0000u) * f0 * f1);
#pragma unroll
                  for (int t = 0; t < kTc5QTerms; ++t) {
                    const uint32_t code = __nv_cvt_float2_to_fp8x2(v, __NV_SATFINITE, __NV_E5M2);
                    const float2 part = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2(code, __NV_E5M2)));
                    v.x -= part.x;
                    v.y -= part.y;
                    if (e % 2 == 0) w4[t][2 * x + e / 2] = code;
                    else w4[t][2 * x + e / 2] |= code << 16;
                  }
                }
              }
              uint8_t* dst = gen + tc5_sw8<D>(r, h * (NC / 2) + c / 2);
#pragma unroll
              for (int t = 0; t < kTc5QTerms; ++t)
                *reinterpret_cast<uint4*>(dst + t * (kRowsPerGroup * D)) = make_uint4(w4[t][0], w4[t][1], w4[t][2], w4[t][3]);
            }
          }
        } else {
          if (piece > 0) ok = warp_wait(q_free, (piece - 1) & 1);
          if (!ok) break;
          if (warp_has_rows && h < 2) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {                      // 64-column blocks of 128-byte rows, 128-byte swizzle
              const int ch = h * NC + c;
              *reinterpret_cast<uint4*>(gen + (ch >> 3) * HS + tc5_sw(r, ch & 7)) = qv[c];
            }
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read the tile through the async proxy
        __syncwarp();
        if (lane == 0) mbar_arrive(q_full, 1);
      }
      float m_ref = -INFINITY, l = 0.f;                         // l: the groups of this set, relative to m_ref
      // The last set, which has time until the share's third group, first takes one that is not there: no waits, no arrivals, nothing
      // written.  It fetches the loop's instructions while the producers still look for their pages; the first group's set
      // would wait for every line of them behind the page copies (two steps of one 64K sequence in two layers 164.8 us, 163.8 so, of one of
      // 128K 188.0 and 186.8, of pooled lists 282.3 and 280.0).  Not where a first piece of one or two groups ends before others of the
      // share: the sets meet there, and this one would come late (64 segments, shares of one group 14.0 us, 15.0 with the walk).
      // Longer shares wait for HBM from the start: eight 32K prompts, 36 groups, 420.3 us without it and 420.9 with it.
      int dry = piece == 0 && h == kTc5Sets - 1 && hi - lo < 24 * PG && (seg_end == hi || seg_end - item >= 3 * PG) ? 1 : 0;
      for (int first = item; first < seg_end && ok;) {
        asm volatile("" : "+r"(dry));                           // (one copy of the code)
        const int turn = g % kTc5Sets;
        if (turn != h && !dry) {                                // another set's
          if (warp_has_rows && turn == h_prev) ++n_pub;
          first += PG;
          ++g;
          continue;
        }
        const int ng = min(PG, seg_end - first), ncol = ng * GP;
        volatile int* gmeta = meta + (g % MR) * PG;
        auto valid_of = [&](int j) { return FP8 ? gmeta[j] & 0xff : gmeta[j]; };     // tokens of the group's page j
        if (!dry) ok = warp_wait(s_full + 8 * h, (g / kTc5Sets) & 1);
        if (!ok) break;
        tc5_fence_after();
        // pages with fewer than GP tokens (the last page of a prefix), or a group that ends inside a
        // 32-column chunk, need per-column masks; everything else takes the plain path
        const bool any_short = __any_sync(0xffffffffu, lane < ng && valid_of(min(lane, PG - 1)) < GP && !dry) != 0;
        const bool ragged = any_short || (ncol & 31) != 0;
        if (warp_has_rows) {
          // FP8: the scores of a page carry its key scale, its weights the value scale's part 2^vexp: runs of
          // PW columns, each of one page
          constexpr int PW = GP < 32 ? GP : 32;
          auto run_page = [&](int col) { return min(col / GP, ng - 1); };
          auto run_mul = [&](int col) { return FP8 ? scale2 * kscale_meta[(g % MR) * PG + run_page(col)] : scale2; };
          auto run_exp = [&](int col) { return static_cast<float>((gmeta[run_page(col)] >> 8) - 127); };
          // of columns col .. col + 31 of the scores, those that hold no token become -inf
          auto mask_chunk = [&](uint32_t* v, int col) {
            uint32_t keep = 0;
#pragma unroll
            for (int x = 0; x < 32 / PW; ++x) {
              const int c = col + x * PW, j = c / GP, n = j < ng ? min(max(valid_of(j) - c % GP, 0), PW) : 0;
              keep |= (n >= 32 ? 0xffffffffu : (1u << n) - 1u) << (x * PW % 32);
            }
#pragma unroll
            for (int e = 0; e < 32; ++e) if (!((keep >> e) & 1u)) v[e] = 0xff800000u;
          };
          // The scores are read from tensor memory twice, 32 columns at a time in rolled loops.  With the row in registers
          // and straight code for its 128 columns (two sets of warps), the first group's exponentials of a sparse step
          // took 2,700 to 7,900 cycles for 15 KB of instructions, fetched behind the page copies that have just filled
          // the memory queues (2,100 now); 64 columns at a time: eight 32K prompts, dense step 246 against 230 us.
          // ---- pass 1: the row's maximum over the group (FP8: of the shifted exponents)
          float mx_own = -INFINITY;
#pragma unroll 1
          for (int c0 = 0; c0 < ncol; c0 += 32) {
            uint32_t v[32];
            tc5_ld32_nowait(s_addr + c0, v);
            tc5_wait_ld();
            tc5_pin32(v);
            if (ragged) mask_chunk(v, c0);
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int e = 0; e < 32; ++e) {
              mx[e & 3] = fmaxf(mx[e & 3], __uint_as_float(v[e]));
              if (FP8 && (e + 1) % PW == 0) {
                mx_own = fmaxf(mx_own, fmaf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])), run_mul(c0 + e), run_exp(c0 + e)));
                mx[0] = mx[1] = mx[2] = mx[3] = -INFINITY;
              }
            }
            if (!FP8) mx_own = fmaxf(mx_own, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])));
          }
          // ---- the reference maximum: the one of the group before, moved when it would grow by more than 2^8
          float m_prev = -INFINITY;
          if (first != item) {
            ok = warp_wait(mbar + 8 * (4 * h_prev + quarter), (n_pub - 1) & 1);
            m_prev = mref[h_prev * kRowsPerGroup + r];
          }
          constexpr float LIFT = FP8 ? kTc5Fp8Lift : 0.f;
          const float m_own = FP8 ? mx_own : mx_own * scale2;
          float m_new = m_prev;
          if (m_own > m_prev + (kTc5Tau + LIFT) || (m_prev == -INFINITY && m_own > -INFINITY)) m_new = m_own - LIFT;
          if (!dry) mref[h * kRowsPerGroup + r] = m_new;
          __syncwarp();
          if (lane == 0 && !dry) mbar_arrive(mbar + 8 * (4 * h + quarter), 1);
          if (m_ref != m_new) {
            l *= m_ref == -INFINITY ? 0.f : ex2(m_ref - m_new);
            m_ref = m_new;
          }
          // ---- rescale O (rare): the previous group's P V must have run, this one's waits for P
          if (first != item && __any_sync(0xffffffffu, m_prev != m_new)) {
            const float corr = m_prev == m_new ? 1.f : (m_prev == -INFINITY ? 0.f : ex2(m_prev - m_new));
            ok = ok && warp_wait(s_free + 8 * h_prev, ((g - 1) / kTc5Sets) & 1);
            if (ok) {
              tc5_fence_after();
#pragma unroll 1
              for (int c0 = 0; c0 < D; c0 += 16) {
                uint32_t w[16];
                tc5_ld16(lane_addr + COL_O + c0, w);
#pragma unroll
                for (int e = 0; e < 16; ++e) w[e] = __float_as_uint(__uint_as_float(w[e]) * corr);
                tc5_st16(lane_addr + COL_O + c0, w);
              }
              tc5_wait_st();
            }
          }
          // ---- pass 2: P = 2^(s - m) as 16-bit values, written over the scores (columns 2c, 2c+1 of P take the
          //      place of column c of S, which has been read by then)
          if (ok) {
            const float ms = (m_ref == -INFINITY) ? 0.f : m_ref;
#pragma unroll 1
            for (int c0 = 0; c0 < ncol; c0 += 32) {
              uint32_t v[32];
              tc5_ld32_nowait(s_addr + c0, v);
              tc5_wait_ld();
              tc5_pin32(v);
              if (ragged) mask_chunk(v, c0);
              float sum[4] = {0.f, 0.f, 0.f, 0.f};
              float mul = scale2, add = -ms, vexp = 0.f;
              uint32_t w[16];
#pragma unroll
              for (int e = 0; e < 16; ++e) {
                if (FP8 && (2 * e) % PW == 0) {
                  mul = run_mul(c0 + 2 * e);
                  vexp = run_exp(c0 + 2 * e);
                  add = vexp - ms;
                }
                const float p0 = ex2(fmaf(__uint_as_float(v[2 * e]), mul, add));
                const float p1 = ex2(fmaf(__uint_as_float(v[2 * e + 1]), mul, add));
                sum[e & 3] += p0 + p1;
                w[e] = FP8 ? pack_f16(p0, p1) : pack_bf16(p0, p1);
                if (FP8 && (2 * e + 2) % PW == 0) {     // the page run's sum, without the value scale
                  l = fmaf((sum[0] + sum[1]) + (sum[2] + sum[3]), __int_as_float((127 - static_cast<int>(vexp)) << 23), l);
                  sum[0] = sum[1] = sum[2] = sum[3] = 0.f;
                }
              }
              if (!dry) tc5_st16(s_addr + c0 / 2, w);
              if (!FP8) l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
            }
            tc5_wait_st();
          }
        }
        if (!ok) break;
        if (any_short) {
          // rows of V past the end of the prefix may hold anything (even NaN): clear them once the tile has
          // landed (all warps of the set, whether or not they own rows).  The slot's previous tile must have been
          // used first: until then its barrier may be a phase behind, with the parity that is waited for.
          const int slot = g % NRV;
          if (g >= NRV) ok = warp_wait(vfree + 8 * slot, (g / NRV - 1) & 1);
          ok = ok && warp_wait(vfull + 8 * slot, (g / NRV) & 1);
          if (!ok) break;
          uint8_t* vg = gen + (vring - base) + slot * SLOT;
          for (int j = 0; j < ng; ++j) {
            const int valid = valid_of(j);
            for (int idx = r; idx < (GP - valid) * (D / 8); idx += kTc5SetWarps * 32) {
              const int t = j * GP + valid + idx / (D / 8), ch = idx % (D / 8);
              *reinterpret_cast<uint4*>(vg + (ch >> 3) * HS + tc5_sw(t, ch & 7)) = make_uint4(0u, 0u, 0u, 0u);
            }
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        tc5_fence_before();
        __syncwarp();
        if (dry) {
          dry = 0;
          m_ref = -INFINITY;
          l = 0.f;
          continue;
        }
        if (lane == 0) mbar_arrive(p_full + 8 * h, 1);
        first += PG;
        ++g;
      }
      if (!ok) break;
      // ---- the piece's record: one 16-row tile record per 16 rows, reference maximum in base-2
      //      units; the sets share the columns, set 0 writes the row's maximum and sum.
      // O is complete when the P V of the piece's last group has run.  Only the set that handled that group may wait for it on the
      // group's S buffer: for the others the buffer's barrier can still be a phase behind, with the parity waited for.  The meeting
      // of a quarter's three warps, rows or not, hands the set's knowledge on, and keeps every warp from running ahead: without
      // it one could arrive on o_free for two pieces while another still reads O.  The next piece's sums go to the other buffer: they
      // can be written while set 0 reads these, those of the piece after it only behind its meeting, which waits for o_free.
      if ((g - 1) % kTc5Sets == h) {
        ok = warp_wait(s_free + 8 * h, ((g - 1) / kTc5Sets) & 1);
        if (!ok) break;
        tc5_fence_after();
      }
      const int sums = (piece & 1) * SB * kRowsPerGroup;
      xsum[sums + h * kRowsPerGroup + r] = l;
      xref[sums + h * kRowsPerGroup + r] = m_ref;
      tc5_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(xbar + 8 * quarter, 1);
      ok = warp_wait(xbar + 8 * quarter, piece & 1);
      if (!ok) break;
      tc5_fence_after();
      if (warp_has_rows) {
        float* rec = record_base(p.partials, blockIdx.x + sg, r / kTileRows, D);
        const int rr = r % kTileRows;
#pragma unroll 1
        for (int c0 = 32 * h; c0 < D; c0 += 32 * kTc5Sets) {
          float t[32];
          tc5_ld32(lane_addr + COL_O + c0, t);
          if (r < rows) {
#pragma unroll
            for (int e = 0; e < 32; e += 4)
              *reinterpret_cast<float4*>(rec + 2 * kTileRows + rr * D + c0 + e) = make_float4(t[e], t[e + 1], t[e + 2], t[e + 3]);
          }
        }
        if (h == 0 && r < rows) {
          const float m_last = mref[((g - 1) % kTc5Sets) * kRowsPerGroup + r];
          float total = 0.f;
#pragma unroll
          for (int x = 0; x < kTc5Sets; ++x) {
            const float m_x = xref[sums + x * kRowsPerGroup + r];
            if (m_x != -INFINITY) total = fmaf(xsum[sums + x * kRowsPerGroup + r], ex2(m_x - m_last), total);
          }
          rec[rr] = m_last;
          rec[kTileRows + rr] = total;
        }
      }
      tc5_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(o_free, 1);
      item = seg_end;
      ++sg;
      ++piece;
      while (item < hi && pre[sg + 1] <= item) ++sg;
    }
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
      const bool is_v = warp == kTc5VWarp;
      const bool staging = FP8 && is_v && !narrow;
      const uint32_t full0 = is_v ? (staging ? vstg_full : vfull) : kfull;
      const int NSL = NARROW && narrow ? NN : is_v ? (FP8 ? NSP : NRV) : NRK;
      for (int sl = 0; sl < NSL; ++sl) {
        if (issued < sl) continue;
        const int gl = issued - (issued - sl) % NSL;
        mbar_drain(full0 + 8 * sl, (gl / NSL) & 1);
      }
    }
    if ((warp == kTc5QkWarp || warp == kTc5PvWarp) && elect_one()) {
      const uint32_t bar = drain_bar + (warp == kTc5PvWarp ? 8 : 0);
      tc5_commit(bar);
      mbar_drain(bar, 0);
    }
    __syncthreads();
  }
  };
  // Few rows in all sequences and shares of a group or more: tokens take the lanes (see the narrow path's header).  Every CTA comes to
  // the same answer: with CTAs of both kinds in one grid, which fetch both paths' instructions behind each other's page
  // copies, a grid takes longer than either way alone (shares of eight groups, 64 segments: 27.6 us wide, 22.9 narrow, 36.7 where
  // every other share was a page too short).  Shares of 1 / 3 / 5 / 16 groups, one sequence of 12 rows per KV head: 17.0 / 19.7 /
  // 22.4 / 34.8 us wide, 16.4 / 18.0 / 19.4 / 27.7 narrow.  (warp_uniform: under a branch that might diverge the products take
  // no uniform operands, and the wide path 60.2 us for shares of 32 groups, 56.3 so.)
  if constexpr (BOTH) {
    if (warp_uniform(!many_rows && pre[p.n_seg] >= PG * n_share ? 1 : 0) != 0) roles(std::true_type{});
    else roles(std::false_type{});
  } else {
    roles(std::false_type{});
  }
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(TMEM_COLS) : "memory");
}
