// Stage 4 on FP8 pages, shares of few query rows (sparse steps): the other way round.  Included by
// sparse_prefix_attn_tc5.cuh (same namespace); part of attn_tc5_kernel, which decides for the whole grid, and once more per CTA on
// the value scales.
//
// A sparse step has m active tokens x G heads, 4 to 32 rows for the most part, where the tile of sparse_prefix_attn_tc5.cuh has 128: there the
// softmax is one warp's work per group (128 exponentials per thread, one after the other) while the others of its set idle,
// and the conversion of V and the products' operands move 200 KB per group through shared memory.  Here tokens take the 128
// lanes and up to 16 query rows the columns, and both K and V are operands as they lie:
//   S[128 tokens x rows]  = K . Q^T     A = the group's codes, B = Q's three E5M2 terms (one after the other into the same columns)
//   softmax               thread = token, 16 exponentials; P' = 2^(s - m) vs, vs the page's value scale, in fp16 precision
//   P'                    as three E5M2 terms in shared memory: an E5M2 value is the upper byte of an fp16 one, and three of
//                         them, each rounded to nearest, make up the eleven significant bits of P'
//   O[D x 3 rows]        += V^T . P'    A = the group's codes (MN-major), B = the terms (MN-major), a column each
// E5M2 ends at 2^-16, fp16 at 2^-24: the second term is stored times 2^4, the third times 2^8, which their columns of O take back
// when the piece ends.  What rounding a value below 2^15 leaves is at most 2^11, so no term exceeds 2^15, and the three are P' exactly,
// for every fp16 value of at most 2^15 (the low bits of a subnormal one, too).  The reference is held 2^11 below the
// maximum of the shifted exponents and moves when that grows by 2^4 (P' <= 2^15): a weight loses bits no earlier than 2^-25 of its
// row's largest, with the wide path's 2^7 2^-21; where a page's scale is 1 / r of the largest's, 2^-25 r here, and 2^-21 r for what
// of the scales is in P' there.  (Terms without powers of two of their own kept the bits of weights down to 2^-17: pages of
// different scales side by side were off by three times what the wide path's bound allows.)
// A block of eight 32K prompts takes 900 us the wide way and 797 this way: a group of 128 tokens every 1,350 cycles, which is
// HBM's pace, instead of every 2,000.  With V converted to fp16 here as well (P' as fp16) it was hardly faster than the wide way:
// the conversion and 160 KB per group through shared memory bound it.
// The three sets of softmax warps take every third group as in the wide path, but each has its own O and its own references,
// so nothing passes from group to group; they meet at the end of a piece, where their outputs are merged.  The four warps of a
// set agree on a reference in two steps: one flag per warp, and only if one is raised the maxima over the tokens.
// Same producers and records as the wide path; K and V have rings of group-sized slots; the converting warps have nothing to do.
// Only for d = 128 and shares of a group or more (see attn_tc5_kernel); 32 rows as two blocks of columns spill registers and took
// 852 us for the block where one takes 804.  bf16 pages stay with the wide path: it waits for HBM on sparse steps, and its first group has less code to fetch behind the
// page copies (four steps of eight 32K prompts 435 us wide, 441 this way; eight of one 8K sequence 285 and 284).
#pragma once

// What the roles of a CTA share.
struct Tc5Cta {
  uint8_t* gen;                                  // shared memory from `base` on
  uint32_t base, kring, vring;
  uint32_t kfull, kfree, vfull, vfree, s_full, s_free, p_full, q_full, q_free, o_free;
  uint32_t s_read, meet, piece_meet;             // narrow path only
  volatile int* abort_flag;
  const int *pre, *tok_s, *na_s;
  bool staged;
  float* scratch;                                // the exchange arrays
  volatile int* meta;
  volatile float *kscale_meta, *vlog_meta;
  uint32_t tmem;
  int lo, hi, sg0;
  __device__ __forceinline__ int n_active_of(const AttnParams& p, int s) const { return staged ? na_s[s] : clamp_active(p.n_active[s], p.B); }
  __device__ __forceinline__ int token_of(const AttnParams& p, int s, int a) const { return staged ? tok_s[s * p.B + a] : p.active_idx[s * p.B + a]; }
  __device__ __forceinline__ int rows_of(const AttnParams& p, int sg) const {
    return rows_in_group(n_active_of(p, (sg % p.n_sk) / p.Hkv), p.G, sg / p.n_sk);
  }
};
// tensor-memory columns: S of set h, O of set h
constexpr uint32_t kTc5nColS = 0, kTc5nColO = 128;

// The P' terms: MN-major tile of 8-bit values without a swizzle: blocks of 16 rows kTc5nP bytes apart, within one 16 bytes per token.
__device__ __forceinline__ uint64_t tc5n_desc_p(uint32_t saddr) {
  return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>(128 >> 4) << 16) | (static_cast<uint64_t>(kTc5nP >> 4) << 32) | (1ull << 46);
}
// A V tile as the copies leave it: MN-major rows of 128 codes, swizzled over the row.
__device__ __forceinline__ uint64_t tc5n_desc_v(uint32_t saddr) {
  return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) | (1ull << 16) | (static_cast<uint64_t>(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// two fp32 values per instruction, the roundings of one at a time
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmul.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ void tc5_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\ttcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}

// ---- K Q^T issuer (a warp, one elected lane issues)
template <int D, int GP>
__device__ __forceinline__ void tc5n_issue_qk(const AttnParams& p, const Tc5Cta& c) {
  constexpr int NRK = tc5n_slots<D, GP>(), KSLOT = tc5_kslot_bytes<D, true>(), PG = kTc5Tok / GP, SB = kTc5Sets;
  const uint32_t base = warp_uniform(c.base), kring = warp_uniform(c.kring), s_col0 = warp_uniform(c.tmem) + kTc5nColS;
  const int hi = warp_uniform(c.hi);
  auto wait = [&](uint32_t bar, uint32_t parity) { return warp_mbar_wait(bar, parity, c.abort_flag, p.status, p.wait_cycles); };
  int sg = c.sg0, item = warp_uniform(c.lo), piece = 0, g = 0;
  bool ok = true;
  while (item < hi && ok) {
    const int seg_end = warp_uniform(min(hi, c.pre[sg + 1]));
    ok = wait(c.q_full, piece & 1);
    for (int first = item; first < seg_end && ok; first += PG, ++g) {
      const int b = g % SB, use = g / SB, slot = g % NRK;
      ok = wait(c.kfull + 8 * slot, (g / NRK) & 1);
      ok = ok && (use == 0 || wait(c.s_read + 8 * b, (use - 1) & 1));
      if (!ok) break;
      tc5_fence_after();
      if (elect_one()) {
        const uint32_t kt = kring + slot * KSLOT, s_col = s_col0 + b * kTc5nRows;
        // (all 128 rows of the slot, whatever the group holds: a lane without a token is masked by its softmax thread)
        const uint32_t idesc = tc5_idesc(kTc5Tok, kTc5nRows, 0, 0u, 1u);      // E4M3 codes against the E5M2 terms of Q
        const uint64_t kd = tc5_desc8<D>(kt), qd = tc5_desc8<D>(base);
#pragma unroll
        for (int ks = 0; ks < D / 32; ++ks)
#pragma unroll
          for (int t = 0; t < kTc5QTerms; ++t)
            tc5_mma_ss8(s_col, kd + ks * 2, qd + (t * (kTc5nRows * D) + ks * 32) / 16, idesc, ks + t > 0 ? 1u : 0u);
        tc5_commit(c.s_full + 8 * b);
        tc5_commit(c.kfree + 8 * slot);
        if (first + PG >= seg_end) tc5_commit(c.q_free);
      }
      __syncwarp();
    }
    item = seg_end;
    ++sg;
    ++piece;
    while (item < hi && warp_uniform(c.pre[sg + 1]) <= item) ++sg;
  }
}

// ---- V^T P issuer (a warp, one elected lane issues)
template <int D, int GP>
__device__ __forceinline__ void tc5n_issue_pv(const AttnParams& p, const Tc5Cta& c) {
  constexpr int NRV = tc5n_slots<D, GP>(), SLOT = tc5_kslot_bytes<D, true>(), PG = kTc5Tok / GP, SB = kTc5Sets;
  const uint32_t pbuf = warp_uniform(c.base) + tc5n_q_bytes<D>(), vring = warp_uniform(c.vring), o_col0 = warp_uniform(c.tmem) + kTc5nColO;
  const int hi = warp_uniform(c.hi);
  auto wait = [&](uint32_t bar, uint32_t parity) { return warp_mbar_wait(bar, parity, c.abort_flag, p.status, p.wait_cycles); };
  constexpr uint32_t mn_major_a = 1u << 15;
  const uint32_t idesc = tc5_idesc(128, kTc5PTerms * kTc5nRows, 1, 0u, 1u) | mn_major_a;      // E4M3 codes, E5M2 terms; both MN-major
  int sg = c.sg0, item = warp_uniform(c.lo), piece = 0, g = 0;
  bool ok = true;
  while (item < hi && ok) {
    const int seg_end = warp_uniform(min(hi, c.pre[sg + 1])), g0 = g;
    for (int first = item; first < seg_end && ok; first += PG, ++g) {
      const int ng = min(PG, seg_end - first), b = g % SB, use = g / SB, slot = g % NRV;
      ok = wait(c.vfull + 8 * slot, (g / NRV) & 1);
      if (first == item && piece > 0) ok = ok && wait(c.o_free, (piece - 1) & 1);   // all O have been read
      ok = ok && wait(c.p_full + 8 * b, use & 1);
      if (!ok) break;
      tc5_fence_after();
      if (elect_one()) {
        const uint64_t vd = tc5n_desc_v(vring + slot * SLOT), pd = tc5n_desc_p(pbuf + b * tc5n_p_bytes());
        const uint32_t fresh = g - g0 < SB ? 0u : 1u, o_col = o_col0 + b * (kTc5PTerms * kTc5nRows);
        const int n_ks = (ng * GP + 31) / 32;              // (a last half: P' is zero there, and V has been cleared)
        if (n_ks == kTc5Tok / 32) {
#pragma unroll
          for (int ks = 0; ks < kTc5Tok / 32; ++ks) tc5_mma_ss8(o_col, vd + ks * (32 * D / 16), pd + ks * (512 / 16), idesc, ks == 0 ? fresh : 1u);
        } else {
          for (int ks = 0; ks < n_ks; ++ks) tc5_mma_ss8(o_col, vd + ks * (32 * D / 16), pd + ks * (512 / 16), idesc, ks == 0 ? fresh : 1u);
        }
        tc5_commit(c.vfree + 8 * slot);
        tc5_commit(c.s_free + 8 * b);
      }
      __syncwarp();
    }
    item = seg_end;
    ++sg;
    ++piece;
    while (item < hi && warp_uniform(c.pre[sg + 1]) <= item) ++sg;
  }
}

// Rows of V past the end of the prefix may hold anything (even NaN): a set clears them once the tile has landed, and with them the
// second half of a product's 32 tokens where a group ends between.  The slot's previous tile must have been used first: until
// then its barrier may be a phase behind, with the parity that is waited for.
template <int D, int GP, typename Wait, typename Valid>
__device__ __forceinline__ bool tc5n_clear(const Tc5Cta& c, int g, int ng, int tid_in_set, Wait&& warp_wait, Valid&& valid_of) {
  constexpr int NRV = tc5n_slots<D, GP>(), SLOT = tc5_kslot_bytes<D, true>();
  const int slot = g % NRV;
  if (g >= NRV && !warp_wait(c.vfree + 8 * slot, (g / NRV - 1) & 1)) return false;
  if (!warp_wait(c.vfull + 8 * slot, (g / NRV) & 1)) return false;
  uint8_t* vg = c.gen + (c.vring - c.base) + slot * SLOT;
  const int end = (ng * GP + 31) / 32 * 32;                // whole rows: the swizzle stays within one
  for (int idx = tid_in_set; idx < end * (D / 16); idx += kTc5SetWarps * 32) {
    const int t = idx / (D / 16), j = t / GP;
    if (j >= ng || t % GP >= valid_of(j)) *reinterpret_cast<uint4*>(vg + idx * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  return true;
}

// ---- softmax / epilogue warps
// decide(): waits until the path is known, false if it is not this one (or the wait has run out).
// The last set first takes a group that is not there, before the path is known: no waits for other roles, no arrivals, no token
// live, so that nothing changes.  The other sets may be on the wide path by then, at the end of a short first piece even: what
// this set writes of the exchange arrays lies behind all that path has there.  It fetches the loop's instructions while the producers still look for their first pages.  Behind
// the page copies every missed line of them takes 400 cycles and more: the first groups' maxima and weights took 7,300 cycles,
// with the rings full and HBM idle (a block of eight 32K prompts 11 us longer).
template <int D, int GP, typename Decide>
__device__ __forceinline__ void tc5n_softmax(const AttnParams& p, const Tc5Cta& c, Decide&& decide) {
  constexpr int PG = kTc5Tok / GP, MR = kTc5MetaRing, SB = kTc5Sets, NW = kTc5SoftmaxWarps;
  constexpr int OC = kTc5PTerms * kTc5nRows;                    // columns of a set's O
  const __nv_bfloat16* q = static_cast<const __nv_bfloat16*>(p.q);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, quarter = warp & 3, h = warp >> 2;
  const uint32_t lane_addr = c.tmem + (static_cast<uint32_t>(quarter * 32) << 16);
  const uint32_t s_addr = lane_addr + kTc5nColS + h * kTc5nRows, o_addr = lane_addr + kTc5nColO + h * OC;
  uint8_t* ptile = c.gen + tc5n_q_bytes<D>() + h * tc5n_p_bytes();
  // The exchange arrays, in entries from c.scratch on: those of the first two sets, of a piece, of the last set.  (c.scratch is at most three
  // entries behind the wide path's first.)
  constexpr int kSetRefs = 2 * kTc5SetWarps * kTc5nLanes, kSet = kSetRefs + kTc5SetWarps * kTc5nLanes;     // of one set
  constexpr int kSums = (SB - 1) * kSet, kRefs = kSums + 2 * NW * kTc5nLanes, kScale = kRefs + 2 * SB * kTc5nLanes;
  constexpr int kLast = kTc5Xchg, kFlags = kLast + kSet;         // written by the walk without a group
  static_assert(kScale + 2 * kTc5nLanes <= kLast && kLast >= kTc5Xchg, "the last set's entries: behind the others' and the wide path's");
  static_assert(kFlags * 4 + SB * 8 + 3 * 4 <= tc5_xchg_bytes<true>(), "exchange arrays");
  float* own = c.scratch + (h == SB - 1 ? kLast : h * kSet);
  // Per row, a copy per warp: minus the reference maximum, +inf while there is none; the same with 0 for none.
  float* neg_m = own + quarter * 2 * kTc5nLanes;                 // [4][2][32]
  float* neg_use = neg_m + kTc5nLanes;
  float* wmax = own + kSetRefs;                                  // [4][32] maxima over a warp's tokens
  float* xsum = c.scratch + kSums;                               // [piece parity][12][32] row sums of a piece over a warp's tokens ...
  float* xref = c.scratch + kRefs;                               // [piece parity][3][32]  ... and the references they are relative to
  float* qscale = c.scratch + kScale;                            // [piece parity][32] softmax scale times what undoes the row's power of two
  volatile uint8_t* flags = reinterpret_cast<volatile uint8_t*>(c.scratch + kFlags);        // [3][meeting parity][4]
  auto warp_wait = [&](uint32_t bar, uint32_t parity) {         // one answer for the warp: tensor-memory instructions need all lanes
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, c.abort_flag, p.status, p.wait_cycles)) != 0;
  };
  int meetings = 0;
  auto set_meets = [&]() {                                      // the four warps of the set
    __syncwarp();
    if (lane == 0) mbar_arrive(c.meet + 8 * h, 1);
    return warp_wait(c.meet + 8 * h, meetings++ & 1);
  };
  const float scale2 = p.sm_scale * kLog2e;
  int sg = c.sg0, item = c.lo, piece = 0, g = 0;
  int dry = h == SB - 1;
  bool ok = dry || decide();
  while (item < c.hi && ok) {
    asm volatile("" : "+r"(dry));                              // (one copy of the code)
    const int seg_end = min(c.hi, c.pre[sg + 1]);
    const int rg = sg / p.n_sk, sk = sg % p.n_sk, s = sk / p.Hkv, kh = sk % p.Hkv;
    const int rows = c.rows_of(p, sg), g0 = g;
    float* qs = qscale + (piece & 1) * kTc5nLanes;
    // ---- the piece's Q tile: a warp per row, of the first two sets
    neg_m[lane] = INFINITY;
    neg_use[lane] = 0.f;
    __syncwarp();
    if (h < 2) {
      static_assert(D == 128, "M of the second product");
      constexpr int QW = 2 * kTc5SetWarps, EL = D / 32, RPW = kTc5nRows / QW;      // warps, elements per lane, rows per warp
      uint32_t raw[RPW][EL / 2];
#pragma unroll
      for (int i = 0; i < RPW; ++i) {
        const int r = warp + QW * i;
#pragma unroll
        for (int e = 0; e < EL / 2; ++e) raw[i][e] = 0u;
        if (r < rows) {
          const int row = rg * kRowsPerGroup + r, a = row / p.G, gi = row % p.G;
          int tok = c.token_of(p, s, a);
          if (tok < 0 || tok >= p.B) { set_status(p.status, LOSA_ERR_BOUNDS); tok = 0; }
          const __nv_bfloat16* src = q + ((static_cast<size_t>(s) * p.B + tok) * p.Hq + kh * p.G + gi) * D + lane * EL;
          const uint2 v = __ldg(reinterpret_cast<const uint2*>(src));
          raw[i][0] = v.x;
          raw[i][1] = v.y;
        }
      }
      if (piece > 0) ok = warp_wait(c.q_free, (piece - 1) & 1);
      if (!ok) break;
#pragma unroll
      for (int i = 0; i < RPW; ++i) {
        const int r = warp + QW * i;
        {                                                       // (rows without a query are zero)
          // three E5M2 terms under the power of two that brings the row's largest element to 2^15 .. 2^16 (see attn_tc5_kernel)
          uint32_t top = 0;
#pragma unroll
          for (int e = 0; e < EL / 2; ++e) top = max(top, max((raw[i][e] << 16) & 0x7fffffffu, raw[i][e] & 0x7fff0000u));
          top = __reduce_max_sync(0xffffffffu, top);
          const int e_top = max(static_cast<int>(top >> 23), 16), up = 142 - e_top, u0 = up / 2, u1 = up - u0;
          const float f0 = __int_as_float((127 + u0) << 23), f1 = __int_as_float((127 + u1) << 23);
          float sc = scale2 * (__int_as_float((127 - u0) << 23) * __int_as_float((127 - u1) << 23));
          if ((top >> 23) == 255) sc = __int_as_float(top);
          if (lane == 0) qs[r] = sc;
          uint32_t w[kTc5QTerms][EL / 2];
#pragma unroll
          for (int e = 0; e < EL / 2; ++e) {
            float2 v = make_float2(__uint_as_float(raw[i][e] << 16) * f0 * f1, __uint_as_float(raw[i][e] & 0xffff0000u) * f0 * f1);
#pragma unroll
            for (int t = 0; t < kTc5QTerms; ++t) {
              w[t][e] = __nv_cvt_float2_to_fp8x2(v, __NV_SATFINITE, __NV_E5M2);
              const float2 part = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(w[t][e]), __NV_E5M2)));
              v.x -= part.x;
              v.y -= part.y;
            }
          }
          uint8_t* dst = c.gen + tc5_sw8<D>(r, lane * EL / 16) + lane * EL % 16;
#pragma unroll
          for (int t = 0; t < kTc5QTerms; ++t) *reinterpret_cast<uint32_t*>(dst + t * (kTc5nRows * D)) = w[t][0] | w[t][1] << 16;
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read the tile through the async proxy
      __syncwarp();
      if (lane == 0) mbar_arrive(c.q_full, h == 0 ? 2 : 1);            // (the last set's arrivals with the first's)
    }
    const int parity = piece & 1;                               // of the exchange buffers
    float l[kTc5nRows];                                       // this thread's weights
#pragma unroll
    for (int n = 0; n < kTc5nRows; ++n) l[n] = 0.f;
    int first = item;
    g = g0;
#pragma unroll 1
    while (true) {
      if (!dry) {
        while (first < seg_end && g % SB != h) { first += PG; ++g; }    // the set's next group
        if (first >= seg_end) break;
      }
      const int ng = min(PG, seg_end - first), use = g / SB;
      const uint32_t s_at = dry ? lane_addr + kTc5nColO + SB * OC : s_addr;      // (dry: columns nobody writes)
      volatile int* gmeta = c.meta + (g % MR) * PG;
      auto valid_of = [&](int j) { return gmeta[j] & 0xff; };
      if (!dry) ok = warp_wait(c.s_full + 8 * h, use & 1);
      if (!ok) break;
      tc5_fence_after();
      const bool to_clear = !dry && (__any_sync(0xffffffffu, lane < ng && valid_of(min(lane, PG - 1)) < GP) != 0 || (ng * GP & 31) != 0);
      const int t = quarter * 32 + lane, j = min(t / GP, ng - 1), at = (g % MR) * PG + j;      // this thread's token and its page
      const bool live = !dry && t / GP < ng && t % GP < valid_of(j);
      const float ks = c.kscale_meta[at], vlog = c.vlog_meta[at];
      const float2 ks2 = make_float2(ks, ks), vlog2 = make_float2(vlog, vlog);
      // exponents of P' of columns n .. n + 3 from the scores v, under references taken from `neg`
      auto exponents = [&](const float* neg, int n, const uint32_t* v, float2 (&y)[2]) {
        const float4 a = *reinterpret_cast<const float4*>(qs + n), m = *reinterpret_cast<const float4*>(neg + n);
        y[0] = fma2(mul2(make_float2(__uint_as_float(v[0]), __uint_as_float(v[1])), ks2), make_float2(a.x, a.y), add2(make_float2(m.x, m.y), vlog2));
        y[1] = fma2(mul2(make_float2(__uint_as_float(v[2]), __uint_as_float(v[3])), ks2), make_float2(a.z, a.w), add2(make_float2(m.z, m.w), vlog2));
      };
      // ---- has a score outgrown its row's reference?  (No reference yet: yes.)
      bool moved = true;
      if (dry || g - g0 >= SB) {
        bool grown = false;
        uint32_t v[16];
        tc5_ld16(s_at, v);
#pragma unroll
        for (int e = 0; e < 16; e += 4) {
          float2 y[2];
          exponents(neg_m, e, v + e, y);
          grown |= !(y[0].x <= kTc5nTop) | !(y[0].y <= kTc5nTop) | !(y[1].x <= kTc5nTop) | !(y[1].y <= kTc5nTop);
        }
        const bool flag = __any_sync(0xffffffffu, grown && live) != 0;
        volatile uint8_t* f = flags + (2 * h + (meetings & 1)) * 4;
        if (lane == 0) f[quarter] = flag ? 1 : 0;
        ok = set_meets();
        if (!ok) break;
        moved = dry || *reinterpret_cast<volatile uint32_t*>(f) != 0;
      }
      if (!dry && use > 0) ok = warp_wait(c.s_free + 8 * h, (use - 1) & 1);      // the set's last P V has run: P' may be written, O changed
      if (!ok) break;
      tc5_fence_after();
      if (moved) {
        float mine = -INFINITY;                                 // lane n: row n's maximum over the tokens of this warp
#pragma unroll 1
        for (int n = 0; n < kTc5nRows; n += 8) {
          uint32_t v[8];
          tc5_ld8(s_at + n, v);
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float y = live ? fmaf(__uint_as_float(v[e]) * ks, qs[n + e], vlog) : -INFINITY;
            float k;                                            // (as fmaxf: a NaN among the tokens does not count)
            asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(k) : "f"(y));
            if (lane == n + e) mine = k;
          }
        }
        wmax[quarter * kTc5nLanes + lane] = mine;
        ok = set_meets();
        if (!ok) break;
        const float* wm = wmax + lane;
        const float top = fmaxf(fmaxf(wm[0], wm[kTc5nLanes]), fmaxf(wm[2 * kTc5nLanes], wm[3 * kTc5nLanes]));
        const float m_old = -neg_m[lane];
        const float m_new = (top > m_old + kTc5nTop || (m_old == -INFINITY && top > -INFINITY)) ? top - kTc5nLift : m_old;
        __syncwarp();
        neg_m[lane] = -m_new;
        neg_use[lane] = m_new == -INFINITY ? 0.f : -m_new;
        __syncwarp();
        if (!dry && g - g0 >= SB) {                             // O holds this set's earlier groups, l their weights
          const float corr = m_old == m_new ? 1.f : (m_old == -INFINITY ? 0.f : ex2(m_old - m_new));
#pragma unroll 1
          for (int x = 0; x < kTc5PTerms; ++x) {
            uint32_t w[16];
            tc5_ld16(o_addr + 16 * x, w);
#pragma unroll
            for (int e = 0; e < 16; ++e) w[e] = __float_as_uint(__uint_as_float(w[e]) * __shfl_sync(0xffffffffu, corr, e));
            tc5_st16(o_addr + 16 * x, w);
          }
          tc5_wait_st();
#pragma unroll
          for (int e = 0; e < 16; ++e) l[e] *= __shfl_sync(0xffffffffu, corr, e);
        }
      }
      // ---- P' = 2^(s + vlog - m), its sum without the value scale, its three terms
      const float unscale = ex2(-vlog);
      {
        uint32_t v[8], w[kTc5PTerms][4];                          // (the scores in two halves: all 16 spill registers)
#pragma unroll
        for (int e = 0; e < 16; e += 4) {
          if (e % 8 == 0) tc5_ld8(s_at + e, v);
          float2 y[2];
          exponents(neg_use, e, v + e % 8, y);
          y[0] = make_float2(ex2(y[0].x), ex2(y[0].y));
          y[1] = make_float2(ex2(y[1].x), ex2(y[1].y));
          if (live) {                                           // (a lane without a token holds anything)
            const float2 u2 = make_float2(unscale, unscale);
            const float2 l0 = fma2(y[0], u2, make_float2(l[e], l[e + 1])), l1 = fma2(y[1], u2, make_float2(l[e + 2], l[e + 3]));
            l[e] = l0.x; l[e + 1] = l0.y; l[e + 2] = l1.x; l[e + 3] = l1.y;
          }
          uint32_t p0 = live ? pack_f16(y[0].x, y[0].y) : 0u, p1 = live ? pack_f16(y[1].x, y[1].y) : 0u;
#pragma unroll
          for (int k = 0; k < kTc5PTerms; ++k) {                // the nearest multiple of the upper byte's last place, ties away from zero; the rest, times 2^4
            const uint32_t r0 = p0 + 0x00800080u, r1 = p1 + 0x00800080u;
            w[k][e / 4] = __byte_perm(r0, r1, 0x7531);
            if (k + 1 < kTc5PTerms) {
              const uint32_t t0 = r0 & 0xff00ff00u, t1 = r1 & 0xff00ff00u;
              const __half2 up = __float2half2_rn(1.f / kTc5nTermStep);
              const __half2 d0 = __hmul2(__hsub2(*reinterpret_cast<const __half2*>(&p0), *reinterpret_cast<const __half2*>(&t0)), up);
              const __half2 d1 = __hmul2(__hsub2(*reinterpret_cast<const __half2*>(&p1), *reinterpret_cast<const __half2*>(&t1)), up);
              p0 = *reinterpret_cast<const uint32_t*>(&d0);
              p1 = *reinterpret_cast<const uint32_t*>(&d1);
            }
          }
        }
#pragma unroll
        for (int k = 0; k < kTc5PTerms; ++k)
          if (!dry) *reinterpret_cast<uint4*>(ptile + k * kTc5nP + t * 16) = make_uint4(w[k][0], w[k][1], w[k][2], w[k][3]);
      }
      if (to_clear && !tc5n_clear<D, GP>(c, g, ng, threadIdx.x & 127, warp_wait, valid_of)) { ok = false; break; }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc5_fence_before();
      __syncwarp();
      if (dry) break;
      if (lane == 0) {
        mbar_arrive(c.s_read + 8 * h, 1);
        mbar_arrive(c.p_full + 8 * h, 1);
      }
      first += PG;
      ++g;
    }
    if (!ok) break;
    if (dry) {
      dry = 0;
      g = 0;
      ok = decide();
      continue;
    }
    const int n_groups = (seg_end - item + PG - 1) / PG;
    g = g0 + n_groups;
    // the row sums over the warp's tokens, lane n left with row n (every step halves the rows a lane still adds for)
#pragma unroll
    for (int n = 0; n < 16; ++n) l[n] += __shfl_xor_sync(0xffffffffu, l[n], 16);
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) {
      const bool up = (lane & off) != 0;
#pragma unroll
      for (int n = 0; n < off; ++n) {
        const float keep = up ? l[n + off] : l[n], give = up ? l[n] : l[n + off];
        l[n] = keep + __shfl_xor_sync(0xffffffffu, give, off);
      }
    }
    const float row_sum = l[0];
    // ---- the piece's record: the sets' outputs under a common reference.  A set waits for its own last P V, then all meet.
    auto used = [&](int x) { return (x + SB - g0 % SB) % SB < n_groups; };      // set x handled a group of the piece
    if (used(h)) {
      const int last = g - 1 - (g - 1 + SB - h) % SB;
      ok = warp_wait(c.s_free + 8 * h, (last / SB) & 1);
      if (!ok) break;
    }
    xsum[(parity * NW + warp) * kTc5nLanes + lane] = row_sum;
    if (quarter == 0) xref[(parity * SB + h) * kTc5nLanes + lane] = -neg_m[lane];
    tc5_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(c.piece_meet, 1);
    ok = warp_wait(c.piece_meet, piece & 1);
    if (!ok) break;
    tc5_fence_after();
    float w[SB], M = -INFINITY, L = 0.f;                      // lane n: of row n
#pragma unroll
    for (int x = 0; x < SB; ++x) {
      w[x] = xref[(parity * SB + x) * kTc5nLanes + lane];
      M = fmaxf(M, w[x]);
    }
#pragma unroll
    for (int x = 0; x < SB; ++x) {
      w[x] = w[x] == -INFINITY ? 0.f : ex2(w[x] - M);
      const float* xs = xsum + (parity * NW + x * kTc5SetWarps) * kTc5nLanes + lane;
      const float sum = (xs[0] + xs[kTc5nLanes]) + (xs[2 * kTc5nLanes] + xs[3 * kTc5nLanes]);
      if (w[x] > 0.f || sum != sum) L = fmaf(sum, w[x], L);
    }
    if (warp == 0 && lane < rows) {
      float* rec = record_base(p.partials, blockIdx.x + sg, lane / kTileRows, D);
      rec[lane % kTileRows] = M;
      rec[kTileRows + lane % kTileRows] = L;
    }
    const int d = quarter * 32 + lane;
#pragma unroll 1
    for (int n0 = 8 * h; n0 < rows; n0 += 8 * SB) {       // eight rows at a time, dealt out to the sets
      float acc[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] = 0.f;
#pragma unroll
      for (int x = 0; x < SB; ++x) {
        if (!used(x)) continue;
        uint32_t o[kTc5PTerms][8];
#pragma unroll
        for (int k = 0; k < kTc5PTerms; ++k) tc5_ld8(lane_addr + kTc5nColO + x * OC + k * kTc5nRows + n0, o[k]);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float wx = __shfl_sync(0xffffffffu, w[x], n0 + e);
          const float sum = fmaf(fmaf(__uint_as_float(o[2][e]), kTc5nTermStep, __uint_as_float(o[1][e])), kTc5nTermStep, __uint_as_float(o[0][e]));
          if (wx > 0.f) acc[e] = fmaf(sum, wx, acc[e]);
        }
      }
      {
        // a weight that is no number has no term (its rounding ends at zero), but spoils the row's sum: that goes into the outputs
        float* rec = record_base(p.partials, blockIdx.x + sg, n0 / kTileRows, D) + 2 * kTileRows + d;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float row_l = __shfl_sync(0xffffffffu, L, n0 + e);
          if (n0 + e < rows) rec[(n0 % kTileRows + e) * D] = row_l == row_l ? acc[e] : row_l;
        }
      }
    }
    tc5_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(c.o_free, 1);
    item = seg_end;
    ++sg;
    ++piece;
    while (item < c.hi && c.pre[sg + 1] <= item) ++sg;
  }
}
