// In-block attention on the tensor cores, bf16: the work of one CTA (stage 5's kernel in block_cache.cu;
// in a whole step the tail of the candidate refinement's grid in page_select.cu).
#pragma once
#include <type_traits>

#include "kernels.h"

namespace losa {
namespace {

// ---- in-block attention of the whole-step path on the tensor cores (bf16) ---------------------
// The in-block part is a small dense contraction (B keys, all B * G rows of a KV head), and in a whole
// step it runs beside the candidate refinement, where every cycle it holds an SM delays it: mma.sync
// tiles cut its instruction count by more than an order of magnitude against CUDA-core code.
// CTA = 64 query rows of one (sequence, KV head) (row = block token * G + head of the group), one
// warp per 16 rows.  K_b [key][d] and V_b transposed [d][key] are staged in shared memory as bf16
// (rows padded by 16 bytes: the fragment reads are conflict-free); Q fragments come straight from
// global memory.  S = Q K_b^T in fp32 accumulators, softmax in registers (row statistics over the
// four lanes that share a row), P rounded to bf16 as in stage 4, O = P V_b in fp32, normalised by
// the fp32 sum.  BK = B rounded up to 32 or 64; keys >= B are masked, their V rows zero.
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack2_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

constexpr int kMmaRows = 64;       // query rows per CTA
constexpr int kMmaThreads = 128;

template <int D, int BK>
struct BlockAttnSmem {
  static constexpr int KS = D + 8;   // padded row of K_b (elements)
  static constexpr int VS = BK + 8;  // padded row of V_b^T
  __nv_bfloat16 k[BK * KS];
  __nv_bfloat16 vt[D * VS];
};

struct BlockAttnParams {
  const __nv_bfloat16* q;
  const __nv_bfloat16* k_blk;
  const __nv_bfloat16* v_blk;
  const void* o_p;               // MERGE only
  int o_p_bf16;
  const float* lse_p;
  __nv_bfloat16* out;
  float* lse_out;
  float* ob_out;                 // !MERGE only
  int B, Hq, Hkv;
  float sm_scale;
};

// MERGE = true (stage 5 of the six-call path): the in-block part is merged with the prefix
// statistics by log-sum-exp and the attention output is written (Section 2.2 / 4.3); MERGE = false
// (whole-step path): the normalised in-block part goes to `ob_out` and L_b to `lse_out`.
// Row tile rt (64 rows) of (sequence s, KV head kh), by the kMmaThreads threads of a CTA.  CW: columns of O
// per pass.  All D at once is the faster way (K_b V_b and o_p are requested once); 64 take 32 registers
// less, which the refinement's CTAs do not have.
template <int D, int BK, bool MERGE, int CW>
__device__ __forceinline__ void block_attn_mma_cta(const BlockAttnParams& p, BlockAttnSmem<D, BK>& sm, int rt, int kh, int s) {
  const int B = p.B, Hq = p.Hq, Hkv = p.Hkv;
  const float sm_scale = p.sm_scale;
  constexpr int KS = BlockAttnSmem<D, BK>::KS, VS = BlockAttnSmem<D, BK>::VS;
  constexpr int NT = BK / 8;         // key tiles of S
  constexpr int NO = CW / 8;         // column tiles of O per pass
  __nv_bfloat16* Ks = sm.k;
  __nv_bfloat16* Vt = sm.vt;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = Hq / Hkv, nrow = B * G;
  // ---- this warp's 16 rows: rows g and g + 8 of the tile for this lane; the queries are
  //      requested before the staging's stores, which the compiler cannot tell apart from these loads
  const int g = lane >> 2, t4 = lane & 3;
  const int lr0 = rt * kMmaRows + warp * 16 + g, lr1 = lr0 + 8;
  auto global_row = [&](int lr) {
    const int c = min(lr, nrow - 1);
    return (static_cast<size_t>(s) * B + c / G) * Hq + kh * G + c % G;
  };
  const size_t gr0 = global_row(lr0), gr1 = global_row(lr1);
  const uint32_t* q0 = reinterpret_cast<const uint32_t*>(p.q + gr0 * D);
  const uint32_t* q1 = reinterpret_cast<const uint32_t*>(p.q + gr1 * D);
  uint32_t qa[D / 16][4];
#pragma unroll
  for (int ks = 0; ks < D / 16; ++ks) {
    qa[ks][0] = q0[ks * 8 + t4];
    qa[ks][1] = q1[ks * 8 + t4];
    qa[ks][2] = q0[ks * 8 + 4 + t4];
    qa[ks][3] = q1[ks * 8 + 4 + t4];
  }
  // ---- stage K_b (row-major) and V_b (transposed); keys >= B are zero
  for (int idx = tid; idx < BK * (D / 8); idx += kMmaThreads) {
    const int t = idx % BK, ch = idx / BK;             // key fastest: the transposed stores of a warp fall into one row
    uint4 kv = make_uint4(0u, 0u, 0u, 0u), vv = kv;
    if (t < B) {
      const size_t src = ((static_cast<size_t>(s) * B + t) * Hkv + kh) * D + ch * 8;
      kv = *reinterpret_cast<const uint4*>(p.k_blk + src);
      vv = *reinterpret_cast<const uint4*>(p.v_blk + src);
    }
    *reinterpret_cast<uint4*>(Ks + t * KS + ch * 8) = kv;
    const __nv_bfloat16* ve = reinterpret_cast<const __nv_bfloat16*>(&vv);
#pragma unroll
    for (int e = 0; e < 8; ++e) Vt[(ch * 8 + e) * VS + t] = ve[e];
  }
  __syncthreads();
  if (rt * kMmaRows + warp * 16 >= nrow) return;       // no row of this warp exists
  // ---- S = Q K_b^T
  float sc[NT][4];
#pragma unroll
  for (int j = 0; j < NT; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) sc[j][e] = 0.f;
#pragma unroll
  for (int ks = 0; ks < D / 16; ++ks) {
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const uint32_t* kr = reinterpret_cast<const uint32_t*>(Ks + (8 * j + g) * KS + 16 * ks);
      mma_bf16_16816(sc[j], qa[ks], kr[t4], kr[4 + t4]);
    }
  }
  // ---- softmax over the keys (natural exponent; the log-normaliser is exported in natural units)
  float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
  for (int j = 0; j < NT; ++j) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int key = 8 * j + 2 * t4 + (e & 1);
      sc[j][e] = key < B ? sc[j][e] * sm_scale : -INFINITY;
    }
    m0 = fmaxf(m0, fmaxf(sc[j][0], sc[j][1]));
    m1 = fmaxf(m1, fmaxf(sc[j][2], sc[j][3]));
  }
  m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, 1));
  m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, 2));
  m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, 1));
  m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, 2));
  float l0 = 0.f, l1 = 0.f;
  uint32_t pa[NT][2];                // P as bf16 pairs: [j][0] row g, [j][1] row g + 8
#pragma unroll
  for (int j = 0; j < NT; ++j) {
    const float p0 = expf(sc[j][0] - m0), p1 = expf(sc[j][1] - m0);
    const float p2 = expf(sc[j][2] - m1), p3 = expf(sc[j][3] - m1);
    l0 += p0 + p1;
    l1 += p2 + p3;
    pa[j][0] = pack2_bf16(p0, p1);
    pa[j][1] = pack2_bf16(p2, p3);
  }
  l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
  l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
  // ---- O = P V_b
  const float Lb0 = m0 + logf(l0), Lb1 = m1 + logf(l1);
#pragma unroll
  for (int j0 = 0; j0 < D / 8; j0 += NO) {
    float o[NO][4];
#pragma unroll
    for (int jn = 0; jn < NO; ++jn)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[jn][e] = 0.f;
#pragma unroll
    for (int kk = 0; kk < BK / 16; ++kk) {
      const uint32_t a[4] = {pa[2 * kk][0], pa[2 * kk][1], pa[2 * kk + 1][0], pa[2 * kk + 1][1]};
#pragma unroll
      for (int jn = 0; jn < NO; ++jn) {
        const uint32_t* vr = reinterpret_cast<const uint32_t*>(Vt + (8 * (j0 + jn) + g) * VS + 16 * kk);
        mma_bf16_16816(o[jn], a, vr[t4], vr[4 + t4]);
      }
    }
    // rows g (accumulator halves 0, 1) and g + 8 (halves 2, 3)
    auto finish_row = [&](int lr, size_t gr, float Lb, float l, int e0) {
      if (lr >= nrow) return;
      const size_t at = gr * D + 8 * j0 + 2 * t4;
      if (MERGE) {
        const float Lp = p.lse_p[gr];
        const float M2 = fmaxf(Lp, Lb);
        const float L = M2 + logf(expf(Lp - M2) + expf(Lb - M2));
        const float wp = expf(Lp - L), wb = expf(Lb - L) / l;
        // the cached prefix output as it is stored (fp32 or bf16); all of it is requested before the first store,
        // which the compiler cannot tell apart from these loads (stage 5 in a graph: 5.7 us, one by one 11.7)
        float2 pv[NO];
        if (p.o_p_bf16) {
#pragma unroll
          for (int jn = 0; jn < NO; ++jn) pv[jn] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(static_cast<const __nv_bfloat16*>(p.o_p) + at + 8 * jn));
        } else {
#pragma unroll
          for (int jn = 0; jn < NO; ++jn) pv[jn] = *reinterpret_cast<const float2*>(static_cast<const float*>(p.o_p) + at + 8 * jn);
        }
#pragma unroll
        for (int jn = 0; jn < NO; ++jn) {
          const float x = (wp > 0.f ? wp * pv[jn].x : 0.f) + wb * o[jn][e0];
          const float y = (wp > 0.f ? wp * pv[jn].y : 0.f) + wb * o[jn][e0 + 1];
          *reinterpret_cast<__nv_bfloat162*>(p.out + at + 8 * jn) = __floats2bfloat162_rn(x, y);
        }
        if (j0 == 0 && p.lse_out && t4 == 0) p.lse_out[gr] = L;
      } else {
        const float inv = 1.f / l;
#pragma unroll
        for (int jn = 0; jn < NO; ++jn)
          *reinterpret_cast<float2*>(p.ob_out + at + 8 * jn) = make_float2(o[jn][e0] * inv, o[jn][e0 + 1] * inv);
        if (j0 == 0 && t4 == 0) p.lse_out[gr] = Lb;
      }
    };
    finish_row(lr0, gr0, Lb0, l0, 0);
    finish_row(lr1, gr1, Lb1, l1, 2);
  }
}

// the in-block part alone, into the workspace
inline BlockAttnParams block_attn_params(losa_ctx* c, const void* q, const void* k_blk, const void* v_blk) {
  const losa_shape_t& sh = c->shape;
  BlockAttnParams p = {};
  p.q = static_cast<const __nv_bfloat16*>(q);
  p.k_blk = static_cast<const __nv_bfloat16*>(k_blk);
  p.v_blk = static_cast<const __nv_bfloat16*>(v_blk);
  p.B = sh.block_size;
  p.Hq = sh.n_q_heads;
  p.Hkv = sh.n_kv_heads;
  p.sm_scale = sh.sm_scale;
  p.lse_out = reinterpret_cast<float*>(c->ws + c->lay.block_lse);
  p.ob_out = reinterpret_cast<float*>(c->ws + c->lay.block_o);
  return p;
}

inline int block_attn_tiles(const losa_shape_t& sh) {       // row tiles of a (sequence, KV head)
  return (sh.block_size * (sh.n_q_heads / sh.n_kv_heads) + kMmaRows - 1) / kMmaRows;
}

// f(D, BK) with the kernel's head dimension and padded key count as compile-time constants
template <typename F>
inline void with_block_attn_shape(const losa_shape_t& sh, F&& f) {
  using std::integral_constant;
  const bool wide = sh.block_size > 32;
  if (sh.head_dim == 128) {
    if (wide) f(integral_constant<int, 128>{}, integral_constant<int, 64>{});
    else f(integral_constant<int, 128>{}, integral_constant<int, 32>{});
  } else {
    if (wide) f(integral_constant<int, 64>{}, integral_constant<int, 64>{});
    else f(integral_constant<int, 64>{}, integral_constant<int, 32>{});
  }
}

}  // namespace
}  // namespace losa
