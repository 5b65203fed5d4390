// Stage 4, fp32, CUDA cores: included by sparse_prefix_attn.cu (same namespace; the flat work
// decomposition, the partial-record format and the combine kernel are described there).
//
// Shared-memory bandwidth bounds a CUDA-core attention (a 16-byte read per lane takes the SM four cycles,
// in which it could do four warp-wide FMAs), so both products are tiled in registers:
//   S = Q K^T   the query rows stay in registers for the whole piece.  Lane (rs, dg) holds d elements
//               dg*4 + 32 i .. +3 of rows rs + 4 j, reads 16 bytes of a key per JM rows x 4 elements, and the
//               partial dots are reduce-scattered over the eight dg lanes.
//   O += P V    a thread keeps 8 rows x 8 columns (16 rows x 4) and reads P and V once for them
// Two kinds of piece:
//   up to 16 rows (sparse steps): every warp streams tokens of its own, eight at a time, through its own ring of
//               cp.async copies, with its own softmax state for all the rows; no barrier, and the warps meet
//               when the piece's record is written.  A sparse step of three active tokens 35 -> 23 us.
//   more rows   tiles of 32 tokens through a ring of three slots for the whole CTA.  A warp works on 32 rows;
//               with NB = 1, 2, 4 blocks of 32 rows the tokens of a tile are shared by 8 / NB warps in the first
//               product and 4 / NB in the second (their sums meet when the record is written).  P goes
//               through shared memory; two barriers per tile.  Dense step of two prompts of 4096 and 2875
//               tokens, 32 / 8 heads x 128: 126 us.
#pragma once

constexpr int kF32Threads = 256, kF32Warps = 8;
constexpr int kF32Tok = 32;         // tokens per tile
constexpr int kF32Stages = 3;
constexpr int kF32Chunk = 256;      // pages whose numbers are resolved at once

// CTAs that share the list of T pages: at least 64 tokens each (a CTA's start-up costs more than their
// arithmetic, and every further CTA is another record for the combine kernel to merge one after the
// other: 64 pages of 16 tokens as 64 records took that kernel 25 us, as 16 records 5.8 us).
__device__ __forceinline__ int f32_ctas(int T, int n_ctas, int page) {
  if (T >= 64 * n_ctas) return n_ctas;
  return min(n_ctas, max(1, (T * page + 63) / 64));
}

constexpr int kF32Few = 16;         // rows of a piece whose tokens are dealt out to the warps
constexpr int kF32WTok = 8;         // tokens a warp takes at a time there (at most a page)

template <int D> struct F32Tiles {
  float k[kF32Stages][kF32Tok * D];
  float v[kF32Stages][kF32Tok * D];     // k and v together hold the partial outputs when a piece ends
  float p[kF32Tok * kRowsPerGroup];     // [token][row position]
  float red[kF32Warps * 32];
  float corr[kRowsPerGroup];
};
template <int D> struct F32Warps {
  float kv[kF32Warps][kF32Stages][2][kF32WTok * D];   // K and V; the warps' outputs when a piece ends
  float p[kF32Warps][kF32WTok * kF32Few];             // [token][row]
  float corr[kF32Warps][kF32Few];
  float m[kF32Warps][kF32Few], l[kF32Warps][kF32Few];
};
template <int D> struct F32Smem {
  union { F32Tiles<D> t; F32Warps<D> w; };
  int phys[kF32Chunk], valid[kF32Chunk];
  int pre[kMaxSegments + 1];
  uint32_t ubits[kUnionWords];
  uint16_t ubefore[kUnionWords];
  __device__ __forceinline__ UnionBits lists(int W) { return UnionBits{ubits, ubefore, W}; }
};

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<unsigned long long&>(r))
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)),
        "l"(reinterpret_cast<unsigned long long&>(c)));
  return r;
}
__device__ __forceinline__ void cp_async16_or_zero(uint32_t dst, const void* src, bool full) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(full ? 16 : 0) : "memory");
}
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Pages c0 .. c0 + n - 1 of list sk (n <= kF32Chunk): physical page and number of valid tokens; the caller synchronises.
// BITS, here and below: the lists are page bitmaps (whole step).  A kernel of its own: with the choice at run time the dense pass
// over lists (4,096 + 2,875 tokens, 128 rows) took 114 us instead of 111.
template <int D, int GP, bool BITS>
__device__ __forceinline__ void f32_resolve(const AttnParams& p, F32Smem<D>& sm, int sk, int c0, int n, int len) {
  const int tid = threadIdx.x, s = sk / p.Hkv;
  if (tid < n) {
    const int page = BITS ? sm.lists(p.W).page(sk, c0 + tid) : p.union_pages[static_cast<size_t>(sk) * p.Pmax + c0 + tid];
    bool ok = page >= 0 && page < p.Pmax;
    const int phys = ok ? p.page_table[static_cast<size_t>(s) * p.Pmax + page] : 0;
    ok = ok && phys >= 0 && phys < p.n_phys;
    const int valid = ok ? min(GP, len - page * GP) : 0;
    if (!ok || valid <= 0) set_status(p.status, LOSA_ERR_BOUNDS);
    sm.phys[tid] = ok ? phys : 0;
    sm.valid[tid] = max(valid, 0);
  }
}

// One piece, more than kF32Few rows: union positions u0 .. u1 - 1 of segment sg.
template <int D, int GP, int NB, bool BITS>
__device__ __forceinline__ void f32_piece(const AttnParams& p, F32Smem<D>& sm, int sg, int u0, int u1) {
  constexpr int DI = D / 32, JM = 8;                // 16-byte reads of a key per lane, rows per lane
  constexpr int TS = kF32Warps / NB, TPW = kF32Tok / TS;   // warps per row block, tokens of a tile per warp
  constexpr int NSC = TPW;                          // scores per lane and tile
  constexpr int RG = 4 * NB, TG = 4 / NB, TPT = kF32Tok / TG;   // second product: row groups of 8, token groups, tokens per thread
  constexpr int CV = D / 64;                        // 16-byte column runs per thread
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rg = sg / p.n_sk, sk = sg % p.n_sk, s = sk / p.Hkv, kh = sk % p.Hkv;
  const int rows = rows_in_group(clamp_active(p.n_active[s], p.B), p.G, rg);
  const int len = p.kv_len[s];
  const float* kp = static_cast<const float*>(p.k_pages) + static_cast<size_t>(kh) * p.stride_head;
  const float* vp = static_cast<const float*>(p.v_pages) + static_cast<size_t>(kh) * p.stride_head;

  const int rb = warp / TS, ts = warp % TS, rs = lane >> 3, dg = lane & 7;
  const int my_row = rb * 32 + rs + 4 * dg;   // the row whose scores this lane ends up with
  const int my_pos = (my_row % RG) * 8 + my_row / RG;                            // its position in P, corr
  const int cg = tid & 15, rgp = (tid >> 4) % RG, tg = (tid >> 4) / RG;          // second product

  float2 q[JM][2 * DI];
#pragma unroll
  for (int j = 0; j < JM; ++j) {
    const int r = rb * 32 + rs + 4 * j;
    const float* src = nullptr;
    if (r < rows) {
      const int row = rg * kRowsPerGroup + r, a = row / p.G, gi = row % p.G;
      int tok = p.active_idx[s * p.B + a];
      if (tok < 0 || tok >= p.B) { set_status(p.status, LOSA_ERR_BOUNDS); tok = 0; }
      src = static_cast<const float*>(p.q) + ((static_cast<size_t>(s) * p.B + tok) * p.Hq + kh * p.G + gi) * D + dg * 4;
    }
#pragma unroll
    for (int i = 0; i < DI; ++i) {
      const float4 t = src ? *reinterpret_cast<const float4*>(src + i * 32) : make_float4(0.f, 0.f, 0.f, 0.f);
      q[j][2 * i] = make_float2(t.x, t.y);
      q[j][2 * i + 1] = make_float2(t.z, t.w);
    }
  }
  float2 acc[JM][2 * CV];
#pragma unroll
  for (int j = 0; j < JM; ++j)
#pragma unroll
    for (int c = 0; c < 2 * CV; ++c) acc[j][c] = make_float2(0.f, 0.f);
  float m = -INFINITY, l = 0.f;                     // of my_row; l: this warp's tokens only

  for (int c0 = u0; c0 < u1; c0 += kF32Chunk) {
    const int n = min(kF32Chunk, u1 - c0), n_tiles = (n * GP + kF32Tok - 1) / kF32Tok;
    __syncthreads();                                // the tiles and page numbers of the previous chunk (or piece) are done with
    f32_resolve<D, GP, BITS>(p, sm, sk, c0, n, len);
    __syncthreads();
    auto valid_token = [&](int t) {                 // token t of the chunk
      const int it = t / GP;
      return it < n && t % GP < sm.valid[it];
    };
    auto load = [&](int tile) {
      if (tile < n_tiles) {
        constexpr int LPR = D / 4, RPI = kF32Threads / LPR;     // lanes per row, rows per pass
        const int c = (tid % LPR) * 4;
#pragma unroll
        for (int i = 0; i < kF32Tok / RPI; ++i) {
          const int t = tid / LPR + i * RPI, tt = tile * kF32Tok + t, it = min(tt / GP, n - 1);
          const bool ok = valid_token(tt);
          const size_t off = static_cast<size_t>(sm.phys[it]) * p.stride_page + static_cast<size_t>(ok ? tt % GP : 0) * p.stride_tok + c;
          cp_async16_or_zero(smem_u32(&sm.t.k[tile % kF32Stages][t * D + c]), kp + off, ok);
          cp_async16_or_zero(smem_u32(&sm.t.v[tile % kF32Stages][t * D + c]), vp + off, ok);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    load(0);
    load(1);
    cp_async_wait<1>();
    __syncthreads();
    for (int tile = 0; tile < n_tiles; ++tile) {
      const float* ks = sm.t.k[tile % kF32Stages];
      const float* vs = sm.t.v[tile % kF32Stages];
      // ---- scores of this warp's tokens
      float sc[NSC];
      float mx = -INFINITY;
#pragma unroll
      for (int x = 0; x < TPW; x += 2) {
        const int t0 = ts * TPW + x;
        float2 a0[JM], a1[JM];
#pragma unroll
        for (int j = 0; j < JM; ++j) a0[j] = a1[j] = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < DI; ++i) {
          const float4 k0 = *reinterpret_cast<const float4*>(ks + t0 * D + i * 32 + dg * 4);
          const float4 k1 = *reinterpret_cast<const float4*>(ks + (t0 + 1) * D + i * 32 + dg * 4);
#pragma unroll
          for (int j = 0; j < JM; ++j) {
            a0[j] = fma2(q[j][2 * i], make_float2(k0.x, k0.y), a0[j]);
            a1[j] = fma2(q[j][2 * i], make_float2(k1.x, k1.y), a1[j]);
            a0[j] = fma2(q[j][2 * i + 1], make_float2(k0.z, k0.w), a0[j]);
            a1[j] = fma2(q[j][2 * i + 1], make_float2(k1.z, k1.w), a1[j]);
          }
        }
        const bool ok0 = valid_token(tile * kF32Tok + t0), ok1 = valid_token(tile * kF32Tok + t0 + 1);
        const bool b2 = dg & 4, b1 = dg & 2, b0 = dg & 1;
        // rows over the three bits of dg, token by token
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          const float2* a = y ? a1 : a0;
          float r4[4], r2[2];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float lo = a[j].x + a[j].y, hi = a[j + 4].x + a[j + 4].y;
            r4[j] = (b2 ? hi : lo) + __shfl_xor_sync(0xffffffffu, b2 ? lo : hi, 4);
          }
#pragma unroll
          for (int j = 0; j < 2; ++j) r2[j] = (b1 ? r4[j + 2] : r4[j]) + __shfl_xor_sync(0xffffffffu, b1 ? r4[j] : r4[j + 2], 2);
          const float r = (b0 ? r2[1] : r2[0]) + __shfl_xor_sync(0xffffffffu, b0 ? r2[0] : r2[1], 1);
          sc[x + y] = (y ? ok1 : ok0) ? r * p.sm_scale : -INFINITY;
          mx = fmaxf(mx, sc[x + y]);
        }
      }
      sm.t.red[warp * 32 + lane] = mx;
      __syncthreads();                              // A: maxima written; every thread has finished the previous tile
      load(tile + 2);
#pragma unroll
      for (int i = 0; i < TS; ++i) mx = fmaxf(mx, sm.t.red[(rb * TS + i) * 32 + lane]);
      const float m_new = fmaxf(m, mx);
      const float corr = (m_new == -INFINITY) ? 1.f : expf(m - m_new);
      m = m_new;
      l *= corr;
      if (ts == 0) sm.t.corr[my_pos] = corr;
#pragma unroll
      for (int x = 0; x < NSC; ++x) {
        const float pr = (sc[x] == -INFINITY) ? 0.f : expf(sc[x] - m_new);
        l += pr;
        const int t = ts * TPW + x;
        sm.t.p[t * kRowsPerGroup + my_pos] = pr;
      }
      cp_async_wait<1>();                           // this thread's copies of the next tile
      __syncthreads();                              // B: P, corr and the next tile's copies are visible
      // ---- O += P V
#pragma unroll
      for (int j = 0; j < JM; ++j) {
        const float cj = sm.t.corr[rgp * 8 + j];
#pragma unroll
        for (int c = 0; c < 2 * CV; ++c) { acc[j][c].x *= cj; acc[j][c].y *= cj; }
      }
#pragma unroll 2
      for (int x = 0; x < TPT; ++x) {
        const int t = tg * TPT + x;
        float pj[JM];
#pragma unroll
        for (int j = 0; j < JM; j += 4) {
          const float4 a = *reinterpret_cast<const float4*>(&sm.t.p[t * kRowsPerGroup + rgp * 8 + j]);
          pj[j] = a.x; pj[j + 1] = a.y; pj[j + 2] = a.z; pj[j + 3] = a.w;
        }
#pragma unroll
        for (int c = 0; c < CV; ++c) {
          const float4 v = *reinterpret_cast<const float4*>(vs + t * D + c * 64 + cg * 4);
#pragma unroll
          for (int j = 0; j < JM; ++j) {
            acc[j][2 * c] = fma2(make_float2(pj[j], pj[j]), make_float2(v.x, v.y), acc[j][2 * c]);
            acc[j][2 * c + 1] = fma2(make_float2(pj[j], pj[j]), make_float2(v.z, v.w), acc[j][2 * c + 1]);
          }
        }
      }
    }
    cp_async_wait<0>();
  }
  // ---- the piece's record: partial outputs of the token groups and partial row sums meet in shared memory
  __syncthreads();
  sm.t.red[warp * 32 + lane] = l;
  float* part = sm.t.k[0];                            // [TG][32 NB rows][D]
#pragma unroll
  for (int j = 0; j < JM; ++j)
#pragma unroll
    for (int c = 0; c < CV; ++c)
      *reinterpret_cast<float4*>(part + (tg * 32 * NB + rgp + RG * j) * D + c * 64 + cg * 4) =
          make_float4(acc[j][2 * c].x, acc[j][2 * c].y, acc[j][2 * c + 1].x, acc[j][2 * c + 1].y);
  __syncthreads();
  if (ts == 0 && my_row < rows) {
#pragma unroll
    for (int i = 1; i < TS; ++i) l += sm.t.red[(rb * TS + i) * 32 + lane];
    float* rec = record_base(p.partials, blockIdx.x + sg, my_row / kTileRows, D);
    rec[my_row % kTileRows] = m;
    rec[kTileRows + my_row % kTileRows] = l;
  }
  for (int idx = tid * 4; idx < rows * D; idx += kF32Threads * 4) {
    const int r = idx / D;
    float4 o = *reinterpret_cast<const float4*>(part + idx);
#pragma unroll
    for (int g = 1; g < TG; ++g) {
      const float4 t = *reinterpret_cast<const float4*>(part + g * 32 * NB * D + idx);
      o.x += t.x; o.y += t.y; o.z += t.z; o.w += t.w;
    }
    *reinterpret_cast<float4*>(record_base(p.partials, blockIdx.x + sg, r / kTileRows, D) + 2 * kTileRows + (r % kTileRows) * D + idx % D) = o;
  }
}

// One piece of at most kF32Few rows: every warp has tokens of its own.
template <int D, int GP, bool BITS>
__device__ __forceinline__ void f32_piece_few(const AttnParams& p, F32Smem<D>& sm, int sg, int u0, int u1) {
  constexpr int DI = D / 32, JM = 4, WT = kF32WTok;  // a lane's rows rs + 4 j
  constexpr int NSC = WT / 2;                        // scores per lane and step: lane bit 2 picks the token of a pair
  constexpr int CL = D / 32, NR2 = kF32Few / 2;      // columns per lane, pairs of rows in the second product
  static_assert(GP % WT == 0, "a step's tokens lie in one page");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rg = sg / p.n_sk, sk = sg % p.n_sk, s = sk / p.Hkv, kh = sk % p.Hkv;
  const int rows = rows_in_group(clamp_active(p.n_active[s], p.B), p.G, rg);
  const int len = p.kv_len[s];
  const float* kp = static_cast<const float*>(p.k_pages) + static_cast<size_t>(kh) * p.stride_head;
  const float* vp = static_cast<const float*>(p.v_pages) + static_cast<size_t>(kh) * p.stride_head;
  const int rs = lane >> 3, dg = lane & 7, my_row = rs + 4 * (dg & 3);   // the row whose scores this lane ends up with

  float2 q[JM][2 * DI];
#pragma unroll
  for (int j = 0; j < JM; ++j) {
    const int r = rs + 4 * j;
    const float* src = nullptr;
    if (r < rows) {
      const int row = rg * kRowsPerGroup + r, a = row / p.G, gi = row % p.G;
      int tok = p.active_idx[s * p.B + a];
      if (tok < 0 || tok >= p.B) { set_status(p.status, LOSA_ERR_BOUNDS); tok = 0; }
      src = static_cast<const float*>(p.q) + ((static_cast<size_t>(s) * p.B + tok) * p.Hq + kh * p.G + gi) * D + dg * 4;
    }
#pragma unroll
    for (int i = 0; i < DI; ++i) {
      const float4 t = src ? *reinterpret_cast<const float4*>(src + i * 32) : make_float4(0.f, 0.f, 0.f, 0.f);
      q[j][2 * i] = make_float2(t.x, t.y);
      q[j][2 * i + 1] = make_float2(t.z, t.w);
    }
  }
  float2 acc[NR2][CL];                               // rows 2 a and 2 a + 1, columns lane * CL + c
#pragma unroll
  for (int a = 0; a < NR2; ++a)
#pragma unroll
    for (int c = 0; c < CL; ++c) acc[a][c] = make_float2(0.f, 0.f);
  float m = -INFINITY, l = 0.f;                      // of my_row over this warp's tokens; l: this lane's only
  float* wp = sm.w.p[warp];
  float* wc = sm.w.corr[warp];

  for (int c0 = u0; c0 < u1; c0 += kF32Chunk) {
    const int n = min(kF32Chunk, u1 - c0), n_steps = n * (GP / WT);
    __syncthreads();                                 // the page numbers and rings of the previous chunk (or piece) are done with
    f32_resolve<D, GP, BITS>(p, sm, sk, c0, n, len);
    __syncthreads();
    auto load = [&](int step, int slot) {
      if (step < n_steps) {
        constexpr int LPR = D / 4, RPI = 32 / LPR;              // lanes per row, rows per pass
        const int it = step / (GP / WT), t0 = step % (GP / WT) * WT, valid = sm.valid[it], c = (lane % LPR) * 4;
        const size_t off = static_cast<size_t>(sm.phys[it]) * p.stride_page + c;
#pragma unroll
        for (int i = 0; i < WT / RPI; ++i) {
          const int t = lane / LPR + i * RPI;
          const bool ok = t0 + t < valid;
          const size_t at = off + static_cast<size_t>(ok ? t0 + t : 0) * p.stride_tok;
          cp_async16_or_zero(smem_u32(&sm.w.kv[warp][slot][0][t * D + c]), kp + at, ok);
          cp_async16_or_zero(smem_u32(&sm.w.kv[warp][slot][1][t * D + c]), vp + at, ok);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    load(warp, 0);
    load(warp + kF32Warps, 1);
    int slot = 0;
    for (int step = warp; step < n_steps; step += kF32Warps) {
      cp_async_wait<1>();
      __syncwarp();                                  // the whole warp's copies, and it has finished the slot that is refilled now
      load(step + 2 * kF32Warps, slot == 0 ? 2 : slot - 1);
      const float* ks = sm.w.kv[warp][slot][0];
      const float* vs = sm.w.kv[warp][slot][1];
      slot = slot == 2 ? 0 : slot + 1;
      const int valid = sm.valid[step / (GP / WT)] - step % (GP / WT) * WT;
      // ---- scores
      float sc[NSC];
      float mx = -INFINITY;
#pragma unroll
      for (int x = 0; x < NSC; ++x) {
        float2 a0[JM], a1[JM];
#pragma unroll
        for (int j = 0; j < JM; ++j) a0[j] = a1[j] = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < DI; ++i) {
          const float4 k0 = *reinterpret_cast<const float4*>(ks + 2 * x * D + i * 32 + dg * 4);
          const float4 k1 = *reinterpret_cast<const float4*>(ks + (2 * x + 1) * D + i * 32 + dg * 4);
#pragma unroll
          for (int j = 0; j < JM; ++j) {
            a0[j] = fma2(q[j][2 * i], make_float2(k0.x, k0.y), a0[j]);
            a1[j] = fma2(q[j][2 * i], make_float2(k1.x, k1.y), a1[j]);
            a0[j] = fma2(q[j][2 * i + 1], make_float2(k0.z, k0.w), a0[j]);
            a1[j] = fma2(q[j][2 * i + 1], make_float2(k1.z, k1.w), a1[j]);
          }
        }
        // the token over bit 2 of dg, rows over the other two
        const bool b2 = dg & 4, b1 = dg & 2, b0 = dg & 1;
        float r4[4], r2[2];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float lo = a0[j].x + a0[j].y, hi = a1[j].x + a1[j].y;
          r4[j] = (b2 ? hi : lo) + __shfl_xor_sync(0xffffffffu, b2 ? lo : hi, 4);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) r2[j] = (b1 ? r4[j + 2] : r4[j]) + __shfl_xor_sync(0xffffffffu, b1 ? r4[j] : r4[j + 2], 2);
        const float r = (b0 ? r2[1] : r2[0]) + __shfl_xor_sync(0xffffffffu, b0 ? r2[0] : r2[1], 1);
        sc[x] = 2 * x + (dg >> 2) < valid ? r * p.sm_scale : -INFINITY;
        mx = fmaxf(mx, sc[x]);
      }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
      const float m_new = fmaxf(m, mx), corr = (m_new == -INFINITY) ? 1.f : expf(m - m_new);
      const bool moved = __any_sync(0xffffffffu, corr != 1.f);
      m = m_new;
      l *= corr;
      if (dg < 4) wc[my_row] = corr;
#pragma unroll
      for (int x = 0; x < NSC; ++x) {
        const float pr = (sc[x] == -INFINITY) ? 0.f : expf(sc[x] - m_new);
        l += pr;
        wp[(2 * x + (dg >> 2)) * kF32Few + my_row] = pr;
      }
      __syncwarp();
      // ---- O += P V
      if (moved) {
#pragma unroll
        for (int a = 0; a < NR2; ++a) {
          const float2 cr = *reinterpret_cast<const float2*>(wc + 2 * a);
#pragma unroll
          for (int c = 0; c < CL; ++c) { acc[a][c].x *= cr.x; acc[a][c].y *= cr.y; }
        }
      }
#pragma unroll 2
      for (int t = 0; t < WT; ++t) {
        float v[CL];
        ldv<CL>(vs + t * D + lane * CL, v);
#pragma unroll
        for (int a = 0; a < NR2; a += 2) {
          const float4 pr = *reinterpret_cast<const float4*>(wp + t * kF32Few + 2 * a);
#pragma unroll
          for (int c = 0; c < CL; ++c) {
            const float2 vv = make_float2(v[c], v[c]);
            acc[a][c] = fma2(make_float2(pr.x, pr.y), vv, acc[a][c]);
            acc[a + 1][c] = fma2(make_float2(pr.z, pr.w), vv, acc[a + 1][c]);
          }
        }
      }
    }
    cp_async_wait<0>();
  }
  // ---- the piece's record: the warps' partial results meet in shared memory
  l += __shfl_xor_sync(0xffffffffu, l, 4);
  __syncthreads();                                   // every warp has done with its ring
  if (dg < 4) { sm.w.m[warp][my_row] = m; sm.w.l[warp][my_row] = l; }
  float* part = &sm.w.kv[0][0][0][0];                // [warp][row][D]
  static_assert(sizeof(sm.w.kv) >= sizeof(float) * kF32Warps * kF32Few * D, "the partial outputs fit the rings");
#pragma unroll
  for (int a = 0; a < NR2; ++a) {
    float x[CL], y[CL];
#pragma unroll
    for (int c = 0; c < CL; ++c) { x[c] = acc[a][c].x; y[c] = acc[a][c].y; }
    stv<CL>(part + (warp * kF32Few + 2 * a) * D + lane * CL, x);
    stv<CL>(part + (warp * kF32Few + 2 * a + 1) * D + lane * CL, y);
  }
  __syncthreads();
  for (int idx = tid * 4; idx < rows * D; idx += kF32Threads * 4) {
    const int r = idx / D;
    float M = -INFINITY, L = 0.f;
#pragma unroll
    for (int w = 0; w < kF32Warps; ++w) M = fmaxf(M, sm.w.m[w][r]);
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kF32Warps; ++w) {
      const float mw = sm.w.m[w][r], f = mw == -INFINITY ? 0.f : expf(mw - M);
      const float4 t = *reinterpret_cast<const float4*>(part + w * kF32Few * D + idx);
      L = fmaf(sm.w.l[w][r], f, L);
      if (f != 0.f) { o.x = fmaf(t.x, f, o.x); o.y = fmaf(t.y, f, o.y); o.z = fmaf(t.z, f, o.z); o.w = fmaf(t.w, f, o.w); }
    }
    float* rec = record_base(p.partials, blockIdx.x + sg, r / kTileRows, D);
    *reinterpret_cast<float4*>(rec + 2 * kTileRows + (r % kTileRows) * D + idx % D) = o;
    if (idx % D == 0) {
      rec[r % kTileRows] = M;
      rec[kTileRows + r % kTileRows] = L;
    }
  }
}

template <int D, int GP, bool BITS>
__global__ void __launch_bounds__(kF32Threads, 1) attn_f32_kernel(AttnParams p) {
  grid_dep_wait();
  extern __shared__ __align__(16) uint8_t f32_smem[];
  F32Smem<D>& sm = *reinterpret_cast<F32Smem<D>*>(f32_smem);
  static_assert(sizeof(float) * 2 * kF32Stages * kF32Tok * D >= sizeof(float) * kRowsPerGroup * D, "the partial outputs fit the tiles");
  const UnionBits lists = sm.lists(p.W);
  if constexpr (BITS) {
    lists.load(p.union_bits, p.n_sk, threadIdx.x >> 5, kF32Warps, threadIdx.x & 31);
    __syncthreads();
  }
  if (threadIdx.x < 32) segment_prefix(sm.pre, p.n_seg, p.n_rg, p.Hkv, p.G, p.n_active, [&](int sk) { return BITS ? lists.count(sk) : p.union_count[sk]; }, p.B, threadIdx.x);
  else if (BITS && threadIdx.x < 64) lists.write(p, threadIdx.x & 31);
  __syncthreads();
  const int T_all = sm.pre[p.n_seg];
  const int n = f32_ctas(T_all, p.n_ctas, GP);
  for (int seg = blockIdx.x * kF32Threads + threadIdx.x; seg < p.n_seg; seg += gridDim.x * kF32Threads)
    p.seg_records[seg] = segment_records(T_all, n, sm.pre[seg], sm.pre[seg + 1]);
  if (static_cast<int>(blockIdx.x) >= n) return;
  const int lo = cta_lo(T_all, blockIdx.x, n), hi = cta_lo(T_all, blockIdx.x + 1, n);
  int sg = 0, item = lo;
  while (item < hi) {
    while (sm.pre[sg + 1] <= item) ++sg;
    const int seg_end = min(hi, sm.pre[sg + 1]), u0 = item - sm.pre[sg], u1 = seg_end - sm.pre[sg];
    const int rows = rows_in_group(clamp_active(p.n_active[(sg % p.n_sk) / p.Hkv], p.B), p.G, sg / p.n_sk);
    if (rows <= kF32Few) f32_piece_few<D, GP, BITS>(p, sm, sg, u0, u1);
    else if (rows <= 32) f32_piece<D, GP, 1, BITS>(p, sm, sg, u0, u1);
    else if (rows <= 64) f32_piece<D, GP, 2, BITS>(p, sm, sg, u0, u1);
    else f32_piece<D, GP, 4, BITS>(p, sm, sg, u0, u1);
    item = seg_end;
  }
}
