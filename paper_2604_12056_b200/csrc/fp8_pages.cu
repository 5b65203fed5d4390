// FP8 (E4M3) K/V pages with one power-of-two scale per (physical page, KV head) and tensor: an
// extension of the cache format (the paper names quantised attention as orthogonal to the method,
// Section 6, and quotes the cached state in FP16, Section 4.5).  Halves the bytes stage 4 streams.
//
//   amax  = largest |x| over the page's valid tokens and d dimensions
//   scale = 2^e, e = the smallest integer with amax <= 448 * 2^e, clamped to [-6, 7]
//   code  = round-to-nearest-even of x / scale onto the E4M3 grid, saturated at +-448
//   dequantised value = scale * value(code): four significant bits, exact in bf16 and in fp16
// Slots of a page past the prefix's end get code 0.  Appending a block re-quantises every touched
// page from its dequantised old values and the new rows together (the scale may have to grow).
// The page summaries (Section 2.3) are the element-wise min / max of the DEQUANTISED keys, so that
// stage 2 bounds the keys stage 4 actually uses.
//
// One warp per (logical page, KV head, tensor, sequence).  The path is a copy with a reduction in it,
// so HBM bounds it: a lane takes eight consecutive elements of a row per load (16 bytes of bf16, 8 of
// codes), the whole slice is requested at once and stays in registers (8 KiB per warp at 32 x 128),
// the maximum is a warp reduction, and the codes leave as 8-byte stores.  Warps of a CTA take
// neighbouring heads of a page, which lie next to one another in the pool.  Encoding is monotone, so
// the summaries are the encoded column extremes of the source; -0 orders below +0 in both.
// Quantising 90,000 tokens of 8 heads x 128 (565 MB in and out): 261 us with a thread per column
// that walked the tokens three times, 116 us now.
#include <cuda_fp8.h>

#include "kernels.h"

namespace losa {
namespace {

// eight codes -> values, eight values -> codes (round to nearest even, saturate at +-448)
__device__ __forceinline__ void fp8_decode8(uint2 w, float (&v)[8]) {
  const uint32_t x[2] = {w.x, w.y};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __half2_raw h = __nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(x[i >> 1] >> (16 * (i & 1))), __NV_E4M3);
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h));
    v[2 * i] = f.x;
    v[2 * i + 1] = f.y;
  }
}
__device__ __forceinline__ uint2 fp8_encode8(const float (&v)[8], float inv_scale) {
  uint32_t x[4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    x[i] = __nv_cvt_float2_to_fp8x2(make_float2(v[2 * i] * inv_scale, v[2 * i + 1] * inv_scale), __NV_SATFINITE, __NV_E4M3);
  return make_uint2(x[0] | (x[1] << 16), x[2] | (x[3] << 16));
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }   // -126 <= e <= 127
// e = the smallest integer in [-6, 7] with amax <= 448 * 2^e = 1.75 * 2^(e + 8)
__device__ __forceinline__ int fp8_scale_exp(float amax) {
  const uint32_t b = __float_as_uint(amax);
  const int e = static_cast<int>(b >> 23) - 127 - 8 + ((b & 0x7fffffu) > 0x600000u ? 1 : 0);
  return min(7, max(-6, e));
}

struct Fp8Params {
  const __nv_bfloat16* k_src;        // bf16 pool (quantise) — strides below; null otherwise
  const __nv_bfloat16* v_src;
  int64_t src_stride_page, src_stride_head, src_stride_tok;
  uint8_t* k_codes;                  // fp8 pool
  uint8_t* v_codes;
  int64_t stride_page, stride_head, stride_tok;
  float* k_scale;
  float* v_scale;
  __nv_bfloat16* kmin;
  __nv_bfloat16* kmax;
  const int32_t* page_table;
  const int32_t* kv_len;
  const __nv_bfloat16* k_blk;        // [N, B, H_kv, d] (append)
  const __nv_bfloat16* v_blk;
  int blk_aligned;                   // the block rows may be read 16 bytes at a time
  int32_t* status;
  int B, Hkv, Pmax, n_phys;
};

// MODE 0: quantise a bf16 pool page by page (+ summaries); MODE 1: summaries of an FP8 pool;
// MODE 2: append the block to the touched pages (re-quantising them, + summaries).
constexpr int kFp8Warps = 8;

template <int MODE, int D, int GP>
__global__ void __launch_bounds__(kFp8Warps * 32) fp8_pages_kernel(Fp8Params p) {
  constexpr int LPR = D / 8, RPI = 32 / LPR, NI = GP / RPI;      // lanes per row, rows per load, loads per slice
  static_assert(GP % RPI == 0, "whole rows per load");
  grid_dep_wait();
  const int lane = threadIdx.x & 31, w = blockIdx.x * kFp8Warps + (threadIdx.x >> 5);
  const int kh = w % p.Hkv, s = blockIdx.z;
  const bool is_v = blockIdx.y != 0;
  const int L0 = p.kv_len[s];
  int page = w / p.Hkv, n_old, n_all;
  if (MODE == 2) {
    page += L0 / GP;
    if (page > (L0 + p.B - 1) / GP) return;
    if (page >= p.Pmax) { if (lane == 0) set_status(p.status, LOSA_ERR_BOUNDS); return; }
    n_old = max(0, L0 - page * GP);
    n_all = min(L0 + p.B, (page + 1) * GP) - page * GP;
  } else {
    n_old = n_all = min(GP, L0 - page * GP);
  }
  // (modes 0 and 1: requested beside the length; a table entry past the prefix is not used)
  if (MODE != 2 && page >= p.Pmax) return;
  const int phys = p.page_table[static_cast<size_t>(s) * p.Pmax + page];
  if (n_all <= 0) return;
  if (phys < 0 || phys >= p.n_phys) { if (lane == 0) set_status(p.status, LOSA_ERR_BOUNDS); return; }
  const int t0 = lane / LPR, j = (lane % LPR) * 8;
  uint8_t* codes = (is_v ? p.v_codes : p.k_codes) + static_cast<size_t>(phys) * p.stride_page + static_cast<size_t>(kh) * p.stride_head + j;
  float* scale = (is_v ? p.v_scale : p.k_scale) + static_cast<size_t>(phys) * p.Hkv + kh;
  const float old_scale = MODE == 0 ? 1.f : *scale;

  // the lane's rows, as bf16: source rows, old rows dequantised (exact: four significant bits), new rows
  uint4 raw[NI];
  uint2 old[MODE == 0 ? 1 : NI];
  if constexpr (MODE != 0) {
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int t = t0 + i * RPI;
      old[i] = t < n_old ? *reinterpret_cast<const uint2*>(codes + static_cast<size_t>(t) * p.stride_tok) : make_uint2(0u, 0u);
    }
  }
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    const int t = t0 + i * RPI;
    raw[i] = make_uint4(0u, 0u, 0u, 0u);
    if (MODE == 0) {
      if (t < n_all)
        raw[i] = __ldcs(reinterpret_cast<const uint4*>((is_v ? p.v_src : p.k_src) + static_cast<size_t>(phys) * p.src_stride_page +
                                                       static_cast<size_t>(kh) * p.src_stride_head + static_cast<size_t>(t) * p.src_stride_tok + j));
    } else if (MODE == 2 && t >= n_old && t < n_all) {
      const int row = page * GP + t - L0;                          // block token
      const __nv_bfloat16* src = (is_v ? p.v_blk : p.k_blk) + ((static_cast<size_t>(s) * p.B + row) * p.Hkv + kh) * D + j;
      if (p.blk_aligned) {
        raw[i] = *reinterpret_cast<const uint4*>(src);
      } else {
        alignas(16) __nv_bfloat16 e[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) e[x] = src[x];
        raw[i] = *reinterpret_cast<const uint4*>(e);
      }
    }
  }
  if constexpr (MODE != 0) {
#pragma unroll
    for (int i = 0; i < NI; ++i)
      if (t0 + i * RPI < n_old) {
        float v[8];
        fp8_decode8(old[i], v);
        alignas(16) __nv_bfloat162 h[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) h[x] = __floats2bfloat162_rn(v[2 * x] * old_scale, v[2 * x + 1] * old_scale);
        raw[i] = *reinterpret_cast<const uint4*>(h);
      }
  }
  // extremes of the lane's columns over its rows, then of the slice
  float lo[8], hi[8];
#pragma unroll
  for (int x = 0; x < 8; ++x) { lo[x] = INFINITY; hi[x] = -INFINITY; }
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    if (t0 + i * RPI < n_all) {
      float v[8];
      load8(reinterpret_cast<const __nv_bfloat16*>(&raw[i]), v);
#pragma unroll
      for (int x = 0; x < 8; ++x) { lo[x] = fminf(lo[x], v[x]); hi[x] = fmaxf(hi[x], v[x]); }
    }
  }
  float new_scale = old_scale, inv = 1.f;
  if (MODE != 1) {
    float amax = 0.f;
#pragma unroll
    for (int x = 0; x < 8; ++x)
      if (lo[x] <= hi[x]) amax = fmaxf(amax, fmaxf(fabsf(lo[x]), fabsf(hi[x])));   // (else: no rows in this lane)
    const int e = fp8_scale_exp(warp_max(amax));
    new_scale = pow2f(e);
    inv = pow2f(-e);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int t = t0 + i * RPI;
      float v[8];
      load8(reinterpret_cast<const __nv_bfloat16*>(&raw[i]), v);
      *reinterpret_cast<uint2*>(codes + static_cast<size_t>(t) * p.stride_tok) = t < n_all ? fp8_encode8(v, inv) : make_uint2(0u, 0u);
    }
    if (lane == 0) *scale = new_scale;
  }
  if (is_v) return;
#pragma unroll
  for (int o = LPR; o < 32; o <<= 1)
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      lo[x] = fminf(lo[x], __shfl_xor_sync(0xffffffffu, lo[x], o));
      hi[x] = fmaxf(hi[x], __shfl_xor_sync(0xffffffffu, hi[x], o));
    }
  if (t0 == 0) {
    if (MODE != 1) {                                                // through the codes (mode 1: the rows came from them)
      float a[8], b[8];
      fp8_decode8(fp8_encode8(lo, inv), a);
      fp8_decode8(fp8_encode8(hi, inv), b);
#pragma unroll
      for (int x = 0; x < 8; ++x)
        if (lo[x] <= hi[x]) { lo[x] = a[x] * new_scale; hi[x] = b[x] * new_scale; }
    }
    alignas(16) __nv_bfloat162 a[4], b[4];                                      // exact: four significant bits
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      a[x] = __floats2bfloat162_rn(lo[2 * x], lo[2 * x + 1]);
      b[x] = __floats2bfloat162_rn(hi[2 * x], hi[2 * x + 1]);
    }
    const size_t at = (static_cast<size_t>(phys) * p.Hkv + kh) * D + j;
    *reinterpret_cast<uint4*>(p.kmin + at) = *reinterpret_cast<const uint4*>(a);
    *reinterpret_cast<uint4*>(p.kmax + at) = *reinterpret_cast<const uint4*>(b);
  }
}

template <int MODE, int D>
void launch_fp8_d(const losa_shape_t& sh, const Fp8Params& p, int pages, cudaStream_t st) {
  const dim3 grid((pages * sh.n_kv_heads + kFp8Warps - 1) / kFp8Warps, MODE == 1 ? 1 : 2, sh.batch);
  auto launch = [&](void (*kernel)(Fp8Params)) {      // (mode 2 is a small kernel between the steps of two blocks)
    if (MODE == 2) launch_k(kernel, grid, kFp8Warps * 32, 0, st, p);
    else launch_streaming(kernel, grid, kFp8Warps * 32, 0, st, p);
  };
  switch (sh.page_size) {
    case 16: launch(fp8_pages_kernel<MODE, D, 16>); break;
    case 32: launch(fp8_pages_kernel<MODE, D, 32>); break;
    default: launch(fp8_pages_kernel<MODE, D, 64>); break;
  }
}
// `pages`: logical pages per sequence that the grid covers
template <int MODE>
int32_t launch_fp8(losa_ctx* c, const Fp8Params& p, int pages, cudaStream_t st) {
  if (c->shape.head_dim == 128) launch_fp8_d<MODE, 128>(c->shape, p, pages, st);
  else launch_fp8_d<MODE, 64>(c->shape, p, pages, st);
  return after_launch(c);
}

Fp8Params base_params(losa_ctx* c, const losa_kv_t* kv) {
  const losa_shape_t& sh = c->shape;
  Fp8Params p = {};
  p.k_codes = static_cast<uint8_t*>(kv->k_pages);
  p.v_codes = static_cast<uint8_t*>(kv->v_pages);
  p.stride_page = kv->stride_page;
  p.stride_head = kv->stride_head;
  p.stride_tok = kv->stride_tok;
  p.k_scale = kv->k_scale;
  p.v_scale = kv->v_scale;
  p.kmin = static_cast<__nv_bfloat16*>(kv->kmin);
  p.kmax = static_cast<__nv_bfloat16*>(kv->kmax);
  p.page_table = kv->page_table;
  p.kv_len = kv->kv_len;
  p.status = status_ptr(c);
  p.B = sh.block_size;
  p.Hkv = sh.n_kv_heads;
  p.Pmax = sh.max_pages_per_seq;
  p.n_phys = kv->n_phys_pages;
  return p;
}

}  // namespace

int32_t launch_fp8_quantize(losa_ctx* c, const losa_kv_t* src, losa_kv_t* dst, cudaStream_t st) {
  const losa_shape_t& sh = c->shape;
  if (sh.max_pages_per_seq == 0) return LOSA_OK;
  Fp8Params p = base_params(c, dst);
  p.k_src = static_cast<const __nv_bfloat16*>(src->k_pages);
  p.v_src = static_cast<const __nv_bfloat16*>(src->v_pages);
  p.src_stride_page = src->stride_page;
  p.src_stride_head = src->stride_head;
  p.src_stride_tok = src->stride_tok;
  return launch_fp8<0>(c, p, sh.max_pages_per_seq, st);
}

int32_t launch_fp8_summaries(losa_ctx* c, losa_kv_t* kv, cudaStream_t st) {
  const losa_shape_t& sh = c->shape;
  if (sh.max_pages_per_seq == 0) return LOSA_OK;
  return launch_fp8<1>(c, base_params(c, kv), sh.max_pages_per_seq, st);
}

// the kv_len / step counters are bumped by the caller's usual counter kernel afterwards
int32_t launch_fp8_append(losa_ctx* c, losa_kv_t* kv, const void* k_blk, const void* v_blk, cudaStream_t st) {
  const losa_shape_t& sh = c->shape;
  Fp8Params p = base_params(c, kv);
  p.k_blk = static_cast<const __nv_bfloat16*>(k_blk);
  p.v_blk = static_cast<const __nv_bfloat16*>(v_blk);
  p.blk_aligned = ((reinterpret_cast<uintptr_t>(k_blk) | reinterpret_cast<uintptr_t>(v_blk)) & 15u) == 0;
  return launch_fp8<2>(c, p, (sh.block_size + sh.page_size - 1) / sh.page_size + 1, st);
}

}  // namespace losa
