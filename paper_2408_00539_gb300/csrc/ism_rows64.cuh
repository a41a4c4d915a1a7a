// Rows of the head_dim 64 tensor-core kernels whose result is not finite, over
// again on the CUDA cores.
//
// The tensor cores contract whole 128-row tiles, with weight zero where the mask
// hides a key or query.  A NaN or Inf in a hidden row, be it of the next dialogue
// in the buffer, would reach every row of the tile all the same (0 * NaN), and an
// Inf that a row does see would come out as NaN (the low part of a split weight
// may be zero or negative).  Every such case leaves a NaN or Inf in the
// accumulators, so the epilogues look at those and send the rows here: fp32
// sums over the visible keys or queries alone, as the CUDA-core kernels do them.
// Finite inputs never come here; the look costs an FMA an element.  With NaN
// throughout, 6001 tokens of 16 heads take 8 ms forward and 28 back (the CUDA-core
// kernels 44 and 159); the block's other warps wait meanwhile, within the two
// seconds of a bounded wait up to dialogues of some 500 thousand rows (one of 32768
// with eight heads on a KV head takes 0.3 and 1.3 s in all).
//
// Each function is called by a whole warp for one row; lane d returns the
// unnormalised sums of columns d and d + 32.
#pragma once

#include "ism_tc_common.cuh"

namespace ism {
namespace tc {
namespace rows64 {

constexpr int kHD = 64;

// Zero while every x so far is finite, NaN from then on.
__device__ __forceinline__ float not_finite(uint32_t x, float so_far) { return fmaf(__uint_as_float(x), 0.f, so_far); }

__device__ __forceinline__ float dot(const __nv_bfloat16* x, const __nv_bfloat16* y) {
  float s = 0.f;
#pragma unroll
  for (int c = 0; c < kHD / 8; ++c) {
    const uint4 u = reinterpret_cast<const uint4*>(x)[c], v = reinterpret_cast<const uint4*>(y)[c];
    const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&u);
    const __nv_bfloat162* q = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 f = __bfloat1622float2(p[e]), g = __bfloat1622float2(q[e]);
      s = fmaf(f.x, g.x, fmaf(f.y, g.y, s));
    }
  }
  return s;
}
// acc += weight of lane t times the row that lane t names, for the first n lanes.
__device__ __forceinline__ void add_rows(float w, const __nv_bfloat16* row, int n, float2& acc) {
  const int lane = threadIdx.x & 31;
  for (int t = 0; t < n; ++t) {
    const float f = __shfl_sync(0xffffffffu, w, t);
    const __nv_bfloat16* r =
        reinterpret_cast<const __nv_bfloat16*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(row), t));
    acc.x = fmaf(f, __bfloat162float(r[lane]), acc.x);
    acc.y = fmaf(f, __bfloat162float(r[lane + 32]), acc.y);
  }
}

// (Not inlined: the hot loops keep their registers.)
#define ISM_ROW_FN [[maybe_unused]] static __device__ __noinline__ float2

// Sum over keys [k0, k1) of 2^(scaled score - m) V.
ISM_ROW_FN out_row(const AttnArgs& a, int32_t q_row, int32_t k_base, int h, int k0, int k1, float m) {
  const int lane = threadIdx.x & 31, g = h / (a.hq / a.hkv);
  const float sl2 = a.scale * kLog2e;
  const __nv_bfloat16* q = static_cast<const __nv_bfloat16*>(a.q) + ((int64_t)q_row * a.hq + h) * kHD;
  float2 acc = make_float2(0.f, 0.f);
  for (int kb = k0; kb < k1; kb += 32) {
    const int key = min(kb + lane, k1 - 1);
    const int64_t row = a.pages.table ? paged_row(a.pages, k_base, key) : (int64_t)k_base + key;
    const int64_t off = (row * a.hkv + g) * kHD;
    const float p = ex2(dot(q, static_cast<const __nv_bfloat16*>(a.k) + off) * sl2 - m);
    add_rows(p, static_cast<const __nv_bfloat16*>(a.v) + off, min(32, k1 - kb), acc);
  }
  return acc;
}

// Sum over keys [0, ke) of dS K.
ISM_ROW_FN dq_row(const AttnArgs& a, int32_t q_row, int32_t k_base, int h, int ke, float lse2, float delta) {
  const int lane = threadIdx.x & 31, g = h / (a.hq / a.hkv);
  const float sl2 = a.scale * kLog2e;
  const int64_t qo = ((int64_t)q_row * a.hq + h) * kHD;
  const __nv_bfloat16 *q = static_cast<const __nv_bfloat16*>(a.q) + qo,
                      *dout = static_cast<const __nv_bfloat16*>(a.dout) + qo;
  float2 acc = make_float2(0.f, 0.f);
  for (int kb = 0; kb < ke; kb += 32) {
    const int key = min(kb + lane, ke - 1);
    const int64_t off = (((int64_t)k_base + key) * a.hkv + g) * kHD;
    const __nv_bfloat16* k = static_cast<const __nv_bfloat16*>(a.k) + off;
    const float ds = ex2(dot(q, k) * sl2 - lse2) * (dot(dout, static_cast<const __nv_bfloat16*>(a.v) + off) - delta);
    add_rows(ds, k, min(32, ke - kb), acc);
  }
  return acc;
}

// Sum over the query heads of KV head g and the query rows that see key `key`
// of the sequence, of P dO (dV), or with dk of dS Q (dK).
ISM_ROW_FN dkdv_row(const AttnArgs& a, int32_t q_base, int q_len, int32_t k_base, int32_t kv_base, int g, int key,
                    bool dk) {
  const int lane = threadIdx.x & 31, group = a.hq / a.hkv;
  const float sl2 = a.scale * kLog2e;
  const int64_t ko = (((int64_t)k_base + key) * a.hkv + g) * kHD;
  const __nv_bfloat16 *k = static_cast<const __nv_bfloat16*>(a.k) + ko, *v = static_cast<const __nv_bfloat16*>(a.v) + ko;
  const int32_t* kv_end = a.kv_end + kv_base;
  int lo = 0, hi = q_len;  // bounds do not decrease: rows from the first one past the key
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (kv_end[mid] > key) hi = mid; else lo = mid + 1;
  }
  float2 acc = make_float2(0.f, 0.f);
  for (int h = g * group; h < (g + 1) * group; ++h)
    for (int jb = lo; jb < q_len; jb += 32) {
      const int64_t row = (int64_t)q_base + min(jb + lane, q_len - 1);
      const int64_t off = (row * a.hq + h) * kHD, at = (int64_t)h * a.q_rows + row;
      const __nv_bfloat16 *q = static_cast<const __nv_bfloat16*>(a.q) + off,
                          *dout = static_cast<const __nv_bfloat16*>(a.dout) + off;
      float x = ex2(dot(k, q) * sl2 - a.lse_in[at] * kLog2e);
      if (dk) x *= dot(v, dout) - a.delta[at];
      add_rows(x, dk ? q : dout, min(32, q_len - jb), acc);
    }
  return acc;
}

__device__ __forceinline__ void store_row(__nv_bfloat16* row, float2 x) {
  const int lane = threadIdx.x & 31;
  row[lane] = __float2bfloat16_rn(x.x);
  row[lane + 32] = __float2bfloat16_rn(x.y);
}
// The same behind the transposed rotation of position pos (rope_back_pack).
__device__ __forceinline__ void store_row_back(__nv_bfloat16* row, float2 x, const AttnArgs& a, int pos) {
  const int64_t at = (int64_t)pos * (kHD / 2) + (threadIdx.x & 31);
  const float c = a.rope_cos[at], s = a.rope_sin[at];
  store_row(row, make_float2(x.x * c + x.y * s, x.y * c - x.x * s));
}

#undef ISM_ROW_FN

}  // namespace rows64
}  // namespace tc
}  // namespace ism
