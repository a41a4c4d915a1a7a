// CUDA-core attention under the ISM mask: the fp32 path (and bf16 under
// ISM_FORCE_CUDA_CORES=1).  fp32 arithmetic with natural-base exponentials
// throughout; forward (Eq. e_ISM with softmax, online over key blocks) and the
// standard softmax-attention gradients.
//
// All three kernels have one shape.  A block owns W * R rows (queries in the
// forward and dQ, keys in dK/dV), a group of S warps R of them; the other side
// streams through shared memory in blocks of S * SB rows, each warp of a group
// taking SB of them.  A lane computes the scores of its SB / 32 streamed rows
// against the R rows (the streamed rows padded to D + 4 floats, so that 32
// lanes reading one column group of 32 rows hit all banks; the own rows are
// broadcasts), the weights pass through warp-private shared memory, and the
// accumulation has the lanes over the head dimension.  The next block's global
// loads are in registers while this one is computed.
//
// What bounds it: shared-memory reads.  A step of four columns costs a warp
// 4 SB / 32 + R wavefronts for 4 R SB / 32 FMAs, so R = 8, S = 1 feeds the FMA
// pipes.  While blocks of 64 rows would leave SMs without one (a small
// problem, bound by the serial walk), 16 rows a block with S = 4 shorten the
// walk fourfold and put four warps on each scheduler.  A 256-token dialogue
// with 2 heads of 64 (the tiny fp32 step): forward 952 -> 14.6 us, dQ with
// Delta 1675 -> 18.0 us, dK/dV 2324 -> 19.3 us against one warp a row over
// unstaged keys (with S = 1: 19.5, 17.6 and 21.9 us; a whole step of 1000
// tokens and 4 heads 225 us with S = 1, 174 with S = 4).
#include "ism_internal.cuh"

namespace ism {
namespace {

constexpr int kTileRows = 128;  // tile size of the work lists

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st2(float* p, float x, float y) { *reinterpret_cast<float2*>(p) = make_float2(x, y); }
__device__ __forceinline__ void st2(__nv_bfloat16* p, float x, float y) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(x, y);
}

__device__ __forceinline__ float warp_max(float x) {
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}
__device__ __forceinline__ float warp_sum(float x) {
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// W row groups of R rows, each served by S warps that take every S-th part of
// a streamed block (SB rows) and add up at the end.
template <typename T_, int D_, int R_, int W_, int S_, int SB_>
struct Cfg {
  using T = T_;
  static constexpr int D = D_, R = R_, W = W_, S = S_, SB = SB_;
  static constexpr int TH = W * S * 32, ROWS = R * W;
  static constexpr int BLK = S * SB;     // streamed rows a block
  static constexpr int KPL = SB / 32;    // of a warp's part per lane
  static constexpr int DPL = D / 32;     // accumulator columns per lane
  static constexpr int LD = D + 4;       // padded row of a streamed tile
  static constexpr int NV = BLK * D / 4 / TH;  // float4 of a streamed tile per thread
  static constexpr int SUB = kTileRows / ROWS;
  // floats: own rows, streamed tiles, weights
  static constexpr int OWN = ROWS * D, TILE = BLK * LD, WGT = ROWS * BLK;
  static_assert(BLK * D / 4 % TH == 0 && (R % S == 0 || S == 1), "whole loads and rows");
  static_assert(S * ROWS * (D + 2) <= 2 * TILE, "the partial sums fit the streamed tiles");
};

// A streamed tile on its way from global memory (registers) to shared memory.
template <class C>
struct Stage {
  float4 r[C::NV];
  template <class Row>
  __device__ __forceinline__ void load(const typename C::T* base, int n, Row row_ptr_offset) {
#pragma unroll
    for (int i = 0; i < C::NV; ++i) {
      const int e = threadIdx.x + i * C::TH, row = e / (C::D / 4), c = e % (C::D / 4);
      r[i] = row < n ? ld4(base + row_ptr_offset(row) + c * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __device__ __forceinline__ void store(float* tile) const {
#pragma unroll
    for (int i = 0; i < C::NV; ++i) {
      const int e = threadIdx.x + i * C::TH, row = e / (C::D / 4), c = e % (C::D / 4);
      *reinterpret_cast<float4*>(tile + row * C::LD + c * 4) = r[i];
    }
  }
};

// The warp's own rows [first, first + R) into shared memory (lanes over columns), zero past n_rows.
template <class C>
__device__ __forceinline__ void load_own(float* dst, const typename C::T* base, int64_t stride, int first,
                                         int n_rows) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < C::R * C::D / 128; ++i) {
    const int e = lane + 32 * i, row = e / (C::D / 4), c = e % (C::D / 4);
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (first + row < n_rows) x = ld4(base + (first + row) * stride + c * 4);
    *reinterpret_cast<float4*>(dst + row * C::D + c * 4) = x;
  }
}

// s[r][j] = own row r . streamed row (lane + 32 j)
template <class C>
__device__ __forceinline__ void dots(const float* own, const float* tile, float (&s)[C::R][C::KPL]) {
  const float* t = tile + (threadIdx.x & 31) * C::LD;  // (the warp's part of the tile)
#pragma unroll
  for (int r = 0; r < C::R; ++r)
#pragma unroll
    for (int j = 0; j < C::KPL; ++j) s[r][j] = 0.f;
#pragma unroll 4
  for (int d = 0; d < C::D; d += 4) {
    float4 k[C::KPL];
#pragma unroll
    for (int j = 0; j < C::KPL; ++j) k[j] = ld4(t + j * 32 * C::LD + d);
#pragma unroll
    for (int r = 0; r < C::R; ++r) {
      const float4 q = ld4(own + r * C::D + d);
#pragma unroll
      for (int j = 0; j < C::KPL; ++j)
        s[r][j] = fmaf(q.x, k[j].x, fmaf(q.y, k[j].y, fmaf(q.z, k[j].z, fmaf(q.w, k[j].w, s[r][j]))));
    }
  }
}

// acc[r][:] += sum over streamed rows n of w[r][n] * tile[n][lane's columns].
// kMasked: only over the rows n with lo[r] <= n < hi[r] (a NaN or Inf in a row
// that r does not see stays out of it); else over all, with weight 0 where
// unseen.  Only blocks on the mask's edge pay for the selects.
template <class C, bool kMasked>
__device__ __forceinline__ void accumulate(const float* w, const float* tile, float (&acc)[C::R][C::DPL],
                                           const int (&lo)[C::R], const int (&hi)[C::R]) {
  const float* t = tile + (threadIdx.x & 31) * C::DPL;
#pragma unroll 2
  for (int n = 0; n < C::SB; n += 4) {
    float v[4][C::DPL];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if constexpr (C::DPL == 2) {
        const float2 x = *reinterpret_cast<const float2*>(t + (n + e) * C::LD);
        v[e][0] = x.x; v[e][1] = x.y;
      } else {
        const float4 x = ld4(t + (n + e) * C::LD);
        v[e][0] = x.x; v[e][1] = x.y; v[e][2] = x.z; v[e][3] = x.w;
      }
    }
#pragma unroll
    for (int r = 0; r < C::R; ++r) {
      const float4 p = ld4(w + r * C::SB + n);
      if constexpr (kMasked) {
        const float pe[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
        for (int e = 3; e >= 0; --e)
          if (n + e >= lo[r] && n + e < hi[r])
#pragma unroll
            for (int i = 0; i < C::DPL; ++i) acc[r][i] = fmaf(pe[e], v[e][i], acc[r][i]);
      } else {
#pragma unroll
        for (int i = 0; i < C::DPL; ++i)
          acc[r][i] = fmaf(p.x, v[0][i], fmaf(p.y, v[1][i], fmaf(p.z, v[2][i], fmaf(p.w, v[3][i], acc[r][i]))));
      }
    }
  }
}

// The visible streamed rows [0, hi) of the warp's query rows in its part of a
// block, which starts at key kb; whether every (row, key) of it is visible.
template <class C>
__device__ __forceinline__ bool visible_keys(const int (&ke)[C::R], int kb, int (&lo)[C::R], int (&hi)[C::R]) {
  bool all = true;
#pragma unroll
  for (int r = 0; r < C::R; ++r) {
    lo[r] = 0;
    hi[r] = ke[r] - kb;
    all = all && hi[r] >= C::SB;
  }
  return all;
}

template <class C>
__device__ __forceinline__ void store_row(typename C::T* row, const float (&x)[C::DPL], float f) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < C::DPL; i += 2) st2(row + lane * C::DPL + i, x[i] * f, x[i + 1] * f);
}

// Adds up acc over the S warps of each row group, in `red` (S * ROWS * D
// floats, free for every warp of the block); the warp of part sw then holds
// rows r = sw, sw + S, ... .  scale(r, s) weights part s of row r.
template <class C, class F>
__device__ __forceinline__ void add_parts(float* red, float (&acc)[C::R][C::DPL], int rw, int sw, F scale) {
  if constexpr (C::S > 1) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < C::R; ++r)
#pragma unroll
      for (int i = 0; i < C::DPL; ++i) red[((sw * C::W + rw) * C::R + r) * C::D + lane * C::DPL + i] = acc[r][i];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < C::R; ++r) {
      if (r % C::S != sw) continue;
#pragma unroll
      for (int i = 0; i < C::DPL; ++i) acc[r][i] = 0.f;
#pragma unroll
      for (int s = 0; s < C::S; ++s) {
        const float f = scale(r, s);
#pragma unroll
        for (int i = 0; i < C::DPL; ++i)
          acc[r][i] = fmaf(f, red[((s * C::W + rw) * C::R + r) * C::D + lane * C::DPL + i], acc[r][i]);
      }
    }
    __syncthreads();  // red is free again
  }
}

// The rows of block `b` of a launch over n_heads x tiles x SUB: the head is
// the fastest index, the tiles come in cost order (tile_at).
template <class C, class At>
__device__ __forceinline__ Tile own_rows(const Tile* tiles, At tile_at, int n_heads, int* head, int* row0) {
  const int64_t b = blockIdx.x;
  *head = (int)(b % n_heads);
  const int64_t t = b / n_heads;
  const Tile w = tiles[tile_at(t / C::SUB)];
  *row0 = w.tile * kTileRows + (int)(t % C::SUB) * C::ROWS;
  return w;
}

template <class C>
__global__ void __launch_bounds__(C::TH) simt_fwd_kernel(const AttnArgs a) {
  using T = typename C::T;
  pdl_wait();
  advance_cache_len(a);
  extern __shared__ __align__(16) float sm[];
  float *own = sm, *kt = own + C::OWN, *vt = kt + C::TILE, *wt = vt + C::TILE;
  int h, row0;
  const Tile w = own_rows<C>(a.qtiles, [&](int64_t p) { return q_tile_at(a, p); }, a.hq, &h, &row0);
  if (row0 >= w.q_len) return;
  const int g = h / (a.hq / a.hkv);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rw = warp % C::W, sw = warp / C::W;
  const int64_t qstride = (int64_t)a.hq * C::D, kstride = (int64_t)a.hkv * C::D;
  const T* K = static_cast<const T*>(a.k) + (int64_t)g * C::D;
  const T* V = static_cast<const T*>(a.v) + (int64_t)g * C::D;
  const int r0 = row0 + rw * C::R;  // the warp's first row
  float* myq = own + rw * C::R * C::D;
  float* myw = wt + warp * C::R * C::SB;
  if (sw == 0) load_own<C>(myq, static_cast<const T*>(a.q) + (int64_t)w.q_base * qstride + (int64_t)h * C::D, qstride, r0, w.q_len);
  int ke[C::R];
#pragma unroll
  for (int r = 0; r < C::R; ++r) ke[r] = r0 + r < w.q_len ? a.kv_end[w.kv_base + r0 + r] : 0;
  // kv_end does not decrease: the block's last row sees the most keys
  const int n_keys = a.kv_end[w.kv_base + min(row0 + C::ROWS, w.q_len) - 1];
  float m[C::R], l[C::R], acc[C::R][C::DPL];  // l: this lane's share of the sum
#pragma unroll
  for (int r = 0; r < C::R; ++r) {
    m[r] = -INFINITY;
    l[r] = 0.f;
#pragma unroll
    for (int i = 0; i < C::DPL; ++i) acc[r][i] = 0.f;
  }
  Stage<C> sk, sv;
  auto fetch = [&](int kb) {
    auto at = [&](int row) -> int64_t {  // through the page table for a paged cache
      return (a.pages.table ? paged_row(a.pages, w.k_base, kb + row) : (int64_t)w.k_base + kb + row) * kstride;
    };
    sk.load(K, n_keys - kb, at);
    sv.load(V, n_keys - kb, at);
  };
  fetch(0);
  for (int kb = 0; kb < n_keys; kb += C::BLK) {
    __syncthreads();
    sk.store(kt);
    sv.store(vt);
    __syncthreads();
    if (kb + C::BLK < n_keys) fetch(kb + C::BLK);
    float s[C::R][C::KPL];
    const int k0 = kb + sw * C::SB;  // this warp's part
    dots<C>(myq, kt + sw * C::SB * C::LD, s);
#pragma unroll
    for (int r = 0; r < C::R; ++r) {
      float mx = -INFINITY;
#pragma unroll
      for (int j = 0; j < C::KPL; ++j) {
        s[r][j] = k0 + lane + 32 * j < ke[r] ? s[r][j] * a.scale : -INFINITY;
        mx = fmaxf(mx, s[r][j]);
      }
      const float mn = fmaxf(m[r], warp_max(mx));
      const float alpha = m[r] == -INFINITY ? 0.f : expf(m[r] - mn);
      l[r] *= alpha;
#pragma unroll
      for (int j = 0; j < C::KPL; ++j) {
        const float p = k0 + lane + 32 * j < ke[r] ? expf(s[r][j] - mn) : 0.f;
        l[r] += p;
        myw[r * C::SB + lane + 32 * j] = p;
      }
#pragma unroll
      for (int i = 0; i < C::DPL; ++i) acc[r][i] *= alpha;
      m[r] = mn;
    }
    __syncwarp();
    int lo[C::R], hi[C::R];
    if (visible_keys<C>(ke, k0, lo, hi))
      accumulate<C, false>(myw, vt + sw * C::SB * C::LD, acc, lo, hi);
    else
      accumulate<C, true>(myw, vt + sw * C::SB * C::LD, acc, lo, hi);
    __syncwarp();
  }
#pragma unroll
  for (int r = 0; r < C::R; ++r) l[r] = warp_sum(l[r]);
  if constexpr (C::S > 1) {
    // each part has its own maximum and sum: (m, l) of part s, row r
    __syncthreads();
    float* ml = kt + C::S * C::OWN;
    if (lane == 0)
#pragma unroll
      for (int r = 0; r < C::R; ++r) {
        ml[((sw * C::W + rw) * C::R + r) * 2] = m[r];
        ml[((sw * C::W + rw) * C::R + r) * 2 + 1] = l[r];
      }
    __syncthreads();
    float f[C::R][C::S];
#pragma unroll
    for (int r = 0; r < C::R; ++r) {
      float ms[C::S], ls[C::S], top = -INFINITY, sum = 0.f;
#pragma unroll
      for (int i = 0; i < C::S; ++i) {
        ms[i] = ml[((i * C::W + rw) * C::R + r) * 2];
        ls[i] = ml[((i * C::W + rw) * C::R + r) * 2 + 1];
        top = fmaxf(top, ms[i]);
      }
#pragma unroll
      for (int i = 0; i < C::S; ++i) {
        f[r][i] = ms[i] == -INFINITY && ls[i] == 0.f ? 0.f : expf(ms[i] - top);  // no visible key: nothing
        sum = fmaf(f[r][i], ls[i], sum);
      }
      m[r] = top;
      l[r] = sum;
    }
    add_parts<C>(kt, acc, rw, sw, [&](int r, int i) { return f[r][i]; });
  }
#pragma unroll
  for (int r = 0; r < C::R; ++r) {
    if (r % C::S != sw || r0 + r >= w.q_len) continue;
    const int64_t qrow = (int64_t)w.q_base + r0 + r;
    store_row<C>(static_cast<T*>(a.out) + qrow * qstride + (int64_t)h * C::D, acc[r], 1.f / l[r]);
    if (a.lse && lane == 0) a.lse[(int64_t)h * a.q_rows + qrow] = m[r] + logf(l[r]);
  }
}

// dQ, and Delta = rowsum(dO * O) of its rows, which the dK/dV kernel reads.
template <class C>
__global__ void __launch_bounds__(C::TH) simt_dq_kernel(const AttnArgs a) {
  using T = typename C::T;
  pdl_wait();
  extern __shared__ __align__(16) float sm[];
  float *own_q = sm, *own_do = own_q + C::OWN, *kt = own_do + C::OWN, *vt = kt + C::TILE, *wt = vt + C::TILE;
  int h, row0;
  const Tile w = own_rows<C>(a.qtiles, [&](int64_t p) { return q_tile_at(a, p); }, a.hq, &h, &row0);
  if (row0 >= w.q_len) return;
  const int g = h / (a.hq / a.hkv);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rw = warp % C::W, sw = warp / C::W;
  const int64_t qstride = (int64_t)a.hq * C::D, kstride = (int64_t)a.hkv * C::D;
  const int64_t qoff = (int64_t)w.q_base * qstride + (int64_t)h * C::D;
  const T* K = static_cast<const T*>(a.k) + (int64_t)w.k_base * kstride + (int64_t)g * C::D;
  const T* V = static_cast<const T*>(a.v) + (int64_t)w.k_base * kstride + (int64_t)g * C::D;
  const int n_keys = a.kv_end[w.kv_base + min(row0 + C::ROWS, w.q_len) - 1];
  Stage<C> sk, sv;
  auto fetch = [&](int kb) {
    auto at = [&](int row) -> int64_t { return (int64_t)(kb + row) * kstride; };
    sk.load(K, n_keys - kb, at);
    sv.load(V, n_keys - kb, at);
  };
  fetch(0);
  const int r0 = row0 + rw * C::R;
  float* myq = own_q + rw * C::R * C::D;
  float* mydo = own_do + rw * C::R * C::D;
  float* myw = wt + warp * C::R * C::SB;
  if (sw == 0) load_own<C>(myq, static_cast<const T*>(a.q) + qoff, qstride, r0, w.q_len);
  if (sw == C::S - 1) load_own<C>(mydo, static_cast<const T*>(a.dout) + qoff, qstride, r0, w.q_len);
  __syncthreads();
  int ke[C::R];
  float lse[C::R], dl[C::R], acc[C::R][C::DPL];
#pragma unroll
  for (int r = 0; r < C::R; ++r) {
    const bool valid = r0 + r < w.q_len;
    const int64_t qrow = (int64_t)w.q_base + r0 + r;
    ke[r] = valid ? a.kv_end[w.kv_base + r0 + r] : 0;
    lse[r] = valid ? a.lse_in[(int64_t)h * a.q_rows + qrow] : 0.f;
    float d = 0.f;
    if (valid && lane < C::D / 4) {
      const float4 o = ld4(static_cast<const T*>(a.o) + qrow * qstride + (int64_t)h * C::D + lane * 4);
      const float4 x = ld4(mydo + r * C::D + lane * 4);
      d = fmaf(o.x, x.x, fmaf(o.y, x.y, fmaf(o.z, x.z, o.w * x.w)));
    }
    dl[r] = warp_sum(d);
    if (valid && lane == 0 && sw == 0) a.delta[(int64_t)h * a.q_rows + qrow] = dl[r];
#pragma unroll
    for (int i = 0; i < C::DPL; ++i) acc[r][i] = 0.f;
  }
  for (int kb = 0; kb < n_keys; kb += C::BLK) {
    __syncthreads();
    sk.store(kt);
    sv.store(vt);
    __syncthreads();
    if (kb + C::BLK < n_keys) fetch(kb + C::BLK);
    float s[C::R][C::KPL], dp[C::R][C::KPL];
    const int k0 = kb + sw * C::SB;  // this warp's part
    dots<C>(myq, kt + sw * C::SB * C::LD, s);
    dots<C>(mydo, vt + sw * C::SB * C::LD, dp);
#pragma unroll
    for (int r = 0; r < C::R; ++r)
#pragma unroll
      for (int j = 0; j < C::KPL; ++j) {
        const float p = expf(a.scale * s[r][j] - lse[r]);
        myw[r * C::SB + lane + 32 * j] = k0 + lane + 32 * j < ke[r] ? p * (dp[r][j] - dl[r]) : 0.f;
      }
    __syncwarp();
    int lo[C::R], hi[C::R];
    if (visible_keys<C>(ke, k0, lo, hi))
      accumulate<C, false>(myw, kt + sw * C::SB * C::LD, acc, lo, hi);
    else
      accumulate<C, true>(myw, kt + sw * C::SB * C::LD, acc, lo, hi);
    __syncwarp();
  }
  if (C::S > 1) __syncthreads();
  add_parts<C>(kt, acc, rw, sw, [](int, int) { return 1.f; });
#pragma unroll
  for (int r = 0; r < C::R; ++r)
    if (r % C::S == sw && r0 + r < w.q_len)
      store_row<C>(static_cast<T*>(a.dq) + qoff + (r0 + r) * qstride, acc[r], a.scale);
}

// dK, dV of a block of keys: walks the query heads of the group and the query
// rows that see the block (kv_end does not decrease: from the first row whose
// bound exceeds the first key to the end of the sequence).
template <class C>
__global__ void __launch_bounds__(C::TH) simt_dkdv_kernel(const AttnArgs a) {
  using T = typename C::T;
  pdl_wait();
  extern __shared__ __align__(16) float sm[];
  float *own_k = sm, *own_v = own_k + C::OWN, *qt = own_v + C::OWN, *dot = qt + C::TILE, *pt = dot + C::TILE,
        *dst = pt + C::WGT;
  int g, key0;
  const Tile w = own_rows<C>(a.ktiles, [&](int64_t p) { return a.k_order[p]; }, a.hkv, &g, &key0);
  if (key0 >= w.k_len) return;
  const int group = a.hq / a.hkv;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rw = warp % C::W, sw = warp / C::W;
  const int64_t qstride = (int64_t)a.hq * C::D, kstride = (int64_t)a.hkv * C::D;
  const int64_t koff = (int64_t)w.k_base * kstride + (int64_t)g * C::D;
  const int32_t* kv_end = a.kv_end + w.kv_base;
  int lo = 0, hi = w.q_len;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (kv_end[mid] > key0) hi = mid; else lo = mid + 1;
  }
  const int j0 = lo, n_blk = (w.q_len - j0 + C::BLK - 1) / C::BLK, n_it = n_blk * group;
  const int k0 = key0 + rw * C::R;
  float* myk = own_k + rw * C::R * C::D;
  float* myv = own_v + rw * C::R * C::D;
  float* myp = pt + warp * C::R * C::SB;
  float* myds = dst + warp * C::R * C::SB;
  Stage<C> sq, sdo;
  // per streamed row of this lane: bound (0 past the end), LSE, Delta
  int ke_n[C::KPL];
  float lse_n[C::KPL], dl_n[C::KPL];
  auto fetch = [&](int it) {
    const int h = g * group + it / n_blk, jb = j0 + it % n_blk * C::BLK;
    const int64_t base = ((int64_t)w.q_base + jb) * qstride + (int64_t)h * C::D;
    auto at = [&](int row) -> int64_t { return (int64_t)row * qstride; };
    sq.load(static_cast<const T*>(a.q) + base, w.q_len - jb, at);
    sdo.load(static_cast<const T*>(a.dout) + base, w.q_len - jb, at);
#pragma unroll
    for (int j = 0; j < C::KPL; ++j) {
      const int row = jb + sw * C::SB + lane + 32 * j;  // of the warp's part
      const bool valid = row < w.q_len;
      const int64_t at_row = (int64_t)h * a.q_rows + w.q_base + row;
      ke_n[j] = valid ? kv_end[row] : 0;
      lse_n[j] = valid ? a.lse_in[at_row] : 0.f;
      dl_n[j] = valid ? a.delta[at_row] : 0.f;
    }
  };
  if (n_it > 0) fetch(0);
  if (sw == 0) load_own<C>(myk, static_cast<const T*>(a.k) + koff, kstride, k0, w.k_len);
  if (sw == C::S - 1) load_own<C>(myv, static_cast<const T*>(a.v) + koff, kstride, k0, w.k_len);
  float ak[C::R][C::DPL], av[C::R][C::DPL];
#pragma unroll
  for (int r = 0; r < C::R; ++r)
#pragma unroll
    for (int i = 0; i < C::DPL; ++i) ak[r][i] = av[r][i] = 0.f;
  for (int it = 0; it < n_it; ++it) {
    __syncthreads();
    sq.store(qt);
    sdo.store(dot);
    int ke[C::KPL];
    float lse[C::KPL], dl[C::KPL];
#pragma unroll
    for (int j = 0; j < C::KPL; ++j) {
      ke[j] = ke_n[j];
      lse[j] = lse_n[j];
      dl[j] = dl_n[j];
    }
    __syncthreads();
    // query rows from the warp's part on
    const int n_q = w.q_len - (j0 + it % n_blk * C::BLK + sw * C::SB);
    if (it + 1 < n_it) fetch(it + 1);
    float s[C::R][C::KPL], dp[C::R][C::KPL];
    const float *qp = qt + sw * C::SB * C::LD, *dop = dot + sw * C::SB * C::LD;
    dots<C>(myk, qp, s);
    dots<C>(myv, dop, dp);
#pragma unroll
    for (int r = 0; r < C::R; ++r)
#pragma unroll
      for (int j = 0; j < C::KPL; ++j) {
        const float p = k0 + r < ke[j] ? expf(a.scale * s[r][j] - lse[j]) : 0.f;
        myp[r * C::SB + lane + 32 * j] = p;
        myds[r * C::SB + lane + 32 * j] = k0 + r < ke[j] ? p * (dp[r][j] - dl[j]) : 0.f;
      }
    __syncwarp();
    // queries from the first one that sees the key on (bounds do not decrease;
    // rows past the end are zeros of weight zero)
    int first[C::R], end[C::R];
    bool all = true;
#pragma unroll
    for (int r = 0; r < C::R; ++r) {
      first[r] = 0;
      end[r] = C::SB;
#pragma unroll
      for (int j = 0; j < C::KPL; ++j)
        first[r] += __popc(__ballot_sync(0xffffffffu, lane + 32 * j < n_q && ke[j] <= k0 + r));
      all = all && first[r] == 0;
    }
    if (all) {
      accumulate<C, false>(myp, dop, av, first, end);
      accumulate<C, false>(myds, qp, ak, first, end);
    } else {
      accumulate<C, true>(myp, dop, av, first, end);
      accumulate<C, true>(myds, qp, ak, first, end);
    }
    __syncwarp();
  }
  if (C::S > 1) __syncthreads();
  add_parts<C>(qt, ak, rw, sw, [](int, int) { return 1.f; });
  add_parts<C>(qt, av, rw, sw, [](int, int) { return 1.f; });
#pragma unroll
  for (int r = 0; r < C::R; ++r)
    if (r % C::S == sw && k0 + r < w.k_len) {
      const int64_t off = koff + (k0 + r) * kstride;
      store_row<C>(static_cast<T*>(a.dk) + off, ak[r], a.scale);
      store_row<C>(static_cast<T*>(a.dv) + off, av[r], 1.f);
    }
}

// Launches `kern` over SUB blocks a (tile, head) with its shared memory.
template <class C, class K>
cudaError_t launch_cfg(K kern, int64_t tiles_heads, int floats, const AttnArgs& a, cudaStream_t st) {
  const int smem = floats * (int)sizeof(float);
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return ism::launch(a.dependent, kern, tiles_heads * C::SUB, C::TH, smem, st, a);
}

// 64 rows a block, or 16 with the streamed side split over four warps while
// blocks of 64 would leave SMs without one.
bool few_blocks(int64_t tiles_heads) { return tiles_heads * 2 < sm_count(); }
template <typename T, int D> using Big = Cfg<T, D, 8, 8, 1, 4096 / D>;
template <typename T, int D> using Small = Cfg<T, D, 4, 4, 4, 32>;

template <class C>
cudaError_t fwd_cfg(const AttnArgs& a, cudaStream_t st) {
  return launch_cfg<C>(simt_fwd_kernel<C>, a.nq * a.hq, C::OWN + 2 * C::TILE + C::WGT, a, st);
}
template <class C>
cudaError_t dq_cfg(const AttnArgs& a, cudaStream_t st) {
  return launch_cfg<C>(simt_dq_kernel<C>, a.nq * a.hq, 2 * C::OWN + 2 * C::TILE + C::WGT, a, st);
}
template <class C>
cudaError_t dkdv_cfg(const AttnArgs& a, cudaStream_t st) {
  return launch_cfg<C>(simt_dkdv_kernel<C>, a.nk * a.hkv, 2 * C::OWN + 2 * C::TILE + 2 * C::WGT, a, st);
}

template <typename T, int D>
cudaError_t fwd_impl(const AttnArgs& a, cudaStream_t st) {
  if (a.nq == 0) return cudaSuccess;
  return few_blocks(a.nq * a.hq) ? fwd_cfg<Small<T, D>>(a, st) : fwd_cfg<Big<T, D>>(a, st);
}

template <typename T, int D>
cudaError_t bwd_impl(const AttnArgs& a, cudaStream_t st) {
  if (a.q_rows == 0) return cudaSuccess;
  cudaError_t e;
  if (a.nq) {
    timer_begin(ISM_KERNEL_BWD_DQ, st);
    e = few_blocks(a.nq * a.hq) ? dq_cfg<Small<T, D>>(a, st) : dq_cfg<Big<T, D>>(a, st);
    timer_end(ISM_KERNEL_BWD_DQ, st);
    count_launch();
    if (e != cudaSuccess) return e;
  }
  if (a.nk) {
    timer_begin(ISM_KERNEL_BWD_DKDV, st);
    e = few_blocks(a.nk * a.hkv) ? dkdv_cfg<Small<T, D>>(a, st) : dkdv_cfg<Big<T, D>>(a, st);
    timer_end(ISM_KERNEL_BWD_DKDV, st);
    count_launch();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_simt_fwd(const AttnArgs& a, cudaStream_t st) {
  if (a.dtype == ISM_FP32) return a.d == 64 ? fwd_impl<float, 64>(a, st) : fwd_impl<float, 128>(a, st);
  return a.d == 64 ? fwd_impl<__nv_bfloat16, 64>(a, st) : fwd_impl<__nv_bfloat16, 128>(a, st);
}

cudaError_t launch_simt_bwd(const AttnArgs& a, cudaStream_t st) {
  if (a.dtype == ISM_FP32) return a.d == 64 ? bwd_impl<float, 64>(a, st) : bwd_impl<float, 128>(a, st);
  return a.d == 64 ? bwd_impl<__nv_bfloat16, 64>(a, st) : bwd_impl<__nv_bfloat16, 128>(a, st);
}

}  // namespace ism
