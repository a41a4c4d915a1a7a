// Segment metadata kernels: per-token key bound kv_end (Eq. fj, Section 2.1),
// the (q-tile, k-tile) classification, work lists for the attention kernels
// ordered most expensive first, and the append-prefill plan (Section 2.3).
#include "ism_internal.cuh"

namespace ism {
namespace {

__device__ __forceinline__ int upper_bound_i32(const int32_t* a, int n, int32_t x) {
  // first index i in [0, n) with a[i] > x (n if none); a non-decreasing
  int lo = 0, hi = n;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (a[mid] > x) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// Inclusive prefix sum of one value per thread over the block (blockDim.x a
// multiple of 32, at most 1024): shuffle scans within each warp, then warp 0
// scans the warp totals.  *total receives the block's sum.  Every thread of
// the block calls it (it holds __syncthreads).
template <typename T>
__device__ T block_inclusive_scan(T v, T* total) {
  __shared__ T wsum[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  if (lane == 31) wsum[warp] = v;
  __syncthreads();
  if (warp == 0) {
    T w = lane < nw ? wsum[lane] : T(0);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T t = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += t;
    }
    wsum[lane] = w;  // inclusive over the warps
  }
  __syncthreads();
  const T add = warp > 0 ? wsum[warp - 1] : T(0);
  *total = wsum[nw - 1];
  __syncthreads();  // wsum is free for the next call
  return v + add;
}

// Per-sequence tile offsets computed by every block into shared memory:
// qoff/koff [B+1] (q-tiles / k-tiles before sequence b) and toff [B+1]
// (tile_class bytes before sequence b).  Block-wide scans over chunks of
// blockDim.x sequences with a running carry.
__device__ void seq_offsets_smem(const SegsDev& s, int bm, int bn, int32_t* qoff, int32_t* koff, int64_t* toff) {
  if (threadIdx.x == 0) { qoff[0] = 0; koff[0] = 0; toff[0] = 0; }
  int32_t cq = 0, ck = 0;  // carries, the same in every thread
  int64_t ct = 0;
  for (int base = 0; base < s.num_seqs; base += blockDim.x) {
    const int b = base + threadIdx.x;
    int32_t nq = 0, nk = 0;
    if (b < s.num_seqs) {
      const int32_t L = s.cu_seqlens[b + 1] - s.cu_seqlens[b];
      nq = (L + bm - 1) / bm;
      nk = (L + bn - 1) / bn;
    }
    int32_t tq, tk;
    int64_t tt;
    const int32_t iq = block_inclusive_scan<int32_t>(nq, &tq), ik = block_inclusive_scan<int32_t>(nk, &tk);
    const int64_t it = block_inclusive_scan<int64_t>((int64_t)nq * nk, &tt);
    if (b < s.num_seqs) {
      qoff[b + 1] = cq + iq;
      koff[b + 1] = ck + ik;
      toff[b + 1] = ct + it;
    }
    cq += tq;
    ck += tk;
    ct += tt;
  }
  __syncthreads();
}

// kv_end of every token (Eq. fj): a token of a query segment is bounded by
// the end of its segment, a token of an answer segment by itself.  One block
// per segment (grid-stride); threads over the segment's tokens.
__global__ void kv_end_kernel(SegsDev s, int32_t* kv_end) {
  for (int seg = blockIdx.x; seg < s.num_segs; seg += gridDim.x) {
    int b = upper_bound_i32(s.cu_segs, s.num_seqs + 1, seg) - 1;
    int32_t start = seg > s.cu_segs[b] ? s.seg_end[seg - 1] : 0;
    int32_t end = s.seg_end[seg];
    int32_t base = s.cu_seqlens[b];
    bool query = s.seg_type[seg] == ISM_SEG_QUERY;
    for (int32_t j = start + threadIdx.x; j < end; j += blockDim.x)
      kv_end[base + j] = query ? end : j + 1;
  }
}

// q-tile and k-tile descriptors plus the optional public tile-map arrays.
// Since kv_end is non-decreasing within a sequence, q-tile t has
// floor(kv_end[first row] / bn) leading FULL tiles when all of its rows lie
// inside the sequence (0 otherwise), and ceil(kv_end[last row] / bn)
// non-empty tiles; k-tile c is first reached by the q-tile holding the first
// row whose kv_end exceeds c*bn.
// `dyn` holds the per-sequence offsets ((num_seqs + 1) * 16 bytes).
__device__ void tiles_body(const SegsDev& s, int bm, int bn, const int32_t* kv_end, int64_t nq,
                           int64_t nk, Tile* qtiles, Tile* ktiles, uint8_t* tile_class, int32_t* kt_full_end,
                           int32_t* kt_end, int32_t* qt_begin, unsigned char* dyn) {
  int64_t* toff = reinterpret_cast<int64_t*>(dyn);
  int32_t* qoff = reinterpret_cast<int32_t*>(toff + s.num_seqs + 1);
  int32_t* koff = qoff + s.num_seqs + 1;
  seq_offsets_smem(s, bm, bn, qoff, koff, toff);
  int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < nq; g += stride) {
    int b = upper_bound_i32(qoff, s.num_seqs + 1, (int32_t)g) - 1;
    int32_t t = (int32_t)g - qoff[b];
    int32_t base = s.cu_seqlens[b];
    int32_t L = s.cu_seqlens[b + 1] - base;
    int32_t r0 = t * bm;
    int32_t rl = min(L, r0 + bm) - 1;
    int32_t full = (r0 + bm <= L) ? kv_end[base + r0] / bn : 0;
    int32_t ne = (kv_end[base + rl] + bn - 1) / bn;
    if (qtiles) {
      Tile w;
      w.q_base = base; w.k_base = base; w.q_len = L; w.k_len = L; w.tile = t;
      w.a0 = full; w.a1 = ne; w.kv_base = base;
      qtiles[g] = w;
    }
    if (kt_full_end) kt_full_end[g] = full;
    if (kt_end) kt_end[g] = ne;
    if (tile_class) {
      int32_t nkt = (L + bn - 1) / bn;
      uint8_t* row = tile_class + toff[b] + (int64_t)t * nkt;
      for (int32_t c = 0; c < nkt; ++c)
        row[c] = c < full ? (uint8_t)ISM_TILE_FULL : c < ne ? (uint8_t)ISM_TILE_PARTIAL : (uint8_t)ISM_TILE_EMPTY;
    }
  }
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < nk; g += stride) {
    int b = upper_bound_i32(koff, s.num_seqs + 1, (int32_t)g) - 1;
    int32_t c = (int32_t)g - koff[b];
    int32_t base = s.cu_seqlens[b];
    int32_t L = s.cu_seqlens[b + 1] - base;
    // first row that sees key x = c*bn: kv_end is non-decreasing, and under
    // Eq. fj the first segment ending after x starts that row when it is a
    // query segment, else the row is max(segment start, x)
    const int32_t x = c * bn;
    const int s0 = s.cu_segs[b], s1 = s.cu_segs[b + 1];
    const int seg = s0 + upper_bound_i32(s.seg_end + s0, s1 - s0, x);
    const int32_t start = seg > s0 ? s.seg_end[seg - 1] : 0;
    int32_t j = s.seg_type[seg] == ISM_SEG_QUERY ? start : (x > start ? x : start);
    int32_t qb = j / bm;
    if (qt_begin) qt_begin[g] = qb;
    if (ktiles) {
      Tile w;
      w.q_base = base; w.k_base = base; w.q_len = L; w.k_len = L; w.tile = c;
      w.a0 = qb; w.a1 = (L + bm - 1) / bm; w.kv_base = base;
      ktiles[g] = w;
    }
  }
}

__global__ void __launch_bounds__(256) tiles_kernel(SegsDev s, int bm, int bn, const int32_t* kv_end,
                             int64_t nq, int64_t nk, Tile* qtiles, Tile* ktiles, uint8_t* tile_class,
                             int32_t* kt_full_end, int32_t* kt_end, int32_t* qt_begin) {
  extern __shared__ __align__(16) unsigned char dyn[];
  tiles_body(s, bm, bn, kv_end, nq, nk, qtiles, ktiles, tile_class, kt_full_end, kt_end, qt_begin, dyn);
}

// Work lists ordered by decreasing cost (counting sort, one block).  Cost of
// a q-tile = its non-empty k-tiles; of a k-tile = its non-empty q-tiles.  The
// optional third list holds the q-tiles with an even index in their sequence
// (the first of each pair of neighbouring q-tiles), costed by the pair's
// larger count (the second tile's, kv_end being non-decreasing); the optional
// fourth the k-tiles with an even index (pairs of neighbouring k-tiles),
// costed by the first tile's count, which covers the second's (its first
// non-empty q-tile comes no earlier).
// Items of equal cost come in arbitrary order; results do not depend on it.
__device__ __forceinline__ bool pair_head(const Tile* qtiles, int64_t nq, int64_t i, int* cost) {
  const Tile w = qtiles[i];
  if (w.tile & 1) return false;
  int c = w.a1;
  if (i + 1 < nq) {
    const Tile n = qtiles[i + 1];
    if (n.q_base == w.q_base && n.tile == w.tile + 1) c = max(c, n.a1);
  }
  *cost = c;
  return true;
}

// pairs_first: q_order lists the pair heads of the third list first (in its
// order), then the odd-indexed q-tiles; the forward of an odd group at
// head_dim 64 reads its pairs from there.
__device__ void order_body(const Tile* qtiles, int64_t nq, const Tile* ktiles, int64_t nk,
                           int max_cost, int32_t* q_order, int32_t* k_order, int32_t* pair_order, int32_t* hist,
                           int32_t* kp_order = nullptr, bool pairs_first = false) {
  int32_t heads = 0;  // pair heads listed at the front of q_order (pairs_first)
  for (int pass = 0; pass < 5; ++pass) {
    const bool keys = pass == 1 || pass == 3;
    const Tile* items = keys ? ktiles : qtiles;
    const int64_t n = keys ? nk : nq;
    int32_t* order = pass == 0 ? q_order : pass == 1 ? k_order : pass == 2 ? pair_order : pass == 3 ? kp_order
                     : pairs_first && q_order ? q_order + heads : nullptr;
    if (items == nullptr || order == nullptr || n == 0) continue;
    // cost of item i in this pass (false: not listed in it)
    auto cost_of = [&](int64_t i, int* cost) -> bool {
      if (pass == 2 || (pass == 0 && pairs_first)) {
        if (!pair_head(items, n, i, cost)) return false;
      } else {
        const Tile w = items[i];
        if (pass == 3 && (w.tile & 1)) return false;   // k-tile pairs: the even tile, costed by its query tiles
        if (pass == 4 && !(w.tile & 1)) return false;  // the odd q-tiles
        *cost = keys ? w.a1 - w.a0 : w.a1;
      }
      *cost = min(max(*cost, 0), max_cost);
      return true;
    };
    for (int i = threadIdx.x; i <= max_cost; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
      int cost;
      if (cost_of(i, &cost)) atomicAdd(&hist[cost], 1);
    }
    __syncthreads();
    // exclusive scan from the highest cost down (each thread rewrites the
    // entries it read, so no barrier is needed between the read and the write)
    int32_t run = 0;
    for (int base = 0; base <= max_cost; base += blockDim.x) {
      const int c = max_cost - (base + (int)threadIdx.x);
      const int32_t h = c >= 0 ? hist[c] : 0;
      int32_t tot;
      const int32_t incl = block_inclusive_scan<int32_t>(h, &tot);
      if (c >= 0) hist[c] = run + incl - h;
      run += tot;
    }
    if (pass == 0) heads = run;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
      int cost;
      if (cost_of(i, &cost)) order[atomicAdd(&hist[cost], 1)] = (int32_t)i;
    }
    __syncthreads();
  }
}

// Exclusive prefix over k-tiles of their non-empty q-tile counts (a1 - a0):
// the first (k-tile, q-tile) pair slot of each k-tile.  One block, chunks of
// blockDim.x with a running carry.
__device__ void pair_offsets_body(const Tile* ktiles, int64_t nk, int32_t* kpair_off) {
  int32_t carry = 0;  // the same in every thread
  for (int64_t base = 0; base < nk; base += blockDim.x) {
    const int64_t i = base + threadIdx.x;
    int32_t v = 0;
    if (i < nk) {
      const Tile w = ktiles[i];
      v = w.a1 - w.a0 > 0 ? w.a1 - w.a0 : 0;
    }
    int32_t tot;
    const int32_t incl = block_inclusive_scan<int32_t>(v, &tot);
    if (i < nk) kpair_off[i] = carry + incl - v;
    carry += tot;
  }
}

// All metadata of one attention pass in a single block: kv_end per token
// (Eq. fj, a warp per segment), the q-/k-tile descriptors, the cost-ordered work lists and, for
// the stored-dS backward, the pair offsets.  Global writes of one phase are
// visible to the block's threads after __syncthreads.
__global__ void __launch_bounds__(1024)
    pass_meta_kernel(SegsDev s, int32_t* kv_end, int bm, int bn, int64_t nq, int64_t nk, Tile* qtiles,
                     Tile* ktiles, int max_cost, int32_t* q_order, int32_t* k_order, int32_t* pair_order,
                     int32_t* kpair_off, int32_t* counters, int n_counters, int32_t* kp_order, bool pairs_first) {
  extern __shared__ __align__(16) unsigned char dyn[];
  pdl_wait();
  if ((int)threadIdx.x < n_counters) counters[threadIdx.x] = 0;  // work counters of the kernels that follow
  // kv_end: one warp per segment, lanes over its tokens
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  for (int seg = warp; seg < s.num_segs; seg += nwarps) {
    const int b = upper_bound_i32(s.cu_segs, s.num_seqs + 1, seg) - 1;
    const int32_t start = seg > s.cu_segs[b] ? s.seg_end[seg - 1] : 0;
    const int32_t end = s.seg_end[seg];
    const int32_t base = s.cu_seqlens[b];
    const bool query = s.seg_type[seg] == ISM_SEG_QUERY;
    for (int32_t j = start + lane; j < end; j += 32) kv_end[base + j] = query ? end : j + 1;
  }
  __syncthreads();
  tiles_body(s, bm, bn, kv_end, nq, nk, qtiles, ktiles, nullptr, nullptr, nullptr, nullptr, dyn);
  __syncthreads();
  order_body(qtiles, nq, ktiles, nk, max_cost, q_order, k_order, pair_order, reinterpret_cast<int32_t*>(dyn),
             kp_order, pairs_first);
  if (kpair_off) pair_offsets_body(ktiles, nk, kpair_off);
}

// The same for a small batch (at most kSmallTiles tiles and sequences and
// kSmallSegs segments, bm == bn): the segments are read into shared memory
// once, every bound, descriptor, rank and offset is computed there and in
// registers, one thread a tile, and the results are written at the end.  The
// ranks are counted by comparing every pair of tiles.  The general pass goes
// through global memory and some twenty block barriers of 1024 threads: one
// dialogue of 256 tokens 8.0 us, this one 5.0; 2 x 8192 tokens 11.5 and 10.
constexpr int kSmallTiles = 256, kSmallSegs = 1024, kSmallThreads = 512;

// How many of the n costs come before cost c of item i in the list (higher
// first, equal ones by index); costs below zero are not listed.
__device__ __forceinline__ int rank_of(const int32_t* costs, int n, int32_t c, int i) {
  int r = 0;
  for (int j = 0; j < n; j += 4) {  // (n rounded up: the padding is negative)
    const int4 v = *reinterpret_cast<const int4*>(costs + j);
    r += (v.x > c || (v.x == c && j < i)) + (v.y > c || (v.y == c && j + 1 < i)) +
         (v.z > c || (v.z == c && j + 2 < i)) + (v.w > c || (v.w == c && j + 3 < i));
  }
  return r;
}

__global__ void __launch_bounds__(kSmallThreads)
    pass_meta_small_kernel(SegsDev s, int32_t* kv_end, int bm, int nq, Tile* qtiles, Tile* ktiles, int32_t* q_order,
                           int32_t* k_order, int32_t* pair_order, int32_t* kpair_off, int32_t* counters,
                           int n_counters, bool pairs_first) {
  __shared__ int32_t cu[kSmallTiles + 1], cseg[kSmallTiles + 1], off[kSmallTiles + 1], ends[kSmallSegs];
  __shared__ uint8_t types[kSmallSegs];
  // per list: q-tiles, k-tiles, pair heads, odd q-tiles; -1 where not listed
  __shared__ __align__(16) int32_t cost[4][kSmallTiles + 4];
  const int tid = threadIdx.x;
  pdl_wait();
  for (int i = tid; i <= s.num_seqs; i += kSmallThreads) {
    cu[i] = s.cu_seqlens[i];
    cseg[i] = s.cu_segs[i];
  }
  for (int i = tid; i < s.num_segs; i += kSmallThreads) {
    ends[i] = s.seg_end[i];
    types[i] = s.seg_type[i];
  }
  for (int i = tid; i < 4 * (kSmallTiles + 4); i += kSmallThreads) (&cost[0][0])[i] = -1;
  __syncthreads();
  int32_t total;
  const int32_t n_b = tid < s.num_seqs ? (cu[tid + 1] - cu[tid] + bm - 1) / bm : 0;
  const int32_t incl = block_inclusive_scan<int32_t>(n_b, &total);
  if (tid < s.num_seqs) off[tid + 1] = incl;
  if (tid == 0) off[0] = 0;
  __syncthreads();
  // segment of row (or key) x of sequence b, and the row's key bound (Eq. fj)
  auto seg_of = [&](int b, int x) { return cseg[b] + upper_bound_i32(ends + cseg[b], cseg[b + 1] - cseg[b], x); };
  auto bound = [&](int b, int row) {
    const int g = seg_of(b, row);
    return types[g] == ISM_SEG_QUERY ? ends[g] : row + 1;
  };
  Tile q{}, k{};
  if (tid < nq) {
    const int b = upper_bound_i32(off, s.num_seqs + 1, tid) - 1;
    const int t = tid - off[b], L = cu[b + 1] - cu[b], r0 = t * bm;
    q.q_base = q.k_base = q.kv_base = cu[b];
    q.q_len = q.k_len = L;
    q.tile = t;
    k = q;
    q.a0 = r0 + bm <= L ? bound(b, r0) / bm : 0;
    q.a1 = (bound(b, min(L, r0 + bm) - 1) + bm - 1) / bm;
    // first row that sees key r0 (as in tiles_body)
    const int g = seg_of(b, r0), start = g > cseg[b] ? ends[g - 1] : 0;
    k.a0 = (types[g] == ISM_SEG_QUERY ? start : max(r0, start)) / bm;
    k.a1 = (L + bm - 1) / bm;
    cost[0][tid] = q.a1;
    cost[1][tid] = max(k.a1 - k.a0, 0);
  }
  __syncthreads();
  const bool odd = q.tile & 1;
  if (tid < nq) {
    // a pair costs what its second tile does (the first, when it has none)
    const bool second = tid + 1 < nq && !odd && (q.tile + 1) * bm < q.q_len;
    cost[odd ? 3 : 2][tid] = odd ? q.a1 : max(q.a1, second ? cost[0][tid + 1] : 0);
  }
  __syncthreads();
  int32_t pairs;
  const int32_t before = block_inclusive_scan<int32_t>(tid < nq ? cost[1][tid] : 0, &pairs);
  int rq = 0, rk = 0, rp = 0;
  int32_t heads = 0;
  if (pairs_first) block_inclusive_scan<int32_t>(tid < nq && !odd ? 1 : 0, &heads);
  if (tid < nq) {
    if (!odd && (pair_order || pairs_first)) rp = rank_of(cost[2], nq, cost[2][tid], tid);
    rq = !pairs_first ? rank_of(cost[0], nq, cost[0][tid], tid)
         : odd        ? heads + rank_of(cost[3], nq, cost[3][tid], tid)
                      : rp;
    if (k_order) rk = rank_of(cost[1], nq, cost[1][tid], tid);
  }
  if (tid < n_counters) counters[tid] = 0;
  if (tid < nq) {
    qtiles[tid] = q;
    q_order[rq] = tid;
    if (ktiles) ktiles[tid] = k;
    if (k_order) k_order[rk] = tid;
    if (pair_order && !odd) pair_order[rp] = tid;
    if (kpair_off) kpair_off[tid] = before - cost[1][tid];
  }
  const int warp = tid >> 5, lane = tid & 31;
  for (int seg = warp; seg < s.num_segs; seg += kSmallThreads / 32) {
    const int b = upper_bound_i32(cseg, s.num_seqs + 1, seg) - 1;
    const int start = seg > cseg[b] ? ends[seg - 1] : 0, end = ends[seg];
    const bool query = types[seg] == ISM_SEG_QUERY;
    for (int j = start + lane; j < end; j += 32) kv_end[cu[b] + j] = query ? end : j + 1;
  }
}

__device__ __forceinline__ int32_t chunk_kv_end(const AppendSegs& sg, int32_t j) {
  int32_t start = 0;
  for (int i = 0; i < sg.n; ++i) {
    int32_t e = sg.end[i];
    if (j < e && j >= start) return sg.type[i] == ISM_SEG_QUERY ? e : j + 1;
    start = e;
  }
  return j + 1;
}

// The append plan's share of one thread (grid-stride; see AppendPlan).
__device__ __forceinline__ void append_plan_part(const AppendPlan& p, int batch, const int32_t* cache_len) {
  if (!p.qtiles) return;
  const AppendSegs& sg = p.segs;
  const int32_t Ln = sg.l_new;
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
  if (t0 == 0) *p.counter = 0;
  for (int64_t i = t0; i < (int64_t)batch * Ln; i += stride)
    p.kv_end[i] = cache_len[i / Ln] + chunk_kv_end(sg, (int32_t)(i % Ln));
  const int nqt = (Ln + p.bm - 1) / p.bm, npt = (nqt + 1) / 2;
  for (int64_t g = t0; g < (int64_t)batch * nqt; g += stride) {
    const int b = (int)(g / nqt), t = (int)(g % nqt);
    const int32_t c = cache_len[b], r0 = t * p.bm, rl = min(Ln, r0 + p.bm) - 1;
    Tile w;
    w.q_base = b * Ln; w.k_base = (int32_t)(b * p.kbase_stride);
    w.q_len = Ln; w.k_len = c + Ln; w.tile = t;
    w.a0 = (r0 + p.bm <= Ln) ? (c + chunk_kv_end(sg, r0)) / p.bn : 0;
    w.a1 = (c + chunk_kv_end(sg, rl) + p.bn - 1) / p.bn;
    w.kv_base = b * Ln;
    p.qtiles[g] = w;
    p.q_order[g] = (int32_t)g;
    // q-tile pairs (2i, 2i + 1) of each sequence's chunk for the paired forward
    if (p.pair_order && !(t & 1)) p.pair_order[(int64_t)b * npt + t / 2] = (int32_t)g;
  }
}

// K_new/V_new rows into the caches at [c_snap[b], c_snap[b] + l_new) (rows of
// sequence b from b * cap, or through the page table).
// The attention kernels read keys in tiles of 128 from key 0, so the last
// tile of a sequence runs past its last key.  Masked keys get P = 0, but the
// P V contraction still multiplies those rows of V, and unwritten cache
// memory may hold NaN or Inf bit patterns (0 * NaN = NaN).  Value rows
// [c + l_new, round_up(c + l_new, 128)) are therefore set to zero by every
// cache write (clipped to the capacity of a contiguous cache; a paged tile
// lies within one page).  Keys need no such care: masked scores are replaced,
// not multiplied.
// The cache write also lays out the chunk's plan (one launch less: 3.4 us of
// the 60 us of a 40-token append over 3000 keys were a one-block plan kernel).
// It reads the cache lengths themselves (c_snap = cache_len): they stay as
// they are until the attention kernel after it advances them, and single-token
// steps find a copy in snap_out.
__device__ __forceinline__ void copy_snapshot(int batch, const int32_t* c_snap, int32_t* snap_out) {
  if (!snap_out) return;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < batch; b += (int64_t)gridDim.x * blockDim.x)
    snap_out[b] = c_snap[b];
}

__device__ __forceinline__ void zero_value_tail(int batch, int l_new, int vec_per_row, int64_t cap,
                                                const KvPages& pages, const int32_t* c_snap,
                                                uint4* v_cache) {
  const int64_t total = (int64_t)batch * 128 * vec_per_row;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = i / vec_per_row;
    const int col = (int)(i % vec_per_row);
    const int b = (int)(row / 128);
    const int64_t end = (int64_t)c_snap[b] + l_new;
    const int64_t p = end + row % 128;
    int64_t stop = (end + 127) / 128 * 128;
    if (!pages.table && stop > cap) stop = cap;
    if (p >= stop) continue;
    const int64_t dst = (pages.table ? paged_row(pages, b, p) : (int64_t)b * cap + p) * vec_per_row + col;
    v_cache[dst] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// The cache-write kernels let the attention kernel start as soon as what ran
// before them is complete: what it reads beside the new rows is then in place.
// A rotary decode step over 3000 keys 13.1 -> 10.6 us, 40 ragged caches 70 -> 67,
// e4m3 8 x 16384 keys 50.7 -> 48 (with the decode reading the old keys while
// the new row is written).  Inputs are not __restrict__: nothing may be loaded
// before the wait.
__global__ void cache_write_kernel(int batch, int l_new, int row_bytes, int64_t cap, KvPages pages,
                                   const int32_t* c_snap, const uint4* k_new,
                                   const uint4* v_new, uint4* k_cache, uint4* v_cache,
                                   const __grid_constant__ AppendPlan plan, int32_t* snap_out) {
  pdl_wait();
  append_plan_part(plan, batch, c_snap);
  const int vec_per_row = row_bytes / 16;
  copy_snapshot(batch, c_snap, snap_out);
  const int64_t total = (int64_t)batch * l_new * vec_per_row;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    int64_t row = i / vec_per_row;
    int col = (int)(i % vec_per_row);
    int b = (int)(row / l_new);
    int j = (int)(row % l_new);
    const int64_t p = (int64_t)c_snap[b] + j;
    int64_t dst = (pages.table ? paged_row(pages, b, p) : (int64_t)b * cap + p) * vec_per_row + col;
    k_cache[dst] = k_new[i];
    v_cache[dst] = v_new[i];
  }
  zero_value_tail(batch, l_new, vec_per_row, cap, pages, c_snap, v_cache);
}

// Rotary encoding fused with the cache write.  One thread takes eight
// consecutive coordinates k0..k0+7 of the first half of one head row and
// their partners k0+D/2.. (a query head, a key head, or a value head, which
// is copied as is).  Position of new token j of sequence b: c_snap[b] + j.
// The rotation is in fp32; the results are rounded once to the cache's type:
// bf16, or e4m3 after division by the tensor's dequantisation factor
// (q_descale for the rotated queries, k_descale / v_descale for the cache).
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&x)[8]) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 f = __bfloat1622float2(h[e]);
    x[2 * e] = f.x;
    x[2 * e + 1] = f.y;
  }
}
__device__ __forceinline__ uint32_t e4m3x2(float lo, float hi) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return r;
}
// Eight values stored in the element type of the output: bf16 (descale
// ignored) or e4m3 (x / descale, round to nearest, saturating).
template <bool kE4M3>
__device__ __forceinline__ void store8(void* base, int64_t elem, const float (&x)[8], float descale) {
  if constexpr (kE4M3) {
    uint2 u;
    u.x = e4m3x2(x[0] / descale, x[1] / descale) | (e4m3x2(x[2] / descale, x[3] / descale) << 16);
    u.y = e4m3x2(x[4] / descale, x[5] / descale) | (e4m3x2(x[6] / descale, x[7] / descale) << 16);
    *reinterpret_cast<uint2*>(static_cast<uint8_t*>(base) + elem) = u;
  } else {
    uint4 u;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&u);
#pragma unroll
    for (int e = 0; e < 4; ++e) h[e] = __floats2bfloat162_rn(x[2 * e], x[2 * e + 1]);
    *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(base) + elem) = u;
  }
}

template <bool kE4M3>
__global__ void rope_cache_write_kernel(int batch, int l_new, int hq, int hkv, int d, int64_t cap, KvPages pages,
                                        const int32_t* c_snap, const __nv_bfloat16* q_new,
                                        const __nv_bfloat16* k_new,
                                        const __nv_bfloat16* v_new, const float* cos_t,
                                        const float* sin_t, float q_descale, float k_descale,
                                        float v_descale, void* q_rot, void* k_cache, void* v_cache,
                                        const __grid_constant__ AppendPlan plan, int32_t* snap_out) {
  pdl_wait();
  append_plan_part(plan, batch, c_snap);
  copy_snapshot(batch, c_snap, snap_out);
  const int half = d / 2;
  const int units = half / 8;  // 8-coordinate units in one half of a head row
  const int per_row = (hq + 2 * hkv) * units;
  const int64_t total = (int64_t)batch * l_new * per_row;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = i / per_row;  // b * l_new + j
    const int r = (int)(i % per_row);
    const int head = r / units;
    const int k0 = (r % units) * 8;
    const int b = (int)(row / l_new);
    const int64_t p = (int64_t)c_snap[b] + row % l_new;
    const int64_t dst_row = pages.table ? paged_row(pages, b, p) : (int64_t)b * cap + p;
    const __nv_bfloat16* src;
    void* dst;
    int64_t off;  // element offset of the head row in dst
    float descale;
    if (head < hq) {
      src = q_new + (row * hq + head) * d;
      dst = q_rot;
      off = (row * hq + head) * d;
      descale = q_descale;
    } else if (head < hq + hkv) {
      src = k_new + (row * hkv + (head - hq)) * d;
      dst = k_cache;
      off = (dst_row * hkv + (head - hq)) * d;
      descale = k_descale;
    } else {
      src = v_new + (row * hkv + (head - hq - hkv)) * d;
      off = (dst_row * hkv + (head - hq - hkv)) * d;
      float lo[8], hi[8];
      load8(src + k0, lo);
      load8(src + half + k0, hi);
      store8<kE4M3>(v_cache, off + k0, lo, v_descale);
      store8<kE4M3>(v_cache, off + half + k0, hi, v_descale);
      continue;
    }
    float lo[8], hi[8], c[8], s[8];
    load8(src + k0, lo);
    load8(src + half + k0, hi);
    const float4* cp = reinterpret_cast<const float4*>(cos_t + p * half + k0);
    const float4* sp = reinterpret_cast<const float4*>(sin_t + p * half + k0);
    const float4 c0 = cp[0], c1 = cp[1], s0 = sp[0], s1 = sp[1];
    c[0] = c0.x; c[1] = c0.y; c[2] = c0.z; c[3] = c0.w; c[4] = c1.x; c[5] = c1.y; c[6] = c1.z; c[7] = c1.w;
    s[0] = s0.x; s[1] = s0.y; s[2] = s0.z; s[3] = s0.w; s[4] = s1.x; s[5] = s1.y; s[6] = s1.z; s[7] = s1.w;
    float ol[8], oh[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      ol[e] = lo[e] * c[e] - hi[e] * s[e];
      oh[e] = hi[e] * c[e] + lo[e] * s[e];
    }
    store8<kE4M3>(dst, off + k0, ol, descale);
    store8<kE4M3>(dst, off + half + k0, oh, descale);
  }
  zero_value_tail(batch, l_new, hkv * d * (kE4M3 ? 1 : 2) / 16, cap, pages, c_snap, reinterpret_cast<uint4*>(v_cache));
}

}  // namespace

cudaError_t launch_kv_end(const SegsDev& s, int32_t* kv_end, cudaStream_t st) {
  if (s.num_segs == 0) return cudaSuccess;
  int grid = s.num_segs < 4096 ? s.num_segs : 4096;
  kv_end_kernel<<<grid, 256, 0, st>>>(s, kv_end);
  return cudaGetLastError();
}

cudaError_t launch_tiles(const SegsDev& s, int bm, int bn, const int32_t* kv_end, int64_t nq, int64_t nk,
                         Tile* qtiles, Tile* ktiles, uint8_t* tile_class, int32_t* kt_full_end,
                         int32_t* kt_end, int32_t* qt_begin, cudaStream_t st) {
  int64_t n = nq > nk ? nq : nk;
  if (n == 0) return cudaSuccess;
  int grid = (int)((n + 255) / 256);
  if (grid > 608) grid = 608;
  size_t smem = (size_t)(s.num_seqs + 1) * (sizeof(int64_t) + 2 * sizeof(int32_t));
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(tiles_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  tiles_kernel<<<grid, 256, smem, st>>>(s, bm, bn, kv_end, nq, nk, qtiles, ktiles, tile_class, kt_full_end,
                                        kt_end, qt_begin);
  return cudaGetLastError();
}

cudaError_t launch_pass_meta(const SegsDev& s, int32_t* kv_end, int bm, int bn, int64_t nq, int64_t nk,
                             Tile* qtiles, Tile* ktiles, int max_cost, int32_t* q_order, int32_t* k_order,
                             int32_t* pair_order, int32_t* kpair_off, int32_t* counters, int n_counters,
                             cudaStream_t st, int32_t* kp_order, bool pairs_first, bool dependent) {
  if (bm == bn && nq <= kSmallTiles && s.num_seqs <= kSmallTiles && s.num_segs <= kSmallSegs && !kp_order)
    return launch(dependent, pass_meta_small_kernel, 1, kSmallThreads, 0, st, s, kv_end, bm, (int)nq, qtiles,
                            ktiles, q_order, k_order, pair_order, kpair_off, counters, n_counters, pairs_first);
  size_t a = (size_t)(s.num_seqs + 1) * (sizeof(int64_t) + 2 * sizeof(int32_t));
  size_t b = sizeof(int32_t) * (size_t)(max_cost + 1);
  size_t smem = a > b ? a : b;
  // opted in well below 48 KB: the kernel's static shared memory (the block
  // scans' warp totals) and the dynamic part together must fit what a launch
  // gets without opting in
  if (smem > 16 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(pass_meta_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  return launch(dependent, pass_meta_kernel, 1, 1024, smem, st, s, kv_end, bm, bn, nq, nk, qtiles, ktiles, max_cost,
                          q_order, k_order, pair_order, kpair_off, counters, n_counters, kp_order, pairs_first);
}

namespace {
// A cache-write kernel over `total` threads.
template <class... Params, class... Args>
cudaError_t launch_write(void (*kern)(Params...), int64_t total, cudaStream_t st, Args... args) {
  int64_t grid = (total + 255) / 256;
  const int64_t top = (int64_t)sm_count() * 16;
  if (grid > top) grid = top;
  return launch(true, kern, grid, 256, 0, st, args...);
}
}  // namespace

cudaError_t launch_cache_write(int dtype, int batch, int l_new, int hkv, int d, int64_t cap, const KvPages& pages,
                               const int32_t* c_snap, const void* k_new, const void* v_new,
                               void* k_cache, void* v_cache, const AppendPlan& plan, cudaStream_t st,
                               int32_t* snap_out) {
  int elem = dtype == ISM_BF16 ? 2 : dtype == ISM_E4M3 ? 1 : 4;
  int row_bytes = hkv * d * elem;
  int64_t total = (int64_t)batch * l_new * (row_bytes / 16);
  if (total == 0) return cudaSuccess;
  const int64_t tail = (int64_t)batch * 128 * (row_bytes / 16);  // value rows zeroed past the new end
  if (tail > total) total = tail;
  return launch_write(cache_write_kernel, total, st, batch, l_new, row_bytes, cap, pages, c_snap, (const uint4*)k_new,
                      (const uint4*)v_new, (uint4*)k_cache, (uint4*)v_cache, plan, snap_out);
}

cudaError_t launch_rope_cache_write(int dtype, int batch, int l_new, int hq, int hkv, int d, int64_t cap,
                                   const KvPages& pages, const int32_t* c_snap, const void* q_new,
                                   const void* k_new, const void* v_new, const float* cos_t, const float* sin_t,
                                   float q_descale, float k_descale, float v_descale, void* q_rot, void* k_cache,
                                   void* v_cache, const AppendPlan& plan, cudaStream_t st, int32_t* snap_out) {
  int64_t total = (int64_t)batch * l_new * (hq + 2 * hkv) * (d / 16);
  if (total == 0) return cudaSuccess;
  const bool e4m3 = dtype == ISM_E4M3;
  const int64_t tail = (int64_t)batch * 128 * (hkv * d * (e4m3 ? 1 : 2) / 16);  // value rows zeroed past the new end
  if (tail > total) total = tail;
  return launch_write(e4m3 ? rope_cache_write_kernel<true> : rope_cache_write_kernel<false>, total, st, batch, l_new, hq,
                      hkv, d, cap, pages, c_snap, (const __nv_bfloat16*)q_new, (const __nv_bfloat16*)k_new,
                      (const __nv_bfloat16*)v_new, cos_t, sin_t, q_descale, k_descale, v_descale, q_rot, k_cache,
                      v_cache, plan, snap_out);
}

}  // namespace ism
