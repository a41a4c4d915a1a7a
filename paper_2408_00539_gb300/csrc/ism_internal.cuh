// Internal declarations shared by the libism translation units.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "../../include/ism.h"

namespace ism {

// One tile of work for the attention kernels.  A "sequence" here is one
// query stream attending to one key stream: a packed dialogue for the
// one-pass forward/backward, or (new chunk of sequence b, its KV cache) for
// append-prefill.  Key positions (and kv_end values) are relative to k_base.
struct Tile {
  int32_t q_base;   // global Q/O/dO row of query row 0 of the sequence
  int32_t k_base;   // global K/V row of key 0 of the sequence
  int32_t q_len;    // query rows of the sequence
  int32_t k_len;    // keys of the sequence
  int32_t tile;     // q-tile index t (or k-tile index c) within the sequence
  int32_t a0;       // q-tile: number of leading FULL k-tiles; k-tile: first non-empty q-tile
  int32_t a1;       // q-tile: one past the last non-empty k-tile; k-tile: number of q-tiles
  int32_t kv_base;  // index of the sequence's query row 0 in the kv_end array
};
static_assert(sizeof(Tile) == 32, "Tile layout");

// A load from L2, where another SM's finished writes are.
__device__ __forceinline__ int32_t ld_gpu(const int32_t* p) {
  int32_t v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Paged K/V cache (append-prefill and decode): key p of sequence b sits in
// row table[b * max_pages + p / page_size] * page_size + p % page_size of the
// pools.  With table == nullptr the cache is contiguous: the rows of sequence
// b start at b * cap (append kernels) or at Tile::k_base (attention kernels).
struct KvPages {
  const int32_t* table;
  int32_t page_size, max_pages;
};
__device__ __forceinline__ const int32_t* page_entry(const KvPages& pg, int b, int64_t p) {
  return pg.table + (int64_t)b * pg.max_pages + p / pg.page_size;
}
__device__ __forceinline__ int64_t page_row(const KvPages& pg, int32_t entry, int64_t p) {
  return (int64_t)entry * pg.page_size + p % pg.page_size;
}
// (A plain load of the table: dependent kernels read it behind their wait.)
__device__ __forceinline__ int64_t paged_row(const KvPages& pg, int b, int64_t p) {
  return page_row(pg, *page_entry(pg, b, p), p);
}

// Device view of the segment arrays (device pointers only).
struct SegsDev {
  int32_t num_seqs;
  int32_t num_segs;
  const int32_t* cu_seqlens;
  const int32_t* cu_segs;
  const int32_t* seg_end;
  const uint8_t* seg_type;
};

// Chunk segments of an append, passed to kernels by value.
constexpr int kMaxAppendSegs = 256;
struct AppendSegs {
  int32_t n;
  int32_t l_new;
  int32_t end[kMaxAppendSegs];
  uint8_t type[kMaxAppendSegs];
};

// Meta arrays carved out of a workspace.
struct Meta {
  int32_t* kv_end;      // [kv rows]
  Tile* qtiles;         // [nq]
  Tile* ktiles;         // [nk] (may be null)
  int32_t* q_order;     // [nq] q-tile indices, most expensive first
  int32_t* k_order;     // [nk]
  int64_t nq, nk;
};

// Status word bits recorded by device code.
enum : uint32_t { kStatusTimeout = 1u, kStatusSmemAlign = 2u };

// ---------------------------------------------------------------- dependent launches
// A kernel launched as a programmatic dependent overlaps its launch and set-up
// with the end of the one before it on the stream.  Every such kernel calls
// pdl_wait (all of its threads that touch global memory) before anything that
// depends on earlier work or that earlier work may still use: it waits for the
// kernel before this one to complete.  Only then does it let the next one start
// its set-up, so that a kernel that runs at all has everything before its direct
// predecessor in place.  What it reads is not __restrict__ and not read through
// __ldg: such loads count as constant, and the compiler may move them before the
// wait.  (rope_row may: its addresses come from descriptors that are read behind
// it.)
// A kernel that allocates tensor memory lets the next one start only after its
// allocation (pdl_sync at the top, pdl_trigger behind it): the next kernel may
// allocate before it waits for this one, and would otherwise hold columns that
// a block of this one still needs, each waiting for the other.
// Appends and decode steps are launched so, and the passes of a small batch
// (dependent_pass): one fp32 dialogue of 256 tokens 69.8 -> 55.7 us a step (with the
// small metadata pass), 4000 ragged tokens of 12 heads 162 -> 148.  On large ones
// the blocks that wait on the SMs cost more than the launches: 24 dialogues of
// 32 heads (16001 tokens) 652 -> 686.
__device__ __forceinline__ void pdl_sync() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() {
  pdl_sync();
  pdl_trigger();
}
template <class... Params, class... Args>
cudaError_t launch(bool dependent, void (*kern)(Params...), int64_t grid, int threads, size_t smem, cudaStream_t st,
                   const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, Params(args)...);
}

// ---------------------------------------------------------------- launches
// Each returns cudaSuccess or the launch error.

// Tile-map kernels (ism_meta.cu).
cudaError_t launch_kv_end(const SegsDev& s, int32_t* kv_end, cudaStream_t st);
// At most kMaxSeqs sequences (per-sequence offsets are kept in shared memory).
constexpr int kMaxSeqs = 8192;
cudaError_t launch_tiles(const SegsDev& s, int bm, int bn, const int32_t* kv_end, int64_t nq, int64_t nk,
                         Tile* qtiles, Tile* ktiles, uint8_t* tile_class, int32_t* kt_full_end,
                         int32_t* kt_end, int32_t* qt_begin, cudaStream_t st);
// kv_end, tiles, work lists (and pair offsets when kpair_off is set, the
// k-tile pair list when kp_order is set) in one launch.  pairs_first: q_order
// starts with the even-indexed q-tiles (pair heads, in the pair list's order).
cudaError_t launch_pass_meta(const SegsDev& s, int32_t* kv_end, int bm, int bn, int64_t nq, int64_t nk,
                             Tile* qtiles, Tile* ktiles, int max_cost, int32_t* q_order, int32_t* k_order,
                             int32_t* pair_order, int32_t* kpair_off, int32_t* counters, int n_counters,
                             cudaStream_t st, int32_t* kp_order = nullptr, bool pairs_first = false,
                             bool dependent = false);
// What the forward over an appended chunk reads, written by the cache-write
// kernels along with the cache: the absolute key bound of every new row (all
// cached keys plus Eq. fj within the chunk), one descriptor per (sequence,
// chunk tile) in order, and the pair heads.  kbase_stride: k_base of sequence
// b's tiles is b times it (the cache capacity, or 1 for a paged cache).
// qtiles == nullptr (single-token steps): nothing of it.
struct AppendPlan {
  AppendSegs segs;
  int64_t kbase_stride;
  int32_t bm, bn;
  int32_t* kv_end;
  Tile* qtiles;
  int32_t* q_order;
  int32_t* pair_order;
  int32_t* counter;  // set to zero (the forward's work counter)
};
// cache_len: lengths before the append (read only; the attention kernels
// advance them).  snap_out (nullable): receives a copy of them.
cudaError_t launch_cache_write(int dtype, int batch, int l_new, int hkv, int d, int64_t cap, const KvPages& pages,
                               const int32_t* cache_len, const void* k_new, const void* v_new,
                               void* k_cache, void* v_cache, const AppendPlan& plan, cudaStream_t st,
                               int32_t* snap_out);
// Cache write with the rotary encoding of the new queries and keys (bf16
// inputs, head_dim a multiple of 16): rotated keys and plain values into the
// cache, rotated queries into q_rot [batch * l_new, hq, d], all in the cache's
// type: bf16, or e4m3 (dtype ISM_E4M3) after division by the descales.
cudaError_t launch_rope_cache_write(int dtype, int batch, int l_new, int hq, int hkv, int d, int64_t cap,
                                   const KvPages& pages, const int32_t* cache_len, const void* q_new,
                                   const void* k_new, const void* v_new, const float* cos_t, const float* sin_t,
                                   float q_descale, float k_descale, float v_descale, void* q_rot, void* k_cache,
                                   void* v_cache, const AppendPlan& plan, cudaStream_t st, int32_t* snap_out);

// Rotary encoding of the one-pass path (ism_rope.cu): rotates every query and
// key head row of a packed batch by its position inside its sequence (pairs
// k, k + d/2; tables [rows, d/2] fp32), from q_src / k_src into q_dst / k_dst
// (in place allowed).  sin_sign = -1 applies the transposed rotation.  bf16
// or fp32 rows, d a multiple of 16.
cudaError_t launch_rope_rows(const int32_t* cu_seqlens, int num_seqs, int64_t T, int hq, int hkv, int d, int dtype,
                             const void* q_src, const void* k_src, void* q_dst, void* k_dst, const float* cos_t,
                             const float* sin_t, float sin_sign, cudaStream_t st, bool dependent);

// Multiprocessor count of the current device (looked up once per device).
int sm_count();

// Arguments of the attention kernels: the CUDA-core ones (ism_simt.cu; fp32 or
// bf16 storage, fp32 math) and the tensor-core ones.
struct AttnArgs {
  const void* q; const void* k; const void* v; const void* o; const void* dout;
  void* out; float* lse; const float* lse_in;
  void* dq; void* dk; void* dv;
  float* delta;
  int32_t hq, hkv, d, dtype;
  int64_t q_rows;      // rows of Q (LSE row stride)
  float scale;
  const int32_t* kv_end;
  const Tile* qtiles; const int32_t* q_order; int64_t nq;
  // 0: q_order is in cost order.  Else a plan's whose first order_pairs entries
  // are the even-indexed q-tiles and whose others are the odd ones (q_tile_at).
  int64_t order_pairs;
  const Tile* ktiles; const int32_t* k_order; int64_t nk;
  uint32_t* status;
  // Stored-dS backward: when ds is set, dK/dV also writes each bf16 dS tile
  // (128 queries x 128 keys, 8-query-interleaved, 32 KiB) of (k-tile gk,
  // q-tile t, head h) to slot (kpair_off[gk] + t - qt_begin(gk)) * hq + h,
  // and dQ is a GEMM over them.
  void* ds;
  const int32_t* kpair_off;
  int64_t ds_slots;
  // Query-tile pairs for the paired forward when the query heads of a KV head
  // are odd in number: pair_order lists the even-indexed q-tiles (each with
  // the next q-tile of its sequence, when there is one) in cost order.
  const int32_t* pair_order;
  int64_t npairs;
  bool bucketed;  // their work list in buckets of neighbouring tiles, head by head (fwd_bucketed)
  // Work counter, at zero: of the persistent dK/dV kernel, or of the paired
  // forward (fwd_dynamic).
  int32_t* work_counter;
  // dK/dV on CTA pairs: kp_order lists the even-indexed k-tiles (each with the
  // next k-tile of its sequence, when there is one) in cost order; nkp of them.
  const int32_t* kp_order;
  int64_t nkp;
  // Paged K/V (forward over an appended chunk only): Tile::k_base holds the
  // sequence index and key p's row is paged_row(pages, k_base, p).
  KvPages pages;
  // e4m3 forward: per-tensor dequantisation factors (scores scaled by
  // q_descale * k_descale, the output by v_descale).
  float qk_descale, v_descale;
  // Key-range split of the paired forward: launch items [0, split_whole) run
  // whole; each later item runs as split_parts units over equal shares of its
  // key tiles, writing unnormalised O and (max, sum) to part_o / part_ml,
  // merged by a second kernel.  Off when split_items == 0.
  int64_t split_whole, split_items;
  int32_t split_parts, part_rows;  // part_rows: the most rows of a query tile
  float* part_o;    // [split_items][split_parts][2][part_rows][d] fp32
  float* part_ml;   // [split_items][split_parts][2][part_rows][2] fp32
  // Append-prefill: the cache lengths [adv_batch], advanced by adv_len by the
  // forward kernel (the kernels before it read them; it does not).
  int32_t* adv_cache_len;
  int32_t adv_batch, adv_len;
  // Rotary encoding (tensor-core backward only): when rope_cos is set, the dQ
  // and dK epilogues store the gradients of the unrotated queries and keys,
  // applying the transposed rotation of the row's position in its sequence
  // (tables [rows, d / 2] fp32, the angle of pair k of position p at p * d / 2 + k).
  const float* rope_cos;
  const float* rope_sin;
  bool dependent;  // launch as programmatic dependents (dependent_pass)
  // Bit 0: before an MMA that overwrites tensor memory an earlier MMA reads
  // as its A operand, wait for that earlier MMA to complete.  Clear: rely on
  // MMAs issued by one thread executing in issue order.
  uint32_t flags;
};
enum : uint32_t { kFlagDrainTmemReuse = 1u };
// Whether the kernels of a pass are launched as programmatic dependents: a batch
// of few query tiles.
inline bool dependent_pass(int64_t q_tiles, int heads) { return q_tiles * heads <= 8 * (int64_t)sm_count(); }
// Whether the paired forward takes its units (whole items) from a work counter
// in cost order, or walks them statically.  The counter evens out CTAs that get
// few or unequal units; the static walk starts a unit a little sooner.  Query-
// tile pairs always gain (units of one or two long tiles of many sizes): 4 x 4096
// multi-head 414 -> 387 us, 6 ragged dialogues of 32 heads 692 -> 575, head_dim
// 64 with 16 heads over 6001 tokens 98 -> 67.  Head pairs gain below eight units
// a CTA (16 / 4 heads over 5000 ragged tokens, 2 units a CTA: 46 -> 39) and lose
// on many even ones (2 x 8192, 13 a CTA: 654 -> 662; one dialogue of 32768 4881
// -> 4951).  Planned forwards have no counter and always walk statically.
inline bool fwd_dynamic(int64_t items, bool tile_pairs) { return tile_pairs || items < 8 * (int64_t)sm_count(); }
// Whether that list keeps its buckets (bucket_item) instead of the plain cost
// order: with one query head per KV head, 32 KB tiles and many units, sharing
// tiles in L2 saves about as much (power above all, in a loop of steps) as the
// order's balance gives: 4 x 4096 of 32 heads 1767 us a step against 1786 (the
// forward alone 396 and 387), six ragged dialogues 2684 and 2699, little more than
// two runs differ by.  Half-size
// tiles and few units: e4m3 4 x 4096 333 and 318, head_dim 64 over 6001 tokens 318
// and 302.  The static walk of tile pairs keeps its buckets wherever the heads do
// not share K / V.
inline bool fwd_bucketed(const AttnArgs& a, int64_t items) {
  return a.hq == a.hkv && a.d == 128 && a.dtype == ISM_BF16 && items >= 8 * (int64_t)sm_count();
}
// The q-tile at position `pos` of the cost order.  Where the even and the odd
// tiles stand apart, each half most expensive first, they alternate: the i-th pair
// head goes with a tile of about its cost.
__device__ __forceinline__ int32_t q_tile_at(const AttnArgs& a, int64_t pos) {
  if (a.order_pairs) {
    const int64_t odd = a.nq - a.order_pairs;
    pos = pos >= 2 * odd ? pos - odd : pos & 1 ? a.order_pairs + pos / 2 : pos / 2;
  }
  return a.q_order[pos];
}
// Called by every thread of every block of a forward kernel.
__device__ __forceinline__ void advance_cache_len(const AttnArgs& a) {
  if (a.adv_cache_len && blockIdx.x == 0)
    for (int b = threadIdx.x; b < a.adv_batch; b += blockDim.x) a.adv_cache_len[b] += a.adv_len;
}
cudaError_t launch_simt_fwd(const AttnArgs& a, cudaStream_t st);
cudaError_t launch_simt_bwd(const AttnArgs& a, cudaStream_t st);

// Split-KV decode for single-token appends (ism_decode.cu).
struct DecodeArgs {
  const void* q;         // [B, Hq, D]
  const void* k_cache;   // [B, cap, Hkv, D], or the page pools [pages * page_size, Hkv, D]
  const void* v_cache;
  KvPages pages;         // table == nullptr: contiguous caches
  void* out;             // [B, Hq, D]
  float* lse;            // [Hq, B] or null
  const int32_t* c_snap; // cache length before the append, per sequence
  int32_t batch, hq, hkv, d, dtype;
  int32_t group;         // query heads per KV head (the kernels pad it to a power of two)
  float qk_descale, v_descale;  // e4m3: dequantisation of the scores and of the output
  int64_t cap;
  int64_t kv_rows;       // rows of the K / V tensors: batch * cap, or pages * page_size
  float scale;
  int32_t splits, chunk;
  float* part_o;         // [B, Hq, splits, D]
  float* part_ml;        // [B, Hq, splits, 2]
  int32_t tma;           // stream the cache with TMA (head_dim 128, sm_103)
  int32_t tc;            // tensor-core kernel (bf16 or e4m3, head_dim 128, group <= 16)
  // tpc == 0: equal chunks of a multiple of 128 keys (splits, chunk).  Else
  // (bf16, by decode_row) the 128-key tiles of all (sequence, head group) caches in
  // one row of `shares` shares of tpc tiles, an item at most kDecTcTiles; splits =
  // room for partials per (sequence, KV head).  The row is walked by the device's
  // lengths, and the last share has no end: where they have outgrown the host's
  // copy (a captured step replayed), it takes what the copy did not count.  align: each cache's
  // tiles are padded to a multiple of it in the row (1: not).  start [B]: written
  // with the first tile of each sequence in the row.
  // lanes: KV heads side by side; CTA i takes share i / lanes of head group g's
  // (head g * lanes + i % lanes) part of the row, so lanes neighbours read along
  // the same cache rows.
  int32_t tpc, shares, align, lanes;
  int32_t q_written;     // the queries come from the cache write (rotated)
  int32_t* start;
  uint32_t* status;      // device status word (bounded waits)
  int32_t* cache_len;    // [B] equal to c_snap until the combine kernel advances it by one
};
// Keys one work item of the tensor-core decode covers at most (its scores of
// 24 tiles of 128 keys stay in tensor memory).
constexpr int kDecTcTiles = 24;
constexpr int kDecTcMaxKeys = kDecTcTiles * 128;
__host__ __device__ __forceinline__ int32_t dec_tiles(int32_t cached) { return (cached + 1 + 127) / 128; }
__host__ __device__ __forceinline__ int32_t dec_alloc_tiles(const DecodeArgs& a, int32_t tiles) {
  return a.align == 1 ? tiles : (tiles + a.align - 1) / a.align * a.align;
}
// The share that a tile of the row belongs to.
__host__ __device__ __forceinline__ int32_t dec_share(const DecodeArgs& a, int32_t tile) {
  const int32_t c = tile / a.tpc;
  return c < a.shares ? c : a.shares - 1;
}
// Slot of the j-th item that share c has of the (sequence, KV head) whose tiles start at s.
__host__ __device__ __forceinline__ int32_t dec_slot(const DecodeArgs& a, int32_t s, int32_t c, int32_t j) {
  return (c - dec_share(a, s)) * ((a.tpc + kDecTcTiles - 1) / kDecTcTiles) + j;
}
cudaError_t launch_decode(const DecodeArgs& a, cudaStream_t st);

// Tensor-core kernels (ism_fwd_tc.cu / ism_bwd_tc.cu), bf16 only.
bool tc_available();
bool tc_bwd_available();
cudaError_t launch_tc_mma_tile(const void* a, const void* b, float* c, int mode, uint32_t* status, cudaStream_t st);
namespace tc {
cudaError_t launch_mma_tile_e4m3(const void* a, const void* b, float* c, int mode, uint32_t* status, cudaStream_t st);
}
cudaError_t launch_tc_fwd(const AttnArgs& a, int64_t k_rows, cudaStream_t st);
cudaError_t launch_tc_bwd(const AttnArgs& a, int64_t k_rows, cudaStream_t st);

cudaError_t launch_timeout_probe(uint32_t spin_limit, uint32_t* status, cudaStream_t st);

// Debug and tuning switches from the environment (ISM_*), read once when the
// library is loaded and again by ism_debug_reload_env(), so that no call reads
// the environment.
struct Knobs {
  bool force_cuda_cores;   // ISM_FORCE_CUDA_CORES=1: CUDA-core kernels for bf16 too
  bool drain_tmem_reuse;   // ISM_DRAIN_TMEM_REUSE=1: wait for A-operand readers before overwriting TMEM
  bool fwd_one_head;       // ISM_FWD_ONE_HEAD=1: one-head forward kernel
  bool bwd_recompute_dq;   // ISM_BWD_RECOMPUTE_DQ=1: recompute backward even with a stored-dS workspace
  bool decode_no_tma;      // ISM_DECODE_NO_TMA=1: register-load CUDA-core decode
  bool decode_no_tc;       // ISM_DECODE_NO_TC=1: CUDA-core decode kernels
  int64_t prefill_split;   // ISM_PREFILL_SPLIT=n: n key-range split items in a prefill (-1: chosen by the library)
  int32_t dkdv_grid;       // ISM_DKDV_GRID=n: CTAs of the persistent dK/dV kernel (0: one per SM)
  int32_t dq_grid;         // ISM_DQ_GRID=n: CTAs of the persistent dQ kernel (0: one per SM)
  bool dkdv_pair;          // ISM_DKDV_PAIR=1: dK/dV on CTA pairs (cta_group::2)
};
const Knobs& knobs();
void reload_knobs();

// Measurement hooks (ism_api.cu): events recorded around launches of one
// kernel kind on the calling host thread, and a count of every launch.
void timer_begin(int kernel_id, cudaStream_t st);
void timer_end(int kernel_id, cudaStream_t st);
void count_launch(int n = 1);
// Sets the message returned by ism_last_error() on this host thread.
void set_error(const char* msg);

}  // namespace ism
