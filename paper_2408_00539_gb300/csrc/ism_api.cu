// Host side of the C ABI: argument validation on the host mirrors, workspace
// layout, kernel dispatch and the device status word.
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <atomic>
#include <mutex>
#include <string>
#include <vector>

#include "ism_internal.cuh"

namespace ism {
namespace {

thread_local std::string g_last_error;

ism_status_t fail(ism_status_t st, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_last_error = buf;
  return st;
}

ism_status_t cuda_fail(cudaError_t e, const char* where) {
  return fail(ISM_ERR_CUDA, "%s: %s", where, cudaGetErrorString(e));
}

#define ISM_TRY_CUDA(expr, where)                 \
  do {                                            \
    cudaError_t e_ = (expr);                      \
    if (e_ != cudaSuccess) return cuda_fail(e_, where); \
  } while (0)

// One status word per device; the library's only persistent device state.
__device__ uint32_t g_status_word;

std::mutex g_status_mu;
std::vector<uint32_t*> g_status_ptr;

ism_status_t status_ptr(uint32_t** out) {
  int dev = 0;
  ISM_TRY_CUDA(cudaGetDevice(&dev), "cudaGetDevice");
  std::lock_guard<std::mutex> lk(g_status_mu);
  if ((int)g_status_ptr.size() <= dev) g_status_ptr.resize(dev + 1, nullptr);
  if (!g_status_ptr[dev]) {
    void* p = nullptr;
    ISM_TRY_CUDA(cudaGetSymbolAddress(&p, g_status_word), "cudaGetSymbolAddress(status)");
    g_status_ptr[dev] = static_cast<uint32_t*>(p);
  }
  *out = g_status_ptr[dev];
  return ISM_OK;
}

// ---------------------------------------------------------------- measurement

constexpr int kTimerSlots = 8;
thread_local cudaEvent_t g_timer_start[kTimerSlots];
thread_local cudaEvent_t g_timer_stop[kTimerSlots];
std::atomic<uint64_t> g_launches{0};

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

constexpr int kTile = 128;       // q/k tile rows of the attention kernels and their work lists
constexpr int kMaxSplits = 64;   // split-KV chunks per (sequence, KV head) for decode

struct SegInfo {
  int64_t total_tokens = 0;
  int64_t max_len = 0;
};

ism_status_t check_segments(const ism_segments_t* s, SegInfo* info) {
  if (!s) return fail(ISM_ERR_INVALID_ARG, "segments is NULL");
  if (s->num_seqs < 0 || s->num_segs < 0) return fail(ISM_ERR_INVALID_ARG, "negative counts");
  if (s->num_seqs > kMaxSeqs) return fail(ISM_ERR_UNSUPPORTED, "num_seqs %d > %d", s->num_seqs, kMaxSeqs);
  if (!s->cu_seqlens_host || !s->cu_segs_host || !s->cu_seqlens || !s->cu_segs)
    return fail(ISM_ERR_INVALID_ARG, "cu_seqlens / cu_segs (device and host) must be non-NULL");
  if (s->num_segs > 0 && (!s->seg_end || !s->seg_end_host || !s->seg_type || !s->seg_type_host))
    return fail(ISM_ERR_INVALID_ARG, "seg_end / seg_type (device and host) must be non-NULL");
  const int32_t* cs = s->cu_seqlens_host;
  const int32_t* cg = s->cu_segs_host;
  if (cs[0] != 0 || cg[0] != 0) return fail(ISM_ERR_INVALID_ARG, "cu_seqlens[0] and cu_segs[0] must be 0");
  if (cg[s->num_seqs] != s->num_segs)
    return fail(ISM_ERR_INVALID_ARG, "cu_segs[num_seqs]=%d != num_segs=%d", cg[s->num_seqs], s->num_segs);
  int64_t max_len = 0;
  for (int b = 0; b < s->num_seqs; ++b) {
    int64_t L = (int64_t)cs[b + 1] - cs[b];
    if (L < 0) return fail(ISM_ERR_INVALID_ARG, "cu_seqlens decreases at sequence %d", b);
    if (cg[b + 1] < cg[b]) return fail(ISM_ERR_INVALID_ARG, "cu_segs decreases at sequence %d", b);
    int32_t prev = 0;
    for (int i = cg[b]; i < cg[b + 1]; ++i) {
      int32_t e = s->seg_end_host[i];
      if (e < prev) return fail(ISM_ERR_INVALID_ARG, "seq %d: seg_end not non-decreasing at segment %d", b, i);
      if (s->seg_type_host[i] > 1) return fail(ISM_ERR_INVALID_ARG, "segment %d: type %d is not QUERY/ANSWER", i,
                                               (int)s->seg_type_host[i]);
      prev = e;
    }
    if (prev != L)
      return fail(ISM_ERR_INVALID_ARG, "seq %d: segments end at %d but the sequence has %lld tokens", b, prev,
                  (long long)L);
    if (L > max_len) max_len = L;
  }
  info->total_tokens = cs[s->num_seqs];
  info->max_len = max_len;
  return ISM_OK;
}

ism_status_t check_shape(const ism_attn_shape_t* sh, bool allow_e4m3 = false) {
  if (!sh) return fail(ISM_ERR_INVALID_ARG, "shape is NULL");
  if (sh->num_heads_q <= 0 || sh->num_heads_kv <= 0) return fail(ISM_ERR_INVALID_ARG, "head counts must be > 0");
  if (sh->num_heads_q % sh->num_heads_kv)
    return fail(ISM_ERR_INVALID_ARG, "num_heads_q (%d) is not a multiple of num_heads_kv (%d)", sh->num_heads_q,
                sh->num_heads_kv);
  if (sh->head_dim != 64 && sh->head_dim != 128)
    return fail(ISM_ERR_UNSUPPORTED, "head_dim %d (supported: 64, 128)", sh->head_dim);
  if (sh->dtype == ISM_E4M3) {
    if (!allow_e4m3) return fail(ISM_ERR_UNSUPPORTED, "e4m3 inputs only in ism_attn_fwd_e4m3");
    if (sh->head_dim != 128) return fail(ISM_ERR_UNSUPPORTED, "e4m3 needs head_dim 128");
  } else if (sh->dtype != ISM_BF16 && sh->dtype != ISM_FP32) {
    return fail(ISM_ERR_UNSUPPORTED, "dtype %d", sh->dtype);
  }
  if (!(sh->softmax_scale > 0.f) || sh->softmax_scale != sh->softmax_scale)
    return fail(ISM_ERR_INVALID_ARG, "softmax_scale must be a positive number");
  return ISM_OK;
}

SegsDev dev_view(const ism_segments_t* s) {
  SegsDev d;
  d.num_seqs = s->num_seqs;
  d.num_segs = s->num_segs;
  d.cu_seqlens = s->cu_seqlens;
  d.cu_segs = s->cu_segs;
  d.seg_end = s->seg_end;
  d.seg_type = s->seg_type;
  return d;
}

// Bump allocator over a caller-provided workspace (256-byte aligned pieces).
struct Carve {
  uintptr_t base;
  size_t off = 0;
  explicit Carve(void* p) : base(reinterpret_cast<uintptr_t>(p)) {}
  template <typename T>
  T* take(int64_t n) {
    off = (off + 255) & ~size_t(255);
    T* p = reinterpret_cast<T*>(base + off);
    off += sizeof(T) * (size_t)(n > 0 ? n : 0);
    return p;
  }
};

struct Counts {
  int64_t nq = 0, nk = 0, ntiles = 0;
  int64_t npairs = 0;  // q-tile pairs (neighbouring q-tiles of a sequence, the last one may be alone)
  int max_cost = 0;
};

Counts count_tiles(const ism_segments_t* s, int bm, int bn) {
  Counts c;
  for (int b = 0; b < s->num_seqs; ++b) {
    int64_t L = (int64_t)s->cu_seqlens_host[b + 1] - s->cu_seqlens_host[b];
    int64_t nq = (L + bm - 1) / bm, nk = (L + bn - 1) / bn;
    c.nq += nq;
    c.nk += nk;
    c.npairs += (nq + 1) / 2;
    c.ntiles += nq * nk;
    int mc = (int)(nq > nk ? nq : nk);
    if (mc > c.max_cost) c.max_cost = mc;
  }
  return c;
}

// Visible (k-tile, q-tile) pairs over all sequences at kTile x kTile tiles:
// k-tile c pairs with every q-tile from the one holding the first row whose
// kv_end exceeds c*kTile to the last.  Under Eq. fj that row is the start of
// the first segment ending after c*kTile when it is a query segment, else
// max(segment start, c*kTile).  Host walk over segments and k-tiles.
int64_t count_pairs(const ism_segments_t* s) {
  int64_t pairs = 0;
  for (int b = 0; b < s->num_seqs; ++b) {
    const int32_t L = s->cu_seqlens_host[b + 1] - s->cu_seqlens_host[b];
    const int32_t nt = (L + kTile - 1) / kTile;
    int32_t seg = s->cu_segs_host[b], start = 0;
    const int32_t seg1 = s->cu_segs_host[b + 1];
    for (int32_t c = 0; c < nt; ++c) {
      const int32_t x = c * kTile;
      while (seg < seg1 && s->seg_end_host[seg] <= x) start = s->seg_end_host[seg++];
      if (seg == seg1) break;
      const int32_t j = s->seg_type_host[seg] == ISM_SEG_QUERY ? start : (x > start ? x : start);
      pairs += nt - j / kTile;
    }
  }
  return pairs;
}

// Workspace of the one-pass forward/backward.  ds_slots > 0 adds the
// stored-dS backward's pair offsets and bf16 dS^T tiles (32 KiB a slot).
struct PassLayout {
  int32_t* kv_end;
  Tile *qtiles, *ktiles;
  int32_t *q_order, *k_order;
  float* delta;
  int32_t* kpair_off;
  void* ds;
  int32_t* pair_order;
  int32_t* kp_order;  // k-tile pairs in cost order (backward only)
  int32_t* counters;  // work counters: of dK/dV (backward, plans), of the forward
  size_t bytes;
};
constexpr int kPassCounters = 2;
constexpr int kBwdCounter = 0, kFwdCounter = 1;

PassLayout pass_layout(void* ws, const ism_segments_t* s, const Counts& c, int64_t T, int hq, bool bwd,
                       int64_t ds_slots = 0, bool tile_pairs = false) {
  Carve cv(ws);
  PassLayout L;
  L.kv_end = cv.take<int32_t>(T);
  L.qtiles = cv.take<Tile>(c.nq);
  L.q_order = cv.take<int32_t>(c.nq);
  L.ktiles = bwd ? cv.take<Tile>(c.nk) : nullptr;
  L.k_order = bwd ? cv.take<int32_t>(c.nk) : nullptr;
  L.delta = bwd ? cv.take<float>((int64_t)hq * T) : nullptr;
  L.kpair_off = ds_slots > 0 ? cv.take<int32_t>(c.nk) : nullptr;
  L.ds = ds_slots > 0 ? static_cast<void*>(cv.take<uint16_t>(ds_slots * kTile * kTile)) : nullptr;
  L.pair_order = tile_pairs ? cv.take<int32_t>(c.npairs) : nullptr;
  L.kp_order = bwd ? cv.take<int32_t>(c.npairs) : nullptr;  // k-tile pairs number as q-tile pairs here
  if (bwd) L.counters = cv.take<int32_t>(kPassCounters);
  L.bytes = ((cv.off + 255) & ~size_t(255)) + 256;
  // the forward's lie in the 256 bytes that every layout ends with
  if (!bwd) L.counters = reinterpret_cast<int32_t*>(reinterpret_cast<uintptr_t>(ws) + L.bytes - 256);
  return L;
}

// Device layout of a plan (ism_attn_plan_build): the metadata of both
// passes for one batch of segments and head counts, without the backward's
// Delta and dS tiles, which stay in the backward's workspace.
bool fwd_tile_pairs(const ism_attn_shape_t* sh);
PassLayout plan_layout(void* plan, const Counts& c, int64_t T, bool tile_pairs) {
  Carve cv(plan);
  PassLayout L{};
  L.kv_end = cv.take<int32_t>(T);
  L.qtiles = cv.take<Tile>(c.nq);
  L.q_order = cv.take<int32_t>(c.nq);
  L.ktiles = cv.take<Tile>(c.nk);
  L.k_order = cv.take<int32_t>(c.nk);
  L.kpair_off = cv.take<int32_t>(c.nk);
  L.pair_order = tile_pairs ? cv.take<int32_t>(c.npairs) : nullptr;
  L.counters = cv.take<int32_t>(kPassCounters);
  L.bytes = ((cv.off + 255) & ~size_t(255)) + 256;
  return L;
}

// What a plan was built for: FNV-1a over the segments' host arrays, the head
// counts and whether the forward pairs query tiles (the work lists differ).
uint64_t plan_fingerprint(const ism_segments_t* s, const ism_attn_shape_t* sh, bool tile_pairs) {
  uint64_t h = 1469598103934665603ull;
  auto mix = [&](const void* p, size_t n) {
    const unsigned char* b = static_cast<const unsigned char*>(p);
    for (size_t i = 0; i < n; ++i) h = (h ^ b[i]) * 1099511628211ull;
  };
  const int32_t head[4] = {s->num_seqs, s->num_segs, sh->num_heads_q, sh->num_heads_kv};
  mix(head, sizeof(head));
  const uint8_t tp = tile_pairs ? 1 : 0;
  mix(&tp, 1);
  mix(s->cu_seqlens_host, sizeof(int32_t) * (size_t)(s->num_seqs + 1));
  mix(s->cu_segs_host, sizeof(int32_t) * (size_t)(s->num_seqs + 1));
  if (s->num_segs > 0) {
    mix(s->seg_end_host, sizeof(int32_t) * (size_t)s->num_segs);
    mix(s->seg_type_host, (size_t)s->num_segs);
  }
  return h;
}

bool force_cuda_cores() { return knobs().force_cuda_cores; }

uint32_t tc_flags() { return knobs().drain_tmem_reuse ? kFlagDrainTmemReuse : 0u; }

bool use_tc(const ism_attn_shape_t* sh) {
  return sh->dtype == ISM_BF16 && tc_available() && !force_cuda_cores();
}
bool use_tc_bwd(const ism_attn_shape_t* sh) { return use_tc(sh) && tc_bwd_available(); }

// The tensor-core forward pairs two query heads of a KV head per CTA; with an
// odd number of query heads per KV head it pairs neighbouring query tiles of
// one head instead, from a work list the metadata pass builds.
bool fwd_tile_pairs(const ism_attn_shape_t* sh) {
  if ((sh->num_heads_q / sh->num_heads_kv) % 2 == 0) return false;
  if (sh->dtype == ISM_E4M3) return true;  // the e4m3 forward runs only the paired kernel
  if (!use_tc(sh) || sh->head_dim != 128) return false;
  return !knobs().fwd_one_head;
}

// Whether a plan has the query-tile pair heads at the front of q_order: that of
// an odd group without a pair list of its own.  The head_dim 64 forward pairs
// tiles from there, so its plans are those of the CUDA-core kernels, in size and
// in use: a plan built for fp32 or under ISM_FORCE_CUDA_CORES=1 serves it and the
// other way round (the kernels that want the cost order read it by q_tile_at).
bool plan_pairs_first(const ism_attn_shape_t* sh) {
  return (sh->num_heads_q / sh->num_heads_kv) % 2 != 0 && !fwd_tile_pairs(sh);
}
// The same of a forward's own metadata pass: only where that forward pairs.
bool pairs_first(const ism_attn_shape_t* sh) {
  return plan_pairs_first(sh) && use_tc(sh) && sh->head_dim == 64;
}

// dS tile slots of the stored-dS backward (pairs x query heads), or 0 where
// that path does not apply: CUDA-core backward, head_dim 64 (the tile is as
// large as at 128 and saves half the work), ISM_BWD_RECOMPUTE_DQ=1, or more
// pairs than the 32-bit pair offsets hold.
int64_t stored_ds_slots(const ism_segments_t* s, const ism_attn_shape_t* sh) {
  if (!use_tc_bwd(sh) || sh->head_dim != 128) return 0;
  if (knobs().bwd_recompute_dq) return 0;
  const int64_t pairs = count_pairs(s);
  if (pairs >= (int64_t(1) << 31)) return 0;
  return pairs * sh->num_heads_q;
}

ism_status_t check_ws(void* ws, size_t have, size_t need) {
  if (have < need) return fail(ISM_ERR_WORKSPACE, "workspace of %zu bytes, %zu required", have, need);
  if (need && !ws) return fail(ISM_ERR_WORKSPACE, "workspace is NULL");
  if (reinterpret_cast<uintptr_t>(ws) & 255u) return fail(ISM_ERR_WORKSPACE, "workspace must be 256-byte aligned");
  return ISM_OK;
}

ism_status_t build_pass_meta(const ism_segments_t* s, const Counts& c, const PassLayout& L, bool bwd,
                             cudaStream_t st, int heads, bool heads_first = false) {
  SegsDev d = dev_view(s);
  timer_begin(ISM_KERNEL_META, st);
  ISM_TRY_CUDA(launch_pass_meta(d, L.kv_end, kTile, kTile, c.nq, bwd ? c.nk : 0, L.qtiles, bwd ? L.ktiles : nullptr,
                                c.max_cost, L.q_order, bwd ? L.k_order : nullptr, L.pair_order, L.kpair_off,
                                L.counters, L.counters ? kPassCounters : 0, st,
                                knobs().dkdv_pair ? L.kp_order : nullptr, heads_first, dependent_pass(c.nq, heads)),
               "metadata launch");
  timer_end(ISM_KERNEL_META, st);
  count_launch(1);
  return ISM_OK;
}

}  // namespace

void timer_begin(int id, cudaStream_t st) {
  if (id > 0 && id < kTimerSlots && g_timer_start[id]) cudaEventRecord(g_timer_start[id], st);
}
void timer_end(int id, cudaStream_t st) {
  if (id > 0 && id < kTimerSlots && g_timer_stop[id]) cudaEventRecord(g_timer_stop[id], st);
}
void count_launch(int n) { g_launches.fetch_add((uint64_t)n, std::memory_order_relaxed); }
void set_error(const char* msg) { g_last_error = msg; }

namespace {
bool env_on(const char* name) {
  const char* e = getenv(name);
  return e && e[0] == '1';
}
int64_t env_int(const char* name, int64_t unset) {
  const char* e = getenv(name);
  return (e && e[0]) ? atoll(e) : unset;
}
Knobs read_knobs() {
  Knobs k;
  k.force_cuda_cores = env_on("ISM_FORCE_CUDA_CORES");
  k.drain_tmem_reuse = env_on("ISM_DRAIN_TMEM_REUSE");
  k.fwd_one_head = env_on("ISM_FWD_ONE_HEAD");
  k.bwd_recompute_dq = env_on("ISM_BWD_RECOMPUTE_DQ");
  k.decode_no_tma = env_on("ISM_DECODE_NO_TMA");
  k.decode_no_tc = env_on("ISM_DECODE_NO_TC");
  const int64_t split = env_int("ISM_PREFILL_SPLIT", -1);
  k.prefill_split = split < 0 ? -1 : split;
  const int64_t g1 = env_int("ISM_DKDV_GRID", 0), g2 = env_int("ISM_DQ_GRID", 0);
  k.dkdv_grid = g1 > 0 && g1 < (1 << 20) ? (int32_t)g1 : 0;
  k.dq_grid = g2 > 0 && g2 < (1 << 20) ? (int32_t)g2 : 0;
  k.dkdv_pair = env_on("ISM_DKDV_PAIR");
  return k;
}
Knobs g_knobs = read_knobs();  // read when the library is loaded

std::mutex g_sm_mu;
std::vector<int> g_sm_count;
}  // namespace

const Knobs& knobs() { return g_knobs; }
void reload_knobs() { g_knobs = read_knobs(); }

int sm_count() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 152;
  std::lock_guard<std::mutex> lk(g_sm_mu);
  if ((int)g_sm_count.size() <= dev) g_sm_count.resize(dev + 1, 0);
  if (!g_sm_count[dev]) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return 152;
    g_sm_count[dev] = sms;
  }
  return g_sm_count[dev];
}

}  // namespace ism

using namespace ism;

extern "C" {

const char* ism_status_string(ism_status_t s) {
  switch (s) {
    case ISM_OK: return "ISM_OK";
    case ISM_ERR_INVALID_ARG: return "ISM_ERR_INVALID_ARG";
    case ISM_ERR_UNSUPPORTED: return "ISM_ERR_UNSUPPORTED";
    case ISM_ERR_CUDA: return "ISM_ERR_CUDA";
    case ISM_ERR_TIMEOUT: return "ISM_ERR_TIMEOUT";
    case ISM_ERR_WORKSPACE: return "ISM_ERR_WORKSPACE";
  }
  return "ISM_ERR_UNKNOWN";
}

const char* ism_last_error(void) { return g_last_error.c_str(); }

int32_t ism_has_tensor_cores(void) { return tc_available() ? 1 : 0; }

ism_status_t ism_set_kernel_timer(int32_t kernel_id, void* start_event, void* stop_event) {
  if (kernel_id <= 0 || kernel_id >= kTimerSlots) return fail(ISM_ERR_INVALID_ARG, "kernel_id %d", kernel_id);
  if ((start_event == nullptr) != (stop_event == nullptr))
    return fail(ISM_ERR_INVALID_ARG, "give both events or neither");
  g_timer_start[kernel_id] = static_cast<cudaEvent_t>(start_event);
  g_timer_stop[kernel_id] = static_cast<cudaEvent_t>(stop_event);
  return ISM_OK;
}

uint64_t ism_kernel_launches(void) { return g_launches.load(); }

void ism_debug_reload_env(void) { reload_knobs(); }

ism_status_t ism_tile_map_size(const ism_segments_t* segs, int32_t bm, int32_t bn, int64_t* n_tiles,
                               int64_t* n_qtiles, int64_t* n_ktiles) {
  SegInfo info;
  ism_status_t r = check_segments(segs, &info);
  if (r != ISM_OK) return r;
  if (bm < 16 || bn < 16 || bm > 256 || bn > 256 || bm % 16 || bn % 16)
    return fail(ISM_ERR_UNSUPPORTED, "tile sizes must be multiples of 16 in [16, 256]");
  Counts c = count_tiles(segs, bm, bn);
  if (n_tiles) *n_tiles = c.ntiles;
  if (n_qtiles) *n_qtiles = c.nq;
  if (n_ktiles) *n_ktiles = c.nk;
  return ISM_OK;
}

ism_status_t ism_build_tile_map(const ism_segments_t* segs, int32_t bm, int32_t bn, uint8_t* tile_class,
                                int32_t* kt_full_end, int32_t* kt_end, int32_t* qt_begin, int32_t* kv_end,
                                ism_stream_t stream) {
  int64_t nt, nq, nk;
  ism_status_t r = ism_tile_map_size(segs, bm, bn, &nt, &nq, &nk);
  if (r != ISM_OK) return r;
  if (segs->cu_seqlens_host[segs->num_seqs] == 0) return ISM_OK;
  if (!kv_end) return fail(ISM_ERR_INVALID_ARG, "kv_end output is required (the tile classes are derived from it)");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  SegsDev d = dev_view(segs);
  ISM_TRY_CUDA(launch_kv_end(d, kv_end, st), "kv_end launch");
  if (tile_class || kt_full_end || kt_end || qt_begin)
    ISM_TRY_CUDA(launch_tiles(d, bm, bn, kv_end, nq, qt_begin ? nk : 0, nullptr, nullptr, tile_class, kt_full_end,
                              kt_end, qt_begin, st),
                 "tiles launch");
  return ISM_OK;
}

ism_status_t ism_attn_fwd_workspace_size(const ism_segments_t* segs, const ism_attn_shape_t* shape,
                                         size_t* bytes) {
  SegInfo info;
  ism_status_t r = check_segments(segs, &info);
  if (r != ISM_OK) return r;
  if ((r = check_shape(shape, true)) != ISM_OK) return r;
  if (!bytes) return fail(ISM_ERR_INVALID_ARG, "bytes is NULL");
  Counts c = count_tiles(segs, kTile, kTile);
  *bytes = pass_layout(nullptr, segs, c, info.total_tokens, shape->num_heads_q, false, 0, fwd_tile_pairs(shape)).bytes;
  return ISM_OK;
}

ism_status_t ism_attn_bwd_workspace_size(const ism_segments_t* segs, const ism_attn_shape_t* shape,
                                         size_t* bytes) {
  SegInfo info;
  ism_status_t r = check_segments(segs, &info);
  if (r != ISM_OK) return r;
  if ((r = check_shape(shape)) != ISM_OK) return r;
  if (!bytes) return fail(ISM_ERR_INVALID_ARG, "bytes is NULL");
  Counts c = count_tiles(segs, kTile, kTile);
  *bytes = pass_layout(nullptr, segs, c, info.total_tokens, shape->num_heads_q, true, stored_ds_slots(segs, shape))
               .bytes;
  return ISM_OK;
}

ism_status_t ism_attn_bwd_workspace_size_min(const ism_segments_t* segs, const ism_attn_shape_t* shape,
                                             size_t* bytes) {
  SegInfo info;
  ism_status_t r = check_segments(segs, &info);
  if (r != ISM_OK) return r;
  if ((r = check_shape(shape)) != ISM_OK) return r;
  if (!bytes) return fail(ISM_ERR_INVALID_ARG, "bytes is NULL");
  Counts c = count_tiles(segs, kTile, kTile);
  *bytes = pass_layout(nullptr, segs, c, info.total_tokens, shape->num_heads_q, true).bytes;
  return ISM_OK;
}

}  // extern "C"

namespace {

// Checks the rotary tables of a one-pass call: present, aligned, covering
// every position of the batch (the longest sequence), for bf16 / fp32 inputs.
ism_status_t check_rope_pass(const ism_rope_t* rope, const ism_attn_shape_t* shape, const SegInfo& info) {
  if (!rope) return fail(ISM_ERR_INVALID_ARG, "rope is NULL");
  if (shape->dtype != ISM_BF16 && shape->dtype != ISM_FP32)
    return fail(ISM_ERR_INVALID_ARG, "rotary encoding on the one-pass path needs bf16 or fp32 inputs");
  if (!rope->cos || !rope->sin || !aligned16(rope->cos) || !aligned16(rope->sin))
    return fail(ISM_ERR_INVALID_ARG, "rope tables must be non-NULL and 16-byte aligned");
  if (info.max_len > rope->rows)
    return fail(ISM_ERR_INVALID_ARG, "rope tables cover %d positions, the longest sequence has %lld tokens", rope->rows,
                (long long)info.max_len);
  return ISM_OK;
}

// The one-pass forward for bf16 / fp32 (ism_attn_fwd) and e4m3 inputs
// (ism_attn_fwd_e4m3; qk_descale = q_descale * k_descale); with rope set,
// q and k are first rotated into q_rot / k_rot and the attention reads those.
ism_status_t fwd_impl(const ism_segments_t* segs, const ism_attn_shape_t* shape, const void* q, const void* k,
                      const void* v, void* o, float* lse, void* workspace, size_t workspace_bytes, ism_stream_t stream,
                      float qk_descale, float v_descale, const ism_rope_t* rope = nullptr, void* q_rot = nullptr,
                      void* k_rot = nullptr, const PassLayout* pre = nullptr) {
  SegInfo info;
  ism_status_t r = check_segments(segs, &info);
  if (r != ISM_OK) return r;
  const bool e4m3 = shape && shape->dtype == ISM_E4M3;
  if ((r = check_shape(shape, e4m3)) != ISM_OK) return r;
  if (e4m3 && !tc_available()) return fail(ISM_ERR_UNSUPPORTED, "e4m3 forward needs the sm_103 tensor cores");
  if (rope && (r = check_rope_pass(rope, shape, info)) != ISM_OK) return r;
  if (info.total_tokens == 0) return ISM_OK;
  if (!q || !k || !v || !o) return fail(ISM_ERR_INVALID_ARG, "q, k, v, o must be non-NULL");
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || (lse && !aligned16(lse)))
    return fail(ISM_ERR_INVALID_ARG, "tensors must be 16-byte aligned");
  if (rope && (!q_rot || !k_rot || !aligned16(q_rot) || !aligned16(k_rot)))
    return fail(ISM_ERR_INVALID_ARG, "q_rot and k_rot must be non-NULL and 16-byte aligned");
  Counts c = count_tiles(segs, kTile, kTile);
  // pre: the metadata of a plan (ism_attn_plan_build), already on the device
  PassLayout L = pre ? *pre
                     : pass_layout(workspace, segs, c, info.total_tokens, shape->num_heads_q, false, 0,
                                   fwd_tile_pairs(shape));
  if (!pre && (r = check_ws(workspace, workspace_bytes, L.bytes)) != ISM_OK) return r;
  uint32_t* status;
  if ((r = status_ptr(&status)) != ISM_OK) return r;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (rope) {
    timer_begin(ISM_KERNEL_ROPE, st);
    ISM_TRY_CUDA(launch_rope_rows(segs->cu_seqlens, segs->num_seqs, info.total_tokens, shape->num_heads_q,
                                  shape->num_heads_kv, shape->head_dim, shape->dtype, q, k, q_rot, k_rot, rope->cos,
                                  rope->sin, 1.f, st, dependent_pass(c.nq, shape->num_heads_q)),
                 "rope launch");
    timer_end(ISM_KERNEL_ROPE, st);
    count_launch(1);
    q = q_rot;
    k = k_rot;
  }
  // query-tile pairs: an odd group
  const bool tile_pairs = L.pair_order || pairs_first(shape);
  // A planned forward walks statically: a plan may serve forwards on several
  // streams at once, and the counter would have to lie in it.
  const bool dynamic = !pre && (use_tc(shape) || e4m3) &&
                       fwd_dynamic(tile_pairs ? c.npairs * shape->num_heads_q : c.nq * (shape->num_heads_q / 2),
                                   tile_pairs);
  if (!pre && (r = build_pass_meta(segs, c, L, false, st, shape->num_heads_q, pairs_first(shape))) != ISM_OK)
    return r;

  AttnArgs a{};
  a.q = q; a.k = k; a.v = v; a.out = o; a.lse = lse;
  a.hq = shape->num_heads_q; a.hkv = shape->num_heads_kv; a.d = shape->head_dim; a.dtype = shape->dtype;
  a.q_rows = info.total_tokens; a.scale = shape->softmax_scale;
  a.dependent = dependent_pass(c.nq, shape->num_heads_q);
  a.qk_descale = qk_descale; a.v_descale = v_descale;
  a.kv_end = L.kv_end; a.qtiles = L.qtiles; a.q_order = L.q_order; a.nq = c.nq;
  a.order_pairs = pre && plan_pairs_first(shape) ? c.npairs : 0;
  a.pair_order = L.pair_order; a.npairs = L.pair_order ? c.npairs : 0;
  if (tile_pairs && !a.pair_order) {
    a.pair_order = L.q_order;
    a.npairs = c.npairs;
  }
  a.work_counter = dynamic ? L.counters + kFwdCounter : nullptr;
  a.bucketed = dynamic ? fwd_bucketed(a, a.npairs * a.hq) : a.hq == a.hkv;
  a.status = status;
  a.flags = tc_flags();
  timer_begin(ISM_KERNEL_FWD, st);
  if (use_tc(shape) || e4m3) {
    ISM_TRY_CUDA(launch_tc_fwd(a, info.total_tokens, st), "tensor-core forward launch");
  } else {
    ISM_TRY_CUDA(launch_simt_fwd(a, st), "forward launch");
  }
  timer_end(ISM_KERNEL_FWD, st);
  count_launch(1);
  return ISM_OK;
}

bool valid_descales(float q_descale, float k_descale, float v_descale) {
  const float ds[3] = {q_descale, k_descale, v_descale};
  for (float x : ds)
    if (!(x > 0.f) || x > 3.0e38f) return false;
  return true;
}

}  // namespace

extern "C" {

ism_status_t ism_attn_fwd(const ism_segments_t* segs, const ism_attn_shape_t* shape, const void* q,
                          const void* k, const void* v, void* o, float* lse, void* workspace,
                          size_t workspace_bytes, ism_stream_t stream) {
  if (shape && shape->dtype == ISM_E4M3)
    return fail(ISM_ERR_UNSUPPORTED, "e4m3 inputs only in ism_attn_fwd_e4m3");
  return fwd_impl(segs, shape, q, k, v, o, lse, workspace, workspace_bytes, stream, 1.f, 1.f);
}

ism_status_t ism_attn_fwd_e4m3(const ism_segments_t* segs, const ism_attn_shape_t* shape, const void* q,
                               const void* k, const void* v, float q_descale, float k_descale, float v_descale,
                               void* o, float* lse, void* workspace, size_t workspace_bytes, ism_stream_t stream) {
  if (!shape || shape->dtype != ISM_E4M3)
    return fail(ISM_ERR_INVALID_ARG, "ism_attn_fwd_e4m3 needs shape->dtype ISM_E4M3");
  if (!valid_descales(q_descale, k_descale, v_descale))
    return fail(ISM_ERR_INVALID_ARG, "descales must be positive finite numbers");
  return fwd_impl(segs, shape, q, k, v, o, lse, workspace, workspace_bytes, stream, q_descale * k_descale, v_descale);
}

ism_status_t ism_attn_fwd_rope(const ism_segments_t* segs, const ism_attn_shape_t* shape, const void* q,
                               const void* k, const void* v, const ism_rope_t* rope, void* q_rot, void* k_rot,
                               void* o, float* lse, void* workspace, size_t workspace_bytes, ism_stream_t stream) {
  if (shape && shape->dtype == ISM_E4M3)
    return fail(ISM_ERR_INVALID_ARG, "rotary encoding on the one-pass path needs bf16 or fp32 inputs");
  if (!rope) return fail(ISM_ERR_INVALID_ARG, "rope is NULL");
  return fwd_impl(segs, shape, q, k, v, o, lse, workspace, workspace_bytes, stream, 1.f, 1.f, rope, q_rot, k_rot);
}

}  // extern "C"

namespace {

ism_status_t bwd_impl(const ism_segments_t* segs, const ism_attn_shape_t* shape, const void* q, const void* k,
                      const void* v, const void* o, const float* lse, const void* dout, void* dq, void* dk, void* dv,
                      void* workspace, size_t workspace_bytes, ism_stream_t stream, const ism_rope_t* rope,
                      const PassLayout* pre = nullptr) {
  SegInfo info;
  ism_status_t r = check_segments(segs, &info);
  if (r != ISM_OK) return r;
  if ((r = check_shape(shape)) != ISM_OK) return r;
  if (rope && (r = check_rope_pass(rope, shape, info)) != ISM_OK) return r;
  if (info.total_tokens == 0) return ISM_OK;
  if (!q || !k || !v || !o || !lse || !dout || !dq || !dk || !dv)
    return fail(ISM_ERR_INVALID_ARG, "q, k, v, o, lse, dout, dq, dk, dv must be non-NULL");
  const void* ptrs[] = {q, k, v, o, lse, dout, dq, dk, dv};
  for (const void* p : ptrs)
    if (!aligned16(p)) return fail(ISM_ERR_INVALID_ARG, "tensors must be 16-byte aligned");
  Counts c = count_tiles(segs, kTile, kTile);
  // the stored-dS path when the workspace holds its tiles, else recompute
  int64_t slots = stored_ds_slots(segs, shape);
  PassLayout L;
  if (pre) {
    // metadata from a plan; Delta and the dS tiles from the workspace
    L = *pre;
    Carve cv(workspace);
    L.delta = cv.take<float>((int64_t)shape->num_heads_q * info.total_tokens);
    const size_t need_min = ((cv.off + 255) & ~size_t(255)) + 256;
    void* ds = slots > 0 ? static_cast<void*>(cv.take<uint16_t>(slots * kTile * kTile)) : nullptr;
    const size_t need_full = ((cv.off + 255) & ~size_t(255)) + 256;
    L.ds = ds && workspace_bytes >= need_full ? ds : nullptr;
    if (!L.ds) slots = 0;
    L.bytes = L.ds ? need_full : need_min;
  } else {
    L = pass_layout(workspace, segs, c, info.total_tokens, shape->num_heads_q, true, slots);
    if (slots > 0 && workspace_bytes < L.bytes) {
      L = pass_layout(workspace, segs, c, info.total_tokens, shape->num_heads_q, true);
      slots = 0;
    }
  }
  if ((r = check_ws(workspace, workspace_bytes, L.bytes)) != ISM_OK) return r;
  uint32_t* status;
  if ((r = status_ptr(&status)) != ISM_OK) return r;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (pre) {
    // the plan's work counter starts at zero for this call
    ISM_TRY_CUDA(cudaMemsetAsync(L.counters + kBwdCounter, 0, sizeof(int32_t), st), "work counter reset");
  } else if ((r = build_pass_meta(segs, c, L, true, st, shape->num_heads_q)) != ISM_OK) {
    return r;
  }

  AttnArgs a{};
  a.q = q; a.k = k; a.v = v; a.o = o; a.dout = dout; a.lse_in = lse;
  a.dq = dq; a.dk = dk; a.dv = dv; a.delta = L.delta;
  a.hq = shape->num_heads_q; a.hkv = shape->num_heads_kv; a.d = shape->head_dim; a.dtype = shape->dtype;
  a.q_rows = info.total_tokens; a.scale = shape->softmax_scale;
  a.dependent = dependent_pass(c.nq, shape->num_heads_q);
  a.kv_end = L.kv_end; a.qtiles = L.qtiles; a.q_order = L.q_order; a.nq = c.nq;
  a.order_pairs = pre && plan_pairs_first(shape) ? c.npairs : 0;
  a.ktiles = L.ktiles; a.k_order = L.k_order; a.nk = c.nk;
  a.ds = L.ds; a.kpair_off = L.kpair_off; a.ds_slots = L.ds ? slots : 0;
  a.work_counter = L.counters + kBwdCounter;
  // the k-tile pair list exists only when the CTA-pair dK/dV kernel will run
  // (and a plan holds none)
  a.kp_order = knobs().dkdv_pair && !pre ? L.kp_order : nullptr;
  a.nkp = a.kp_order ? c.npairs : 0;
  a.status = status;
  a.flags = tc_flags();
  if (use_tc_bwd(shape)) {
    if (rope) {  // the dQ and dK epilogues rotate the gradients back
      a.rope_cos = rope->cos;
      a.rope_sin = rope->sin;
    }
    ISM_TRY_CUDA(launch_tc_bwd(a, info.total_tokens, st), "tensor-core backward launch");
  } else {
    ISM_TRY_CUDA(launch_simt_bwd(a, st), "backward launch");
    if (rope) {  // gradients of the rotated rows, rotated back in place
      timer_begin(ISM_KERNEL_ROPE, st);
      ISM_TRY_CUDA(launch_rope_rows(segs->cu_seqlens, segs->num_seqs, info.total_tokens, shape->num_heads_q,
                                    shape->num_heads_kv, shape->head_dim, shape->dtype, dq, dk, dq, dk, rope->cos,
                                    rope->sin, -1.f, st, a.dependent),
                   "rope launch");
      timer_end(ISM_KERNEL_ROPE, st);
      count_launch(1);
    }
  }
  return ISM_OK;
}

}  // namespace

extern "C" {

ism_status_t ism_attn_bwd(const ism_segments_t* segs, const ism_attn_shape_t* shape, const void* q,
                          const void* k, const void* v, const void* o, const float* lse, const void* dout,
                          void* dq, void* dk, void* dv, void* workspace, size_t workspace_bytes,
                          ism_stream_t stream) {
  return bwd_impl(segs, shape, q, k, v, o, lse, dout, dq, dk, dv, workspace, workspace_bytes, stream, nullptr);
}

ism_status_t ism_attn_bwd_rope(const ism_segments_t* segs, const ism_attn_shape_t* shape, const void* q_rot,
                               const void* k_rot, const void* v, const void* o, const float* lse, const void* dout,
                               const ism_rope_t* rope, void* dq, void* dk, void* dv, void* workspace,
                               size_t workspace_bytes, ism_stream_t stream) {
  if (!rope) return fail(ISM_ERR_INVALID_ARG, "rope is NULL");
  return bwd_impl(segs, shape, q_rot, k_rot, v, o, lse, dout, dq, dk, dv, workspace, workspace_bytes, stream, rope);
}

// ---------------------------------------------------------------- plans

ism_status_t ism_attn_plan_size(const ism_segments_t* segs, const ism_attn_shape_t* shape, size_t* bytes) {
  SegInfo info;
  ism_status_t r = check_segments(segs, &info);
  if (r != ISM_OK) return r;
  if ((r = check_shape(shape)) != ISM_OK) return r;
  if (!bytes) return fail(ISM_ERR_INVALID_ARG, "bytes is NULL");
  Counts c = count_tiles(segs, kTile, kTile);
  *bytes = plan_layout(nullptr, c, info.total_tokens, fwd_tile_pairs(shape)).bytes;
  return ISM_OK;
}

ism_status_t ism_attn_plan_build(const ism_segments_t* segs, const ism_attn_shape_t* shape, void* plan,
                                 size_t plan_bytes, ism_attn_plan_info_t* plan_info, ism_stream_t stream) {
  SegInfo info;
  ism_status_t r = check_segments(segs, &info);
  if (r != ISM_OK) return r;
  if ((r = check_shape(shape)) != ISM_OK) return r;
  if (!plan_info) return fail(ISM_ERR_INVALID_ARG, "plan_info is NULL");
  Counts c = count_tiles(segs, kTile, kTile);
  const bool tile_pairs = fwd_tile_pairs(shape);
  PassLayout L = plan_layout(plan, c, info.total_tokens, tile_pairs);
  if ((r = check_ws(plan, plan_bytes, L.bytes)) != ISM_OK) return r;
  if (info.total_tokens > 0) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if ((r = build_pass_meta(segs, c, L, true, st, shape->num_heads_q, plan_pairs_first(shape))) != ISM_OK) return r;
  }
  plan_info->fingerprint = plan_fingerprint(segs, shape, tile_pairs);
  plan_info->bytes = L.bytes;
  return ISM_OK;
}

}  // extern "C"

namespace {

// The layout of a plan for these segments and shape, after checking that the
// plan was built for them.
ism_status_t planned_layout(const ism_segments_t* segs, const ism_attn_shape_t* shape, const void* plan,
                            const ism_attn_plan_info_t* plan_info, PassLayout* L) {
  SegInfo info;
  ism_status_t r = check_segments(segs, &info);
  if (r != ISM_OK) return r;
  if ((r = check_shape(shape)) != ISM_OK) return r;
  if (!plan || !plan_info) return fail(ISM_ERR_INVALID_ARG, "plan and plan_info must be non-NULL");
  if (reinterpret_cast<uintptr_t>(plan) & 255u) return fail(ISM_ERR_INVALID_ARG, "plan must be 256-byte aligned");
  const bool tile_pairs = fwd_tile_pairs(shape);
  if (plan_fingerprint(segs, shape, tile_pairs) != plan_info->fingerprint)
    return fail(ISM_ERR_INVALID_ARG, "the plan was built for other segments or head counts");
  Counts c = count_tiles(segs, kTile, kTile);
  *L = plan_layout(const_cast<void*>(plan), c, info.total_tokens, tile_pairs);
  if (plan_info->bytes < L->bytes) return fail(ISM_ERR_INVALID_ARG, "plan_info does not describe this plan");
  return ISM_OK;
}

}  // namespace

extern "C" {

ism_status_t ism_attn_fwd_planned(const ism_segments_t* segs, const ism_attn_shape_t* shape, const void* plan,
                                  const ism_attn_plan_info_t* plan_info, const void* q, const void* k,
                                  const void* v, void* o, float* lse, ism_stream_t stream) {
  PassLayout L;
  ism_status_t r = planned_layout(segs, shape, plan, plan_info, &L);
  if (r != ISM_OK) return r;
  return fwd_impl(segs, shape, q, k, v, o, lse, nullptr, 0, stream, 1.f, 1.f, nullptr, nullptr, nullptr, &L);
}

ism_status_t ism_attn_bwd_planned(const ism_segments_t* segs, const ism_attn_shape_t* shape, void* plan,
                                  const ism_attn_plan_info_t* plan_info, const void* q, const void* k,
                                  const void* v, const void* o, const float* lse, const void* dout, void* dq,
                                  void* dk, void* dv, void* workspace, size_t workspace_bytes,
                                  ism_stream_t stream) {
  PassLayout L;
  ism_status_t r = planned_layout(segs, shape, plan, plan_info, &L);
  if (r != ISM_OK) return r;
  return bwd_impl(segs, shape, q, k, v, o, lse, dout, dq, dk, dv, workspace, workspace_bytes, stream, nullptr, &L);
}

ism_status_t ism_attn_fwd_rope_planned(const ism_segments_t* segs, const ism_attn_shape_t* shape, const void* plan,
                                       const ism_attn_plan_info_t* plan_info, const void* q, const void* k,
                                       const void* v, const ism_rope_t* rope, void* q_rot, void* k_rot, void* o,
                                       float* lse, ism_stream_t stream) {
  if (!rope) return fail(ISM_ERR_INVALID_ARG, "rope is NULL");
  PassLayout L;
  ism_status_t r = planned_layout(segs, shape, plan, plan_info, &L);
  if (r != ISM_OK) return r;
  return fwd_impl(segs, shape, q, k, v, o, lse, nullptr, 0, stream, 1.f, 1.f, rope, q_rot, k_rot, &L);
}

ism_status_t ism_attn_bwd_rope_planned(const ism_segments_t* segs, const ism_attn_shape_t* shape, void* plan,
                                       const ism_attn_plan_info_t* plan_info, const void* q_rot, const void* k_rot,
                                       const void* v, const void* o, const float* lse, const void* dout,
                                       const ism_rope_t* rope, void* dq, void* dk, void* dv, void* workspace,
                                       size_t workspace_bytes, ism_stream_t stream) {
  if (!rope) return fail(ISM_ERR_INVALID_ARG, "rope is NULL");
  PassLayout L;
  ism_status_t r = planned_layout(segs, shape, plan, plan_info, &L);
  if (r != ISM_OK) return r;
  return bwd_impl(segs, shape, q_rot, k_rot, v, o, lse, dout, dq, dk, dv, workspace, workspace_bytes, stream, rope,
                  &L);
}

// ---------------------------------------------------------------- append

namespace {

struct AppendLayout {
  int32_t* c_snap;
  int32_t* kv_end;
  Tile* qtiles;
  int32_t* q_order;
  int32_t* pair_order;  // neighbouring q-tiles of a chunk, for the paired forward
  int64_t npairs;
  float* part_o;
  float* part_ml;
  void* q_rot;  // rotated queries of a RoPE append (bf16 [batch * l_new, Hq, D]), else null
  // partials of the forward's key-range split (prefill), the last region: as
  // many units as the caller's workspace holds
  size_t part_off;
  int32_t part_rows;   // rows of a unit's half
  size_t bytes;        // what the call requires
  size_t full_bytes;   // what the size query reports: partials for as many units as a split can use
};

// Key-range units of a split forward that the reported workspace holds, at most.
constexpr int64_t kMaxSplitUnits = 512;

// One-head items (query tile, head pair), or (query-tile pair, head) for an odd group.
int64_t append_items(const ism_attn_shape_t* sh, int batch, int l_new, bool tile_pairs) {
  const int64_t nqt = (l_new + kTile - 1) / kTile;
  return batch * (tile_pairs ? (nqt + 1) / 2 * sh->num_heads_q : nqt * (sh->num_heads_q / 2));
}

AppendLayout append_layout(void* ws, const ism_attn_shape_t* sh, int batch, int l_new, bool rope = false) {
  Carve cv(ws);
  AppendLayout L;
  const int64_t nqt_seq = (l_new + kTile - 1) / kTile;
  int64_t nqt = (int64_t)batch * nqt_seq;
  L.c_snap = cv.take<int32_t>(batch);
  L.kv_end = cv.take<int32_t>((int64_t)batch * l_new);
  L.qtiles = cv.take<Tile>(nqt);
  L.q_order = cv.take<int32_t>(nqt);
  L.npairs = (int64_t)batch * ((nqt_seq + 1) / 2);
  L.pair_order = cv.take<int32_t>(L.npairs);
  if (l_new == 1) {
    L.part_o = cv.take<float>((int64_t)batch * sh->num_heads_q * kMaxSplits * sh->head_dim);
    L.part_ml = cv.take<float>((int64_t)batch * sh->num_heads_q * kMaxSplits * 2);
  } else {
    L.part_o = L.part_ml = nullptr;
  }
  L.q_rot = rope ? (void*)cv.take<__nv_bfloat16>((int64_t)batch * l_new * sh->num_heads_q * sh->head_dim) : nullptr;
  L.part_off = (cv.off + 255) & ~size_t(255);
  L.part_rows = l_new < kTile ? l_new : kTile;
  // required: two halves of up to 256 head-pair items with whole tiles
  if (l_new > 1 && sh->num_heads_q % 2 == 0) {
    int64_t items = nqt * (sh->num_heads_q / 2);
    if (items > 256) items = 256;
    cv.take<float>(items * 2 * 2 * kTile * 128);
    cv.take<float>(items * 2 * 2 * kTile * 2);
  }
  L.bytes = ((cv.off + 255) & ~size_t(255)) + 256;
  L.full_bytes = L.bytes;
  if (l_new > 1 && sh->dtype != ISM_FP32) {
    int64_t units = 32 * append_items(sh, batch, l_new, (sh->num_heads_q / sh->num_heads_kv) % 2 != 0);
    if (units > kMaxSplitUnits) units = kMaxSplitUnits;
    const size_t full = L.part_off + (size_t)units * 2 * L.part_rows * (sh->head_dim + 2) * sizeof(float) + 512;
    if (full > L.full_bytes) L.full_bytes = full;
  }
  return L;
}

// How a prefill's items are split over their key range.  All items cost about
// the same (every row sees the whole cache), so with `items` below the SM
// count every item is split, else those of the last, partial round; into the
// number of parts that minimises the rounds of that part of the launch, at
// ceil(tiles / parts) key tiles and about two tiles' time of start-up and
// epilogue each, plus the merge (a dependent launch and the partials written
// and read once, together at about 3 TB/s).  In units of a key tile, 1.46 us.
// Measured: one 40-token query over 3000 keys (16 items of 24 tiles) forward
// 51 us whole, 30 in two halves, 14 in eight parts, and a 6 us merge; 8 x 512
// queries over 16384 keys (512 items of 132 tiles) 826 us a call whole, 770
// with the last 56 split; 20 x 100 over 8000 keys 392 whole, 311 split.
struct KeySplit {
  int64_t items = 0;  // split items (the last ones); 0: none
  int32_t parts = 1;
};
// e4m3: P is rounded to three mantissa bits relative to its part's maximum, so
// another split gives other roundings (3.5 % of the output between two equally
// exact results); it keeps two halves of the last round's items, from 64 key
// tiles on.
KeySplit plan_key_split(const ism_attn_shape_t* sh, int64_t items, int64_t tiles, int rows, int64_t cap_units) {
  const int64_t sms = sm_count();
  const int head_dim = sh->head_dim;
  KeySplit best;
  const int64_t n = items < sms ? items : items % sms;
  if (n == 0) return best;
  if (sh->dtype == ISM_E4M3) {
    if ((sh->num_heads_q / sh->num_heads_kv) % 2 == 0 && items > sms && tiles >= 64) {
      best.items = n * 2 > cap_units ? cap_units / 2 : n;
      best.parts = 2;
    }
    return best;
  }
  double best_cost = 0;
  for (int p = 1; p <= 32 && p <= tiles; ++p) {
    if (p > 1 && n * p > cap_units) break;
    double cost = (double)((n * p + sms - 1) / sms) * (double)((tiles + p - 1) / p + 2);
    if (p > 1) cost += 2.0 + (double)(n * p) * rows * head_dim * 16.0 / 3.0e6 / 1.46;
    if (p == 1 || cost < best_cost) {
      best_cost = cost;
      best.items = p > 1 ? n : 0;
      best.parts = p;
    }
  }
  return best;
}

}  // namespace

ism_status_t ism_attn_prefill_append_workspace_size(const ism_attn_shape_t* shape, int32_t batch, int32_t l_new,
                                                    size_t* bytes) {
  ism_status_t r = check_shape(shape, true);
  if (r != ISM_OK) return r;
  if (batch < 0 || l_new < 0) return fail(ISM_ERR_INVALID_ARG, "batch and l_new must be >= 0");
  if (!bytes) return fail(ISM_ERR_INVALID_ARG, "bytes is NULL");
  *bytes = append_layout(nullptr, shape, batch, l_new).full_bytes;  // (e4m3 shapes included)
  return ISM_OK;
}

ism_status_t ism_attn_prefill_append_rope_workspace_size(const ism_attn_shape_t* shape, int32_t batch,
                                                         int32_t l_new, size_t* bytes) {
  ism_status_t r = check_shape(shape, true);
  if (r != ISM_OK) return r;
  if (batch < 0 || l_new < 0) return fail(ISM_ERR_INVALID_ARG, "batch and l_new must be >= 0");
  if (!bytes) return fail(ISM_ERR_INVALID_ARG, "bytes is NULL");
  *bytes = append_layout(nullptr, shape, batch, l_new, true).full_bytes;
  return ISM_OK;
}

}  // extern "C"

namespace {

// Cache geometry of one append call: contiguous [B, cap] caches, or pages.
constexpr int kMaxDecodeGroup = 16;

struct CacheGeom {
  int64_t cap;       // contiguous: rows per sequence
  int64_t kv_rows;   // rows of the K / V tensors (tensor-map extent)
  int64_t max_keys;  // keys a sequence can hold
  KvPages pages;     // table == nullptr: contiguous
};

// The row split of the bf16 tensor-core decode (DecodeArgs): tiles per CTA so that
// one CTA per SM covers the row, and room for the partials of any (sequence, KV
// head): the CTAs that its tiles touch, times the items of a CTA's share.
// Where that exceeds kMaxSplits (a few very long caches), every cache starts at
// a CTA's share of kDecTcTiles tiles instead.  Neighbouring CTAs take the same
// share for up to eight KV heads (lanes), whose rows lie side by side: 8 caches
// of 12000 to 16384 keys 80.0 -> 76.5 us a step against one row of all heads.
// false: equal chunks, because the caches are about as long as the longest (its
// tiles at most 1.12 of their mean) and the shares are long, or the row has more
// tiles than 32 bits hold.  Equal chunks leave idle at most what the longest is
// above the mean and have fewer short items.  Chunks and row, us a step: 8 x
// 16384 keys (shares of 55 tiles) 82.5 and 86.0, 4 x 16384 (28) 46.4 and 48.8, 4
// of 8400 to 9000 (15) 30.0 and 30.2, 1 x 3000 (2) 11.3 and 10.7; 8 from 0.85 of
// 16384 to all of it (1.08) 79.1 and 82.2, from 0.75 (1.14) 77.7 and 76.5, from
// 0.6 74.5 and 71.4; 32 from 0.75 of 4000 79.3 and 79.0; 24 up to 3000 with 16 / 4
// heads 25.0 and 21.8.
// Error against 64 bits with P in two parts, and in equal chunks with P in bf16: 40
// paged caches up to 4000 keys 0.00166 and 0.00224, 8 up to 16384 0.00166 and
// 0.00228, 20 x 1000 0.00166 and 0.00221, one of 3001, rotated, 0.00237 and 0.00277
// (0.00166 is the rounding of the output); of LSE 5e-8 and 2e-6 to 2e-5.
bool decode_row(DecodeArgs& a, const int32_t* cache_len_host, int32_t batch, int32_t hkv, int sms) {
  int64_t sum = 0;
  int32_t most = 0;
  for (int b = 0; b < batch; ++b) {
    const int32_t n = dec_tiles(cache_len_host[b]);
    sum += n;
    if (n > most) most = n;
  }
  a.align = 1;
  a.lanes = 8;
  while (hkv % a.lanes || sms % a.lanes) a.lanes /= 2;
  const int64_t groups = sms / a.lanes;
  int64_t row = sum * (hkv / a.lanes), tpc = (row + groups - 1) / groups;
  if (tpc > 16 && (int64_t)most * batch * 25 <= sum * 28) return false;
  const int64_t per_cta = (tpc + kDecTcTiles - 1) / kDecTcTiles;
  int64_t slots = ((most + tpc - 1) / tpc + 1) * per_cta;
  if (slots > kMaxSplits) {
    tpc = a.align = kDecTcTiles;
    row = 0;
    for (int b = 0; b < batch; ++b) row += dec_alloc_tiles(a, dec_tiles(cache_len_host[b]));
    row *= hkv / a.lanes;
    slots = (most + tpc - 1) / tpc;
  }
  if (row >= (int64_t(1) << 31) - kDecTcTiles || slots > kMaxSplits) return false;
  a.tpc = (int32_t)tpc;
  a.shares = (int32_t)((row + tpc - 1) / tpc);
  a.splits = kMaxSplits;
  a.chunk = 0;
  return true;
}

ism_status_t append_impl(const ism_attn_shape_t* shape, int32_t batch, const void* q_new, const void* k_new,
                         const void* v_new, int32_t l_new, const int32_t* new_seg_end_host,
                         const uint8_t* new_seg_type_host, int32_t n_new_segs, void* k_cache, void* v_cache,
                         const CacheGeom& cg, int32_t* cache_len, const int32_t* cache_len_host, void* o_new,
                         float* lse_new, void* workspace, size_t workspace_bytes, cudaStream_t st,
                         float q_descale = 1.f, float k_descale = 1.f, float v_descale = 1.f,
                         const ism_rope_t* rope = nullptr) {
  const float qk_descale = q_descale * k_descale;
  ism_status_t r;
  if (!q_new || !k_new || !v_new || !k_cache || !v_cache || !cache_len || !cache_len_host || !o_new)
    return fail(ISM_ERR_INVALID_ARG, "q_new, k_new, v_new, caches, cache_len (device+host), o_new must be non-NULL");
  const void* ptrs[] = {q_new, k_new, v_new, k_cache, v_cache, o_new};
  for (const void* p : ptrs)
    if (!aligned16(p)) return fail(ISM_ERR_INVALID_ARG, "tensors must be 16-byte aligned");
  if (lse_new && !aligned16(lse_new)) return fail(ISM_ERR_INVALID_ARG, "lse_new must be 16-byte aligned");
  if (!new_seg_end_host || !new_seg_type_host || n_new_segs <= 0 || n_new_segs > kMaxAppendSegs)
    return fail(ISM_ERR_INVALID_ARG, "chunk needs 1..%d segments", kMaxAppendSegs);
  AppendSegs sg;
  memset(&sg, 0, sizeof(sg));
  sg.n = n_new_segs;
  sg.l_new = l_new;
  int32_t prev = 0;
  for (int i = 0; i < n_new_segs; ++i) {
    if (new_seg_end_host[i] < prev) return fail(ISM_ERR_INVALID_ARG, "chunk seg_end not non-decreasing");
    if (new_seg_type_host[i] > 1) return fail(ISM_ERR_INVALID_ARG, "chunk segment type %d", (int)new_seg_type_host[i]);
    sg.end[i] = prev = new_seg_end_host[i];
    sg.type[i] = new_seg_type_host[i];
  }
  if (prev != l_new) return fail(ISM_ERR_INVALID_ARG, "chunk segments end at %d, l_new is %d", prev, l_new);
  if ((int64_t)batch * l_new >= (int64_t(1) << 31)) return fail(ISM_ERR_INVALID_ARG, "batch * l_new too large");
  int32_t max_c = 0;
  for (int b = 0; b < batch; ++b) {
    int32_t c = cache_len_host[b];
    if (c < 0 || (int64_t)c + l_new > cg.max_keys)
      return fail(ISM_ERR_INVALID_ARG, "sequence %d: cache_len %d + l_new %d exceeds capacity %lld", b, c, l_new,
                  (long long)cg.max_keys);
    if (c > max_c) max_c = c;
  }
  if (rope) {
    if (!rope->cos || !rope->sin || !aligned16(rope->cos) || !aligned16(rope->sin))
      return fail(ISM_ERR_INVALID_ARG, "rope tables must be non-NULL and 16-byte aligned");
    if ((int64_t)max_c + l_new > rope->rows)
      return fail(ISM_ERR_INVALID_ARG, "rope tables cover %d positions, the append writes up to %lld", rope->rows,
                  (long long)max_c + l_new);
  }
  AppendLayout L = append_layout(workspace, shape, batch, l_new, rope != nullptr);
  if ((r = check_ws(workspace, workspace_bytes, L.bytes)) != ISM_OK) return r;
  uint32_t* status;
  if ((r = status_ptr(&status)) != ISM_OK) return r;
  const int hq = shape->num_heads_q, hkv = shape->num_heads_kv, d = shape->head_dim;
  const bool paged = cg.pages.table != nullptr;

  // decode kernels serve up to kMaxDecodeGroup query heads per KV head; larger
  // groups take the forward kernels (one query row per tile)
  const bool decode = l_new == 1 && (shape->dtype == ISM_BF16 || shape->dtype == ISM_E4M3) && !force_cuda_cores() &&
                      hq / hkv <= kMaxDecodeGroup;
  // The cache write lays out the chunk's plan (a single-token step needs none,
  // but a copy of the cache lengths); the attention kernels advance the lengths.
  AppendPlan plan{};
  if (!decode) {
    plan.segs = sg;
    plan.kbase_stride = paged ? 1 : cg.cap;
    plan.bm = plan.bn = kTile;
    plan.kv_end = L.kv_end; plan.qtiles = L.qtiles; plan.q_order = L.q_order; plan.pair_order = L.pair_order;
    plan.counter = L.c_snap;  // (only single-token steps have lengths there)
  }
  timer_begin(ISM_KERNEL_META, st);
  int32_t* snap_out = decode ? L.c_snap : nullptr;
  if (rope) {
    ISM_TRY_CUDA(launch_rope_cache_write(shape->dtype, batch, l_new, hq, hkv, d, cg.cap, cg.pages, cache_len, q_new,
                                         k_new, v_new, rope->cos, rope->sin, q_descale, k_descale, v_descale,
                                         L.q_rot, k_cache, v_cache, plan, st, snap_out),
                 "rope cache write launch");
    q_new = L.q_rot;  // the attention below reads the rotated queries
  } else {
    ISM_TRY_CUDA(launch_cache_write(shape->dtype, batch, l_new, hkv, d, cg.cap, cg.pages, cache_len, k_new, v_new,
                                    k_cache, v_cache, plan, st, snap_out),
                 "cache write launch");
  }
  timer_end(ISM_KERNEL_META, st);
  count_launch(1);
  if (decode) {
    DecodeArgs a{};
    a.cache_len = cache_len;
    a.q_written = rope != nullptr;
    a.q = q_new; a.k_cache = k_cache; a.v_cache = v_cache; a.pages = cg.pages; a.out = o_new; a.lse = lse_new;
    a.c_snap = L.c_snap;
    a.batch = batch; a.hq = hq; a.hkv = hkv; a.d = d; a.dtype = shape->dtype; a.cap = cg.cap;
    a.group = hq / hkv;
    a.qk_descale = qk_descale; a.v_descale = v_descale;
    a.kv_rows = cg.kv_rows;
    a.scale = shape->softmax_scale;
    int64_t kv_max = (int64_t)max_c + 1;
    int64_t pairs = (int64_t)batch * hkv;
    const int sms = sm_count();
    a.tma = (d == 128 && tc_available() && !knobs().decode_no_tma) ? 1 : 0;
    const bool e4m3 = shape->dtype == ISM_E4M3;
    a.tc = a.tma && !knobs().decode_no_tc && kv_max <= (int64_t)kMaxSplits * kDecTcMaxKeys;
    if (a.tc && !e4m3 && decode_row(a, cache_len_host, batch, hkv, sms)) {
      a.start = L.kv_end;  // (a single-token step has no plan there)
    } else if (a.tc) {
      // equal chunks: the split count that minimises the busiest CTA's work,
      // (items per CTA) x (128-key tiles per item + 1 for the item's hand-offs),
      // over whole tiles up to kDecTcMaxKeys
      int64_t best = -1;
      for (int64_t sp = 1; sp <= kMaxSplits; ++sp) {
        const int64_t ch = ((kv_max + sp - 1) / sp + 127) / 128 * 128;
        if (ch > kDecTcMaxKeys) continue;
        const int64_t used = (kv_max + ch - 1) / ch;
        const int64_t per_cta = (pairs * used + sms - 1) / sms;
        const int64_t cost = per_cta * (ch / 128 + 1);
        if (best < 0 || cost < best) {
          best = cost;
          a.splits = (int32_t)used;
          a.chunk = (int32_t)ch;
        }
      }
    } else {
      // chunks of a multiple of 64 keys, as many as fill whole waves of resident
      // CTAs: 4 per SM for the register kernel (one wave), 2 per SM for the TMA
      // kernel (four waves, so each CTA's ring runs several tiles)
      int64_t want = (a.tma ? 8 * (int64_t)sms : 4 * (int64_t)sms) / pairs;
      int64_t splits = want < 1 ? 1 : want > kMaxSplits ? kMaxSplits : want;
      int64_t chunk = (kv_max + splits - 1) / splits;
      chunk = (chunk + 63) / 64 * 64;
      a.splits = (int32_t)((kv_max + chunk - 1) / chunk);
      a.chunk = (int32_t)chunk;
    }
    a.part_o = L.part_o; a.part_ml = L.part_ml;
    a.status = status;
    timer_begin(ISM_KERNEL_DECODE, st);
    ISM_TRY_CUDA(launch_decode(a, st), "decode launch");
    timer_end(ISM_KERNEL_DECODE, st);
    count_launch(2);
    return ISM_OK;
  }
  AttnArgs a{};
  a.q = q_new; a.k = k_cache; a.v = v_cache; a.out = o_new; a.lse = lse_new;
  a.hq = hq; a.hkv = hkv; a.d = d; a.dtype = shape->dtype;
  a.q_rows = (int64_t)batch * l_new; a.scale = shape->softmax_scale;
  a.dependent = dependent_pass((int64_t)batch * ((l_new + kTile - 1) / kTile), hq);
  a.kv_end = L.kv_end; a.qtiles = L.qtiles; a.q_order = L.q_order;
  a.nq = (int64_t)batch * ((l_new + kTile - 1) / kTile);
  a.pages = cg.pages;
  a.qk_descale = qk_descale;
  a.v_descale = v_descale;
  a.adv_cache_len = cache_len;
  a.adv_batch = batch;
  a.adv_len = l_new;
  a.status = status;
  a.flags = tc_flags();
  if (use_tc(shape) || shape->dtype == ISM_E4M3) {
    const bool odd = (hq / hkv) % 2 != 0;
    const int64_t tiles = ((int64_t)max_c + l_new + kTile - 1) / kTile;
    const int64_t items = append_items(shape, batch, l_new, odd);
    const int64_t cap_units = (int64_t)((workspace_bytes - L.part_off) /
                                        ((size_t)2 * L.part_rows * (d + 2) * sizeof(float)));
    KeySplit sp = plan_key_split(shape, items, tiles, L.part_rows, cap_units);
    if (knobs().prefill_split >= 0) {  // ISM_PREFILL_SPLIT=n: n items as two halves
      sp.items = knobs().prefill_split < items ? knobs().prefill_split : items;
      sp.parts = 2;
      if (sp.items * 2 > cap_units) sp.items = cap_units / 2;
    }
    // An odd group pairs neighbouring q-tiles of a head.  e4m3 and head_dim 64
    // have only the paired kernel; bf16 at 128 takes the one-head kernel
    // instead when no tile has a neighbour (half of a paired CTA would idle),
    // unless its rounds leave a quarter of the SMs idle and the items split:
    // 32 heads over 16 x 4000 keys (512 items, 0.84 of four rounds) one-head
    // 212 us, split pairs 227; over 6 x 16000 keys (192, 0.63) 366 and 314.
    const int64_t rounds = (items + sm_count() - 1) / sm_count();
    const bool one_head = d == 128 && shape->dtype == ISM_BF16 &&
                          (knobs().fwd_one_head ||
                           (odd && l_new <= kTile && (sp.items == 0 || items * 4 > rounds * sm_count() * 3)));
    if (fwd_dynamic(items, odd)) a.work_counter = L.c_snap;
    if (odd && !one_head) {
      a.pair_order = L.pair_order;
      a.npairs = L.npairs;
    }
    if (!one_head && sp.items > 0) {
      a.split_items = sp.items;
      a.split_whole = items - sp.items;
      a.split_parts = sp.parts;
      a.part_rows = L.part_rows;
      a.part_o = reinterpret_cast<float*>(reinterpret_cast<uintptr_t>(workspace) + L.part_off);
      a.part_ml = a.part_o + sp.items * sp.parts * 2 * L.part_rows * d;
    }
  }
  timer_begin(ISM_KERNEL_FWD, st);
  if (use_tc(shape) || shape->dtype == ISM_E4M3) {
    ISM_TRY_CUDA(launch_tc_fwd(a, cg.kv_rows, st), "tensor-core prefill launch");
  } else {
    ISM_TRY_CUDA(launch_simt_fwd(a, st), "prefill launch");
  }
  timer_end(ISM_KERNEL_FWD, st);
  count_launch(a.split_items > 0 ? 2 : 1);  // the key-range halves are merged by a second kernel
  return ISM_OK;
}

}  // namespace

extern "C" {

ism_status_t ism_attn_prefill_append(const ism_attn_shape_t* shape, int32_t batch, const void* q_new,
                                     const void* k_new, const void* v_new, int32_t l_new,
                                     const int32_t* new_seg_end_host, const uint8_t* new_seg_type_host,
                                     int32_t n_new_segs, void* k_cache, void* v_cache, int64_t cache_capacity,
                                     int32_t* cache_len, const int32_t* cache_len_host, void* o_new,
                                     float* lse_new, void* workspace, size_t workspace_bytes,
                                     ism_stream_t stream) {
  ism_status_t r = check_shape(shape);
  if (r != ISM_OK) return r;
  if (batch < 0 || l_new < 0) return fail(ISM_ERR_INVALID_ARG, "batch and l_new must be >= 0");
  if (batch == 0 || l_new == 0) return ISM_OK;
  if (cache_capacity <= 0 || (int64_t)batch * cache_capacity >= (int64_t(1) << 31))
    return fail(ISM_ERR_INVALID_ARG, "batch * cache_capacity must be in (0, 2^31)");
  CacheGeom cg;
  cg.cap = cache_capacity;
  cg.kv_rows = (int64_t)batch * cache_capacity;
  cg.max_keys = cache_capacity;
  cg.pages = KvPages{nullptr, 0, 0};
  return append_impl(shape, batch, q_new, k_new, v_new, l_new, new_seg_end_host, new_seg_type_host, n_new_segs,
                     k_cache, v_cache, cg, cache_len, cache_len_host, o_new, lse_new, workspace, workspace_bytes,
                     reinterpret_cast<cudaStream_t>(stream));
}

ism_status_t ism_attn_prefill_append_e4m3(const ism_attn_shape_t* shape, int32_t batch, const void* q_new,
                                          const void* k_new, const void* v_new, int32_t l_new,
                                          const int32_t* new_seg_end_host, const uint8_t* new_seg_type_host,
                                          int32_t n_new_segs, void* k_cache, void* v_cache, int64_t cache_capacity,
                                          int32_t* cache_len, const int32_t* cache_len_host, float q_descale,
                                          float k_descale, float v_descale, void* o_new, float* lse_new,
                                          void* workspace, size_t workspace_bytes, ism_stream_t stream) {
  ism_status_t r = check_shape(shape, true);
  if (r != ISM_OK) return r;
  if (shape->dtype != ISM_E4M3) return fail(ISM_ERR_INVALID_ARG, "ism_attn_prefill_append_e4m3 needs ISM_E4M3");
  if (!valid_descales(q_descale, k_descale, v_descale))
    return fail(ISM_ERR_INVALID_ARG, "descales must be positive finite numbers");
  if (!tc_available()) return fail(ISM_ERR_UNSUPPORTED, "e4m3 attention needs the sm_103 tensor cores");
  if (batch < 0 || l_new < 0) return fail(ISM_ERR_INVALID_ARG, "batch and l_new must be >= 0");
  if (batch == 0 || l_new == 0) return ISM_OK;
  if (cache_capacity <= 0 || (int64_t)batch * cache_capacity >= (int64_t(1) << 31))
    return fail(ISM_ERR_INVALID_ARG, "batch * cache_capacity must be in (0, 2^31)");
  CacheGeom cg;
  cg.cap = cache_capacity;
  cg.kv_rows = (int64_t)batch * cache_capacity;
  cg.max_keys = cache_capacity;
  cg.pages = KvPages{nullptr, 0, 0};
  return append_impl(shape, batch, q_new, k_new, v_new, l_new, new_seg_end_host, new_seg_type_host, n_new_segs,
                     k_cache, v_cache, cg, cache_len, cache_len_host, o_new, lse_new, workspace, workspace_bytes,
                     reinterpret_cast<cudaStream_t>(stream), q_descale, k_descale, v_descale);
}

ism_status_t ism_attn_prefill_append_rope(const ism_attn_shape_t* shape, int32_t batch, const void* q_new,
                                          const void* k_new, const void* v_new, int32_t l_new,
                                          const int32_t* new_seg_end_host, const uint8_t* new_seg_type_host,
                                          int32_t n_new_segs, void* k_cache, void* v_cache, int64_t cache_capacity,
                                          int32_t* cache_len, const int32_t* cache_len_host, const ism_rope_t* rope,
                                          void* o_new, float* lse_new, void* workspace, size_t workspace_bytes,
                                          ism_stream_t stream) {
  ism_status_t r = check_shape(shape);
  if (r != ISM_OK) return r;
  if (shape->dtype != ISM_BF16) return fail(ISM_ERR_INVALID_ARG, "ism_attn_prefill_append_rope needs ISM_BF16");
  if (!rope) return fail(ISM_ERR_INVALID_ARG, "rope is NULL");
  if (batch < 0 || l_new < 0) return fail(ISM_ERR_INVALID_ARG, "batch and l_new must be >= 0");
  if (batch == 0 || l_new == 0) return ISM_OK;
  if (cache_capacity <= 0 || (int64_t)batch * cache_capacity >= (int64_t(1) << 31))
    return fail(ISM_ERR_INVALID_ARG, "batch * cache_capacity must be in (0, 2^31)");
  CacheGeom cg;
  cg.cap = cache_capacity;
  cg.kv_rows = (int64_t)batch * cache_capacity;
  cg.max_keys = cache_capacity;
  cg.pages = KvPages{nullptr, 0, 0};
  return append_impl(shape, batch, q_new, k_new, v_new, l_new, new_seg_end_host, new_seg_type_host, n_new_segs,
                     k_cache, v_cache, cg, cache_len, cache_len_host, o_new, lse_new, workspace, workspace_bytes,
                     reinterpret_cast<cudaStream_t>(stream), 1.f, 1.f, 1.f, rope);
}

ism_status_t ism_attn_prefill_append_e4m3_rope(const ism_attn_shape_t* shape, int32_t batch, const void* q_new,
                                               const void* k_new, const void* v_new, int32_t l_new,
                                               const int32_t* new_seg_end_host, const uint8_t* new_seg_type_host,
                                               int32_t n_new_segs, void* k_cache, void* v_cache,
                                               int64_t cache_capacity, int32_t* cache_len,
                                               const int32_t* cache_len_host, float q_descale, float k_descale,
                                               float v_descale, const ism_rope_t* rope, void* o_new, float* lse_new,
                                               void* workspace, size_t workspace_bytes, ism_stream_t stream) {
  ism_status_t r = check_shape(shape, true);
  if (r != ISM_OK) return r;
  if (shape->dtype != ISM_E4M3) return fail(ISM_ERR_INVALID_ARG, "ism_attn_prefill_append_e4m3_rope needs ISM_E4M3");
  if (!valid_descales(q_descale, k_descale, v_descale))
    return fail(ISM_ERR_INVALID_ARG, "descales must be positive finite numbers");
  if (!rope) return fail(ISM_ERR_INVALID_ARG, "rope is NULL");
  if (!tc_available()) return fail(ISM_ERR_UNSUPPORTED, "e4m3 attention needs the sm_103 tensor cores");
  if (batch < 0 || l_new < 0) return fail(ISM_ERR_INVALID_ARG, "batch and l_new must be >= 0");
  if (batch == 0 || l_new == 0) return ISM_OK;
  if (cache_capacity <= 0 || (int64_t)batch * cache_capacity >= (int64_t(1) << 31))
    return fail(ISM_ERR_INVALID_ARG, "batch * cache_capacity must be in (0, 2^31)");
  CacheGeom cg;
  cg.cap = cache_capacity;
  cg.kv_rows = (int64_t)batch * cache_capacity;
  cg.max_keys = cache_capacity;
  cg.pages = KvPages{nullptr, 0, 0};
  return append_impl(shape, batch, q_new, k_new, v_new, l_new, new_seg_end_host, new_seg_type_host, n_new_segs,
                     k_cache, v_cache, cg, cache_len, cache_len_host, o_new, lse_new, workspace, workspace_bytes,
                     reinterpret_cast<cudaStream_t>(stream), q_descale, k_descale, v_descale, rope);
}

}  // extern "C"

namespace {

// Validates a paged cache and describes it: every page a sequence reads or
// writes in this call lies in the pool.
ism_status_t paged_geom(int32_t batch, int32_t l_new, int32_t num_pages, int32_t page_size,
                        const int32_t* block_table, const int32_t* block_table_host, int32_t max_pages,
                        const int32_t* cache_len_host, CacheGeom* cg) {
  if (page_size <= 0 || page_size % kTile != 0)
    return fail(ISM_ERR_INVALID_ARG, "page_size %d must be a positive multiple of %d", page_size, kTile);
  if (num_pages <= 0 || (int64_t)num_pages * page_size >= (int64_t(1) << 31))
    return fail(ISM_ERR_INVALID_ARG, "num_pages * page_size must be in (0, 2^31)");
  if (max_pages <= 0 || !block_table || !block_table_host || !cache_len_host)
    return fail(ISM_ERR_INVALID_ARG, "block_table (device+host), cache_len_host and max_pages > 0 are required");
  for (int b = 0; b < batch; ++b) {
    const int64_t keys = (int64_t)cache_len_host[b] + l_new;
    if (cache_len_host[b] < 0 || keys > (int64_t)max_pages * page_size)
      return fail(ISM_ERR_INVALID_ARG, "sequence %d: cache_len %d + l_new %d exceeds its %d pages", b, cache_len_host[b],
                  l_new, max_pages);
    for (int64_t i = 0; i < (keys + page_size - 1) / page_size; ++i) {
      const int32_t pg = block_table_host[(int64_t)b * max_pages + i];
      if (pg < 0 || pg >= num_pages)
        return fail(ISM_ERR_INVALID_ARG, "sequence %d: page %lld of the block table is %d, outside [0, %d)", b,
                    (long long)i, pg, num_pages);
    }
  }
  cg->cap = 0;
  cg->kv_rows = (int64_t)num_pages * page_size;
  cg->max_keys = (int64_t)max_pages * page_size;
  cg->pages = KvPages{block_table, page_size, max_pages};
  return ISM_OK;
}

}  // namespace

extern "C" {

ism_status_t ism_attn_prefill_append_paged(const ism_attn_shape_t* shape, int32_t batch, const void* q_new,
                                           const void* k_new, const void* v_new, int32_t l_new,
                                           const int32_t* new_seg_end_host, const uint8_t* new_seg_type_host,
                                           int32_t n_new_segs, void* k_pool, void* v_pool, int32_t num_pages,
                                           int32_t page_size, const int32_t* block_table,
                                           const int32_t* block_table_host, int32_t max_pages, int32_t* cache_len,
                                           const int32_t* cache_len_host, void* o_new, float* lse_new,
                                           void* workspace, size_t workspace_bytes, ism_stream_t stream) {
  ism_status_t r = check_shape(shape);
  if (r != ISM_OK) return r;
  if (batch < 0 || l_new < 0) return fail(ISM_ERR_INVALID_ARG, "batch and l_new must be >= 0");
  if (batch == 0 || l_new == 0) return ISM_OK;
  CacheGeom cg;
  if ((r = paged_geom(batch, l_new, num_pages, page_size, block_table, block_table_host, max_pages, cache_len_host,
                      &cg)) != ISM_OK)
    return r;
  return append_impl(shape, batch, q_new, k_new, v_new, l_new, new_seg_end_host, new_seg_type_host, n_new_segs,
                     k_pool, v_pool, cg, cache_len, cache_len_host, o_new, lse_new, workspace, workspace_bytes,
                     reinterpret_cast<cudaStream_t>(stream));
}

ism_status_t ism_attn_prefill_append_paged_rope(const ism_attn_shape_t* shape, int32_t batch, const void* q_new,
                                                const void* k_new, const void* v_new, int32_t l_new,
                                                const int32_t* new_seg_end_host, const uint8_t* new_seg_type_host,
                                                int32_t n_new_segs, void* k_pool, void* v_pool, int32_t num_pages,
                                                int32_t page_size, const int32_t* block_table,
                                                const int32_t* block_table_host, int32_t max_pages,
                                                int32_t* cache_len, const int32_t* cache_len_host,
                                                const ism_rope_t* rope, void* o_new, float* lse_new, void* workspace,
                                                size_t workspace_bytes, ism_stream_t stream) {
  ism_status_t r = check_shape(shape);
  if (r != ISM_OK) return r;
  if (shape->dtype != ISM_BF16)
    return fail(ISM_ERR_INVALID_ARG, "ism_attn_prefill_append_paged_rope needs ISM_BF16");
  if (!rope) return fail(ISM_ERR_INVALID_ARG, "rope is NULL");
  if (batch < 0 || l_new < 0) return fail(ISM_ERR_INVALID_ARG, "batch and l_new must be >= 0");
  if (batch == 0 || l_new == 0) return ISM_OK;
  CacheGeom cg;
  if ((r = paged_geom(batch, l_new, num_pages, page_size, block_table, block_table_host, max_pages, cache_len_host,
                      &cg)) != ISM_OK)
    return r;
  return append_impl(shape, batch, q_new, k_new, v_new, l_new, new_seg_end_host, new_seg_type_host, n_new_segs,
                     k_pool, v_pool, cg, cache_len, cache_len_host, o_new, lse_new, workspace, workspace_bytes,
                     reinterpret_cast<cudaStream_t>(stream), 1.f, 1.f, 1.f, rope);
}

// ---------------------------------------------------------------- status

ism_status_t ism_check_status(ism_stream_t stream) {
  uint32_t* status;
  ism_status_t r = status_ptr(&status);
  if (r != ISM_OK) return r;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  ISM_TRY_CUDA(cudaStreamSynchronize(st), "cudaStreamSynchronize");
  uint32_t word = 0;
  ISM_TRY_CUDA(cudaMemcpy(&word, status, sizeof(word), cudaMemcpyDeviceToHost), "status read");
  if (word) {
    uint32_t zero = 0;
    ISM_TRY_CUDA(cudaMemcpy(status, &zero, sizeof(zero), cudaMemcpyHostToDevice), "status clear");
  }
  if (word & kStatusTimeout) return fail(ISM_ERR_TIMEOUT, "a device-side wait gave up (status word 0x%x)", word);
  if (word & kStatusSmemAlign)
    return fail(ISM_ERR_CUDA, "a kernel found its shared memory misaligned and skipped its work (0x%x)", word);
  return ISM_OK;
}

ism_status_t ism_debug_mma_tile(const void* a, const void* b, float* c, int32_t mode, ism_stream_t stream) {
  if (!a || !b || !c || mode < 0 || mode > 15) return fail(ISM_ERR_INVALID_ARG, "a, b, c non-NULL and mode 0..15");
  if (!tc_available()) return fail(ISM_ERR_UNSUPPORTED, "tensor-core kernels need an sm_103 device");
  uint32_t* status;
  ism_status_t r = status_ptr(&status);
  if (r != ISM_OK) return r;
  ISM_TRY_CUDA(launch_tc_mma_tile(a, b, c, mode, status, reinterpret_cast<cudaStream_t>(stream)), "mma tile launch");
  count_launch(1);
  return ISM_OK;
}

ism_status_t ism_debug_mma_tile_e4m3(const void* a, const void* b, float* c, int32_t mode, ism_stream_t stream) {
  if (!a || !b || !c || mode < 0 || mode > 2) return fail(ISM_ERR_INVALID_ARG, "a, b, c non-NULL and mode 0..2");
  if (!tc_available()) return fail(ISM_ERR_UNSUPPORTED, "tensor-core kernels need an sm_103 device");
  uint32_t* status;
  ism_status_t r = status_ptr(&status);
  if (r != ISM_OK) return r;
  ISM_TRY_CUDA(tc::launch_mma_tile_e4m3(a, b, c, mode, status, reinterpret_cast<cudaStream_t>(stream)),
               "e4m3 mma tile launch");
  count_launch(1);
  return ISM_OK;
}

ism_status_t ism_debug_timeout_probe(uint32_t spin_limit, ism_stream_t stream) {
  uint32_t* status;
  ism_status_t r = status_ptr(&status);
  if (r != ISM_OK) return r;
  if (spin_limit == 0 || spin_limit > (1u << 20)) return fail(ISM_ERR_INVALID_ARG, "spin_limit must be in [1, 2^20]");
  ISM_TRY_CUDA(launch_timeout_probe(spin_limit, status, reinterpret_cast<cudaStream_t>(stream)), "probe launch");
  return ISM_OK;
}

}  // extern "C"
