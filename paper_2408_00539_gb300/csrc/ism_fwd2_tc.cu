// ISM attention forward, two (query head, query tile) units per CTA that
// read the same K/V (sm_103a tensor cores).
//
// When the query heads come in pairs that share a KV head (grouped-query
// attention with an even group size), one CTA computes the same 128-row
// query tile for both heads of a pair.  Otherwise (a.pair_order set) it
// computes two neighbouring query tiles of one head; the second tile sees at
// least the keys of the first, so it runs the same key blocks and possibly
// more.  Either way every K/V block is loaded once and used by both units.  The two heads' softmax warpgroups alternate with the tensor
// core (while one warpgroup turns S_A into P_A, the tensor core computes
// S_B, and so on).  P is written back into tensor memory over the S it came
// from and read there as the A operand of O += P V.
//
// Tensor memory (512 columns): S_A [0,128) O_A [128,256) S_B [256,384)
// O_B [384,512).  Shared memory: Q_A, Q_B, and a 2-stage K / V ring.
// Warps 0-3 softmax of head A, 4-7 of head B, 8 TMA producer, 9 MMA issuer, 10
// and 11 idle.
// The mask and the lazy-rescale online softmax are those of the one-head
// kernel (Eq. e_ISM with the bound of Eq. fj; full tiles unmasked).
#include <cfloat>

#include "ism_rows64.cuh"
#include "ism_tc_common.cuh"

namespace ism {
namespace tc {
namespace {

// three warpgroups: two of softmax warps, one with the producer, the MMA issuer
// and two idle warps, so that registers can move between them (setmaxnreg acts
// on whole warpgroups): 168 a thread at launch, 80 + 2 * 208 <= 3 * 168 after.
// A softmax thread holds a row of 128 scores beside its state; at 168 registers
// it spilled 88 bytes in the block loop (480 at head_dim 64).  Forward of 2 x
// 8192 grouped-query 690 -> 663 us, 4 x 4096 multi-head 453 -> 412, head_dim 64
// (16 heads, 6001 tokens) 124 -> 102, e4m3 2 x 8192 567 -> 560.
constexpr int kThreads = 384;
constexpr int kRegsService = 80, kRegsSoftmax = 208;
static_assert(kRegsService + 2 * kRegsSoftmax <= 3 * 168, "the block's registers at launch");
constexpr uint32_t kTmemCols = 512;
// Shared memory: Q_A, Q_B, K ring (2), V ring (2), barriers.  A 128 x 128 tile
// is 32 KB in bf16 (two 64-column swizzled halves) and 16 KB in e4m3 (one); a
// bf16 128 x 64 tile is one such half.
template <bool kE4M3, int kHD>
struct PairLayout {
  static constexpr uint32_t TB = kE4M3 || kHD == 64 ? kHalfBytes : kTileBytes;
  static constexpr uint32_t QA = 0, QB = TB, K = 2 * TB, V = 4 * TB, BAR = 6 * TB;
  static constexpr uint32_t SMEM = BAR + 256 + 1024;
};

constexpr int kUnitSlots = 4;  // units published ahead of the roles that follow them (kDyn)

struct Bars {
  uint64_t q_full, q_empty;
  uint64_t k_full[2], k_empty[2], v_full[2], v_empty[2];
  uint64_t s_full[2], p_half[2], p_full[2], pv_done[2];  // per head of the pair
  uint64_t final_mma;
  uint64_t unit_full[kUnitSlots], unit_read[kUnitSlots];
  int32_t units[kUnitSlots];
  uint32_t tmem_base;
  int32_t abort;
};
static_assert(sizeof(Bars) <= 256, "barrier block");

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}
__device__ __forceinline__ bool aborted(const int32_t* f) { return *reinterpret_cast<const volatile int32_t*>(f) != 0; }
__device__ __forceinline__ void set_abort(int32_t* f) { *reinterpret_cast<volatile int32_t*>(f) = 1; }

// One unit of work: two (query head, query tile) pairs that read the same
// K / V blocks, over key tiles [jb, jb + max(nkb0, nkb1)).
struct Unit {
  Tile w0, w1;
  int h0, h1, nkb0, nkb1;
  int jb;  // first key tile
  int pu;  // index of a part among all parts of the split items (-1: a whole item)
  __device__ int nkb() const { return nkb0 > nkb1 ? nkb0 : nkb1; }
};

// Item `item` of the launch: tiles and heads of its two halves.
template <bool kTilePairs>
__device__ __forceinline__ void decode_item(const AttnArgs& a, int64_t item, Unit& x) {
  if constexpr (!kTilePairs) {
    int64_t tpos;
    int hp;
    bucket_item(item, a.nq, a.hq >> 1, tpos, hp, false);  // head pairs of a tile share K / V
    x.w0 = x.w1 = a.qtiles[a.q_order[tpos]];
    x.h0 = 2 * hp;
    x.h1 = x.h0 + 1;
    x.nkb0 = x.nkb1 = x.w0.a1;
  } else {
    int64_t ppos;
    bucket_item(item, a.npairs, a.hq, ppos, x.h0, a.bucketed);
    x.h1 = x.h0;
    const int gq = a.pair_order[ppos];
    x.w0 = a.qtiles[gq];
    bool second = false;
    if (gq + 1 < a.nq) {
      x.w1 = a.qtiles[gq + 1];
      second = x.w1.q_base == x.w0.q_base && x.w1.tile == x.w0.tile + 1;
    }
    if (!second) x.w1 = x.w0;
    x.nkb0 = x.w0.a1;
    x.nkb1 = second ? x.w1.a1 : 0;
  }
}

template <bool kTilePairs, bool kSplit>
__device__ __forceinline__ Unit decode_unit(const AttnArgs& a, int64_t u) {
  Unit x;
  x.jb = 0;
  x.pu = -1;
  int64_t item = u;
  if (kSplit && u >= a.split_whole) {
    x.pu = (int)(u - a.split_whole);
    item = a.split_whole + x.pu / a.split_parts;
  }
  decode_item<kTilePairs>(a, item, x);
  if (kSplit && x.pu >= 0) {  // an equal share of the key tiles (the second tile sees at least the first's)
    const int top = x.nkb(), part = x.pu % a.split_parts;
    const int lo = top * part / a.split_parts, hi = top * (part + 1) / a.split_parts;
    x.jb = lo;
    x.nkb0 = max(min(x.nkb0, hi) - lo, 0);
    x.nkb1 = max(min(x.nkb1, hi) - lo, 0);
  }
  return x;
}

// The k-th unit of this CTA in a snake walk over the cost-ordered units
// (round r takes position b in even rounds, G - 1 - b in odd ones), so the
// CTAs' totals stay close; -1 past the end.
__device__ __forceinline__ int64_t unit_of(int64_t k, int64_t n_units) {
  const int64_t G = gridDim.x, b = blockIdx.x;
  const int64_t u = k * G + ((k & 1) ? G - 1 - b : b);
  return u < n_units ? u : -1;
}

// kE4M3: Q, K, V in e4m3 (kind::f8f6f4 MMAs, K = 32 a step); the scores are
// scaled by qk_descale, P is rounded to e4m3 for O += P V and O is scaled by
// v_descale (per-tensor dequantisation factors of the inputs).
// kSplit: the launch runs items past a.split_whole as a.split_parts key-range
// parts each; the instantiation without it is the plain kernel.
// Persistent: each CTA walks its units (unit_of) with one set of barriers
// whose phases run on across units.  The next unit's Q is loaded as soon as
// the last score MMA of the current unit has read Q, and its first score MMAs
// are issued right behind the current unit's last P V, so they overlap the
// output epilogue; the first P V of the next unit (which overwrites O) waits
// for the softmax warps' first P of that unit, which they write only after
// reading the previous O.
// kHD: head_dim 128, or 64 (bf16).  At 64, P keeps 16 mantissa bits: it goes
// back as a high and a low bf16 part (hi = bf16(p), lo = bf16(p - hi), columns
// [0, 64) and [64, 128) of S) and O += P V runs over both, because the results
// of that head size are to be those of fp32 probabilities to within the output
// rounding (measured error against 64 bits 0.0017 relative, all of it the bf16
// output's).  A block of two heads is 2 x (4 + 16) MMA steps; the tensor pipe
// still waits for the softmax warps.  One layer of 16 heads over three
// dialogues (6001 tokens): 102 us, against 44.3 ms of the CUDA-core kernel.
// kDyn: the units come from a work counter (see fwd_dynamic) instead of the
// static walk.
template <bool kTilePairs, bool kE4M3, bool kSplit, int kHD, bool kDyn>
__global__ void __launch_bounds__(kThreads, 1)
    fwd_pair_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const __grid_constant__ AttnArgs a, int64_t n_units) {
  static_assert(kHD == 128 || (kHD == 64 && !kE4M3), "head sizes of the paired forward");
  static_assert(!(kSplit && kDyn), "split launches walk statically");
  using L = PairLayout<kE4M3, kHD>;
  constexpr uint32_t kTB = L::TB;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  Bars* bar = reinterpret_cast<Bars*>(smem + L::BAR);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    ptx::mbar_init(&bar->q_full, 1);
    ptx::mbar_init(&bar->q_empty, 1);
    for (int s = 0; s < 2; ++s) {
      ptx::mbar_init(&bar->k_full[s], 1);
      ptx::mbar_init(&bar->k_empty[s], 1);
      ptx::mbar_init(&bar->v_full[s], 1);
      ptx::mbar_init(&bar->v_empty[s], 1);
      ptx::mbar_init(&bar->s_full[s], 1);
      ptx::mbar_init(&bar->p_half[s], 128);
      ptx::mbar_init(&bar->p_full[s], 128);
      ptx::mbar_init(&bar->pv_done[s], 1);
    }
    ptx::mbar_init(&bar->final_mma, 1);
    for (int s = 0; s < kUnitSlots; ++s) {
      ptx::mbar_init(&bar->unit_full[s], 1);
      ptx::mbar_init(&bar->unit_read[s], 9);  // the softmax warps and the MMA warp
    }
    bar->abort = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 9) {
    ptx::tmem_alloc(&bar->tmem_base, kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = bar->tmem_base;
  // the set-up above overlaps the kernel before (a split launch lets the merge
  // start only once every warp of every CTA is done, at the end: its blocks
  // would take issue slots and registers of the running ones)
  if constexpr (kSplit)
    pdl_sync();
  else
    pdl_wait();
  advance_cache_len(a);

  // the k-th unit of this CTA for the warps that follow the producer (-1: none left)
  auto next_unit = [&](int k) -> int64_t {
    if constexpr (!kDyn) return unit_of(k, n_units);
    const int slot = k % kUnitSlots;
    int u = -1;
    if (wait(&bar->unit_full[slot], (k / kUnitSlots) & 1, a.status))
      u = *reinterpret_cast<volatile int32_t*>(&bar->units[slot]);
    u = __reduce_min_sync(0xffffffffu, u);  // one answer for the warp (a wait may give up)
    if (lane == 0) ptx::mbar_arrive(&bar->unit_read[slot]);
    return u;
  };

  if (warp >= 8) {
    ptx::setmaxnreg_dec<kRegsService>();
    if (warp == 8) {
      // ------------------------------------------------------------ producer (the warp waits
      // converged, lane 0 issues the copies)
      // one 128 x 128 tile: two 64-column boxes in bf16, one 128-column box in e4m3
      auto load_tile = [&](uint8_t* dst, const CUtensorMap* map, uint64_t* b, int32_t x, int32_t y) {
        ptx::tma_load_2d(dst, map, b, x, y);
        if (!kE4M3 && kHD == 128) ptx::tma_load_2d(dst + kHalfBytes, map, b, x + 64, y);
      };
      if (lane == 0) {
        ptx::tma_prefetch_desc(&tmQ);
        ptx::tma_prefetch_desc(&tmK);
        ptx::tma_prefetch_desc(&tmV);
      }
      uint32_t nq = 0, it = 0;           // Q loads and K / V blocks so far (all units)
      uint32_t nk[2] = {0, 0}, nv[2] = {0, 0};
      bool ok = true;
      for (int k = 0; ok; ++k) {
        int64_t u;
        if constexpr (kDyn) {
          // the first unit is the block's, the others come from the counter
          if (k >= kUnitSlots &&
              !wait_warp(&bar->unit_read[k % kUnitSlots], (k / kUnitSlots - 1) & 1, a.status)) {
            if (lane == 0) set_abort(&bar->abort);
            ok = false;
            break;
          }
          int v = 0;
          if (lane == 0) {
            v = k == 0 ? (int)blockIdx.x : (int)gridDim.x + atomicAdd(a.work_counter, 1);
            if (v >= n_units) v = -1;
            bar->units[k % kUnitSlots] = v;
            ptx::mbar_arrive(&bar->unit_full[k % kUnitSlots]);  // release: the entry is visible to the waiters
          }
          u = __shfl_sync(0xffffffffu, v, 0);
        } else {
          u = unit_of(k, n_units);
        }
        if (u < 0) break;
        const Unit x = decode_unit<kTilePairs, kSplit>(a, u);
        const int nkb = x.nkb();
        if (nkb == 0) continue;
        const int g = x.h0 / (a.hq / a.hkv);
        const int k_first = x.jb * kRows;
        // the previous unit's score MMAs have read its Q
        if (nq > 0 && !wait_warp(&bar->q_empty, (nq - 1) & 1, a.status)) {
          if (lane == 0) set_abort(&bar->abort);
          ok = false;
          break;
        }
        if (lane == 0) {
          const int32_t qy0 = x.w0.q_base + x.w0.tile * kRows, qy1 = x.w1.q_base + x.w1.tile * kRows;
          ptx::mbar_expect_tx(&bar->q_full, (x.nkb1 > 0 ? 2 : 1) * kTB);
          load_tile(smem + L::QA, &tmQ, &bar->q_full, x.h0 * kHD, qy0);
          if (x.nkb1 > 0) load_tile(smem + L::QB, &tmQ, &bar->q_full, x.h1 * kHD, qy1);
        }
        __syncwarp();
        ++nq;
        for (int j = 0; j < nkb; ++j, ++it) {
          const int s = it & 1;
          const uint32_t n = it >> 1;
          if (__any_sync(0xffffffffu, aborted(&bar->abort))) { ok = false; break; }
          const int32_t ky = a.pages.table
                                 ? (int32_t)paged_row(a.pages, x.w0.k_base, (int64_t)k_first + j * kRows)
                                 : x.w0.k_base + k_first + j * kRows;
          if (it >= 2 && !wait_warp(&bar->k_empty[s], (n - 1) & 1, a.status)) {
            if (lane == 0) set_abort(&bar->abort);
            ok = false;
            break;
          }
          if (lane == 0) {
            ptx::mbar_expect_tx(&bar->k_full[s], kTB);
            load_tile(smem + L::K + s * kTB, &tmK, &bar->k_full[s], g * kHD, ky);
          }
          __syncwarp();
          ++nk[s];
          if (it >= 2 && !wait_warp(&bar->v_empty[s], (n - 1) & 1, a.status)) {
            if (lane == 0) set_abort(&bar->abort);
            ok = false;
            break;
          }
          if (lane == 0) {
            ptx::mbar_expect_tx(&bar->v_full[s], kTB);
            load_tile(smem + L::V + s * kTB, &tmV, &bar->v_full[s], g * kHD, ky);
          }
          __syncwarp();
          ++nv[s];
        }
      }
      if (!ok || __any_sync(0xffffffffu, aborted(&bar->abort))) {
        // let the copies in flight land before the CTA exits
        if (nq) wait_warp(&bar->q_full, (nq - 1) & 1, a.status);
        for (int s = 0; s < 2; ++s) {
          if (nk[s]) wait_warp(&bar->k_full[s], (nk[s] - 1) & 1, a.status);
          if (nv[s]) wait_warp(&bar->v_full[s], (nv[s] - 1) & 1, a.status);
        }
      }
    } else if (warp == 9) {
      // ------------------------------------------------------------ MMA issuer (the whole
      // warp runs the loop, one elected lane issues each instruction)
      constexpr uint32_t idesc_qk = kE4M3 ? ptx::idesc_e4m3_f32(128, 128, 0, 0) : ptx::idesc_bf16_f32(128, 128, 0, 0);
      constexpr uint32_t idesc_pv = kE4M3 ? ptx::idesc_e4m3_f32(128, 128, 0, 1) : ptx::idesc_bf16_f32(128, kHD, 0, 1);
      const uint32_t sQ0 = ptx::smem_u32(smem + L::QA);
      uint32_t nq = 0, it = 0;       // units with key blocks, K / V blocks (all units)
      uint32_t nb[2] = {0, 0};       // blocks of unit x so far (P hand-offs)
      // head x: Q at sQ0 + x * kTB, S at tmem + 256 x, O at tmem + 128 + 256 x
      auto issue_s = [&](int x, uint32_t blk) {
        const uint32_t sK = ptx::smem_u32(smem + L::K + (blk & 1) * kTB);
        const uint32_t sQ = sQ0 + (uint32_t)x * kTB, tS = tmem + 256u * (uint32_t)x;
        if constexpr (kE4M3)  // 128-byte rows: k-steps of 32 bytes
          ptx::mma4_e4m3_ss_warp<2, 2>(tS, desc_kmajor(sQ, 0), desc_kmajor(sK, 0), idesc_qk, 0u);
        else if constexpr (kHD == 64)
          ptx::mma4_bf16_ss_warp<2, 2>(tS, desc_kmajor(sQ, 0), desc_kmajor(sK, 0), idesc_qk, 0u);
        else
          ptx::mma8_bf16_ss_warp<ptx::KMajorSw128, ptx::KMajorSw128>(tS, desc_kmajor(sQ, 0), desc_kmajor(sK, 0),
                                                                    idesc_qk, 0u);
        ptx::mma_commit_warp(&bar->s_full[x]);
      };
      // P V in two halves of 64 keys: the first as soon as the softmax
      // warps have written P of keys [0, 64) (p_half), the second after p_full
      auto issue_pv = [&](int x, uint32_t blk, bool first) -> bool {
        const uint32_t sV = ptx::smem_u32(smem + L::V + (blk & 1) * kTB);
        const uint32_t tS = tmem + 256u * (uint32_t)x, tO = tS + 128u;
        if (!wait_warp(&bar->p_half[x], nb[x] & 1, a.status)) return false;
        ptx::tc_fence_after();
        if constexpr (kE4M3)  // P: four e4m3 a column; V MN-major, 32 rows of 128 bytes a k-step
          ptx::mma2_e4m3_ts_warp<8, 256>(tO, tS, desc_kmajor(sV, 0), idesc_pv, first ? 0u : 1u);
        else
          ptx::mma4_bf16_ts_warp<8, 128>(tO, tS, desc_mnmajor(sV, 0), idesc_pv, first ? 0u : 1u);
        if constexpr (kHD == 64)  // the low parts of P
          ptx::mma4_bf16_ts_warp<8, 128>(tO, tS + 64, desc_mnmajor(sV, 0), idesc_pv, 1u);
        if (!wait_warp(&bar->p_full[x], nb[x] & 1, a.status)) return false;
        ptx::tc_fence_after();
        if constexpr (kE4M3)
          ptx::mma2_e4m3_ts_warp<8, 256>(tO, tS + 16, desc_kmajor(sV, 0) + 512, idesc_pv, 1u);
        else  // keys [64, 128): P columns 32 + 8 kk, V rows 64 + 16 kk
          ptx::mma4_bf16_ts_warp<8, 128>(tO, tS + 32, desc_mnmajor(sV, 4), idesc_pv, 1u);
        if constexpr (kHD == 64) ptx::mma4_bf16_ts_warp<8, 128>(tO, tS + 96, desc_mnmajor(sV, 4), idesc_pv, 1u);
        ptx::mma_commit_warp(&bar->pv_done[x]);
        ++nb[x];
        return true;
      };
      bool ok = true;
      for (int k = 0; ok; ++k) {
        const int64_t u = next_unit(k);
        if (u < 0) break;
        const Unit x = decode_unit<kTilePairs, kSplit>(a, u);
        const int nkb = x.nkb();
        if (nkb == 0) continue;
        // unit y runs key blocks [0, nkb_y); the last unit reading block j
        // releases its K / V stages (unit 1 whenever it has the block: nkb1 is
        // either equal to nkb0, at least nkb0, or 0)
        auto last_user = [&](int j) { return j < x.nkb1 ? 1 : 0; };
        if (__shfl_sync(0xffffffffu, aborted(&bar->abort) ? 1 : 0, 0) ||
            !wait_warp(&bar->q_full, nq & 1, a.status) || !wait_warp(&bar->k_full[it & 1], (it >> 1) & 1, a.status)) {
          ok = false;
          break;
        }
        ++nq;
        // S of block 0 overwrites the previous unit's last P: issued after that
        // unit's last P V (in issue order; the drained variant waits for it)
        if (a.flags & kFlagDrainTmemReuse)
          for (int y = 0; ok && y < 2; ++y)
            if (nb[y] > 0 && !wait_warp(&bar->pv_done[y], (nb[y] - 1) & 1, a.status)) ok = false;
        if (!ok) break;
        ptx::tc_fence_after();
        if (x.nkb0 > 0) issue_s(0, it);
        if (x.nkb1 > 0) issue_s(1, it);
        ptx::mma_commit_warp(&bar->k_empty[it & 1]);
        if (nkb == 1) ptx::mma_commit_warp(&bar->q_empty);  // every score MMA of the unit is issued
        // Per block: PV_A(j), S_A(j+1), PV_B(j), S_B(j+1).  S_x(j+1) overwrites
        // the P_x(j) that PV_x(j) reads; MMAs issued by this thread execute in
        // order, so S_x(j+1) follows PV_x(j) without a wait (kFlagDrainTmemReuse
        // makes it wait for PV_x(j) to complete instead).
        for (int j = 0; ok && j < nkb; ++j) {
          const uint32_t blk = it + (uint32_t)j;
          const int s = blk & 1, s1 = (blk + 1) & 1;
          const bool more = j + 1 < nkb;
          if (__shfl_sync(0xffffffffu, aborted(&bar->abort) ? 1 : 0, 0)) { ok = false; break; }
          if (!wait_warp(&bar->v_full[s], (blk >> 1) & 1, a.status)) { ok = false; break; }
          if (more && !wait_warp(&bar->k_full[s1], ((blk + 1) >> 1) & 1, a.status)) { ok = false; break; }
          for (int y = 0; y < 2; ++y) {
            const int nkby = y ? x.nkb1 : x.nkb0;
            if (j >= nkby) continue;
            if (!issue_pv(y, blk, j == 0)) { ok = false; break; }
            if (y == last_user(j)) ptx::mma_commit_warp(&bar->v_empty[s]);
            if (j + 1 < nkby) {
              if ((a.flags & kFlagDrainTmemReuse) && !wait_warp(&bar->pv_done[y], (nb[y] - 1) & 1, a.status)) {
                ok = false;
                break;
              }
              ptx::tc_fence_after();
              issue_s(y, blk + 1);
              if (y == last_user(j + 1)) {
                ptx::mma_commit_warp(&bar->k_empty[s1]);
                if (j + 2 == nkb) ptx::mma_commit_warp(&bar->q_empty);  // the unit's last score MMA
              }
            }
          }
        }
        it += (uint32_t)nkb;
      }
      if (!ok && lane == 0) set_abort(&bar->abort);
      __syncwarp();
      ptx::mma_commit_warp(&bar->final_mma);
      wait_warp(&bar->final_mma, 0, a.status);
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------ softmax of head x
    ptx::setmaxnreg_inc<kRegsSoftmax>();
    const int xh = warp >> 2;
    const int r = threadIdx.x & 127;
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t tS = tmem + lane_addr + (xh ? 256u : 0u), tO = tmem + lane_addr + (xh ? 384u : 128u);
    const float sl2 = a.scale * kLog2e * (kE4M3 ? a.qk_descale : 1.f);
    uint32_t nb = 0;  // blocks of this head so far (all units)
    bool ok = true;
    for (int k = 0; ok; ++k) {
      const int64_t u = next_unit(k);
      if (u < 0) break;
      int nkbm, kfull, ke;  // key tiles and bounds counted from the unit's first key tile
      {
        const Unit x = decode_unit<kTilePairs, kSplit>(a, u);
        const Tile& wm = xh ? x.w1 : x.w0;
        nkbm = xh ? x.nkb1 : x.nkb0;
        kfull = wm.a0 - x.jb;
        ke = a.kv_end[wm.kv_base + min(wm.tile * kRows + r, wm.q_len - 1)] - x.jb * kRows;
      }
      // a part of a split item may hold no key that this row sees: its maximum
      // stays finite, so that P = 2^(-inf) = 0 and not NaN
      float m_use = kSplit ? -FLT_MAX : -INFINITY, l = 0.f;
      for (int j = 0; ok && j < nkbm; ++j) {
        const uint32_t blk = nb + (uint32_t)j;
        if (!wait(&bar->s_full[xh], blk & 1, a.status)) { ok = false; break; }
        ptx::tc_fence_after();
        float xs[128];
        {
          uint32_t t[4][32];
#pragma unroll
          for (int c = 0; c < 4; ++c) ptx::tmem_ld32(tS + c * 32, t[c]);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            ptx::reg_fence(t[c]);
#pragma unroll
            for (int i = 0; i < 32; ++i) xs[c * 32 + i] = __uint_as_float(t[c][i]);
          }
        }
        // row max on the raw scores (the scale is positive), masked keys at -inf;
        // independent partial maxima, three operands an instruction (64 of them:
        // e4m3 2 x 8192 558 -> 548 us, head_dim 64 102 -> 98, GQA 8K unchanged)
        float mr[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        if (j >= kfull) {
          const int lim = ke - j * kRows;
#pragma unroll
          for (int c = 0; c < 128; ++c) xs[c] = c < lim ? xs[c] : -INFINITY;
        }
#pragma unroll
        for (int c = 0; c < 128; c += 2) mr[(c >> 1) & 3] = max3(mr[(c >> 1) & 3], xs[c], xs[c + 1]);
        const float mraw = max3(fmaxf(mr[0], mr[1]), mr[2], mr[3]);
        const float m_new = fmaxf(m_use, mraw * sl2);
        const bool raise = m_new > m_use + 8.f;
        if (j == 0) {
          m_use = m_new;
        } else if (__any_sync(0xffffffffu, raise)) {
          // bring O (complete through PV(j-1)) and l of the rows that need it to
          // the new max.  The whole warp goes: tensor-memory loads and stores are
          // the warp's, and lanes left behind would never meet them.
          if (!__all_sync(0xffffffffu, wait(&bar->pv_done[xh], (blk - 1) & 1, a.status))) { ok = false; break; }
          ptx::tc_fence_after();
          const float f = raise ? ex2(m_use - m_new) : 1.f;
          l *= f;
#pragma unroll 1
          for (int c = 0; c < kHD / 32; ++c) {
            uint32_t o[32];
            ptx::tmem_ld32(tO + c * 32, o);
            ptx::tmem_ld_wait();
            ptx::reg_fence(o);
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
            ptx::tmem_st32(tO + c * 32, o);
          }
          if (raise) m_use = m_new;
        }
        // P over the first 64 columns of S (already read), 32 columns at a time
        float2 rsv[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        const float2 sl2x2 = make_float2(sl2, sl2), negm = make_float2(-m_use, -m_use);
        if constexpr (kE4M3) {
          // P as e4m3 over the first 32 columns of S: column c holds keys 4c .. 4c + 3,
          // handed over in halves like bf16 P (2 x 8192: 548 -> 526 us)
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            uint32_t pk[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) {
              const float* s4 = xs + 64 * hf + 4 * c;
              const float2 a01 = fma2(make_float2(s4[0], s4[1]), sl2x2, negm);
              const float2 a23 = fma2(make_float2(s4[2], s4[3]), sl2x2, negm);
              const float2 p01 = make_float2(ex2(a01.x), ex2(a01.y)), p23 = make_float2(ex2(a23.x), ex2(a23.y));
              rsv[0] = add2(rsv[0], p01);
              rsv[1] = add2(rsv[1], p23);
              pk[c] = pack_e4m3x4(p01.x, p01.y, p23.x, p23.y);
            }
            ptx::tmem_st16(tS + 16 * hf, pk);
            if (hf == 0) {  // keys [0, 64): the first half of P V may start
              ptx::tmem_st_wait();
              ptx::tc_fence_before();
              ptx::mbar_arrive(&bar->p_half[xh]);
            }
          }
        } else {
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            uint32_t pk[32], plo[kHD == 64 ? 32 : 1];
#pragma unroll
            for (int c = 0; c < 32; ++c) {
              const float2 arg = fma2(make_float2(xs[64 * hf + 2 * c], xs[64 * hf + 2 * c + 1]), sl2x2, negm);
              const float2 pr = make_float2(ex2(arg.x), ex2(arg.y));
              rsv[c & 1] = add2(rsv[c & 1], pr);
              pk[c] = pack_bf16(pr.x, pr.y);
              if constexpr (kHD == 64) plo[c] = pack_bf16_rest(pr.x, pr.y, pk[c]);
            }
            ptx::tmem_st32(tS + 32 * hf, pk);
            if constexpr (kHD == 64) ptx::tmem_st32(tS + 64 + 32 * hf, plo);
            if (hf == 0) {  // keys [0, 64): the first half of P V may start
              ptx::tmem_st_wait();
              ptx::tc_fence_before();
              ptx::mbar_arrive(&bar->p_half[xh]);
            }
          }
        }
        l += (rsv[0].x + rsv[0].y) + (rsv[1].x + rsv[1].y);
        ptx::tmem_st_wait();
        ptx::tc_fence_before();
        ptx::mbar_arrive(&bar->p_full[xh]);
      }
      if (!ok) break;
      // the unit once more for the epilogue: held across the blocks, its fields
      // would not fit the registers beside a row of scores
      const Unit x = decode_unit<kTilePairs, kSplit>(a, u);
      const int h = xh ? x.h1 : x.h0;
      const Tile wm = xh ? x.w1 : x.w0;
      const int row = wm.tile * kRows + r;
      const bool valid = row < wm.q_len;
      if (nkbm > 0) {
        nb += (uint32_t)nkbm;
        // one decision for the whole warp: the epilogue's loads and shuffles are warp-wide
        if (!__all_sync(0xffffffffu, wait(&bar->pv_done[xh], (nb - 1) & 1, a.status))) { ok = false; break; }
        ptx::tc_fence_after();
      }
      if (kSplit && x.pu >= 0) {
        // part of a split item: unnormalised O and (max, sum) for the merge; a
        // part without key tiles leaves max -inf (weight 0, its O is not read)
        const int64_t pu = ((int64_t)x.pu * 2 + xh) * a.part_rows + (valid ? r : 0);
        if (valid) {
          a.part_ml[pu * 2] = nkbm > 0 ? m_use : -INFINITY;
          a.part_ml[pu * 2 + 1] = nkbm > 0 ? l : 0.f;
        }
        if (nkbm > 0) {
          const float f = kE4M3 ? a.v_descale : 1.f;
          float4* dst = reinterpret_cast<float4*>(a.part_o + pu * kHD);
          float bad = 0.f;
#pragma unroll 1
          for (int c = 0; c < kHD / 32; ++c) {
            uint32_t o[32];
            ptx::tmem_ld32(tO + c * 32, o);
            ptx::tmem_ld_wait();
            ptx::reg_fence(o);
            if constexpr (kHD == 64)
#pragma unroll
              for (int i = 0; i < 32; ++i) bad = rows64::not_finite(o[i], bad);
            if (valid)
#pragma unroll
              for (int i = 0; i < 8; ++i)
                dst[c * 8 + i] = make_float4(__uint_as_float(o[4 * i]) * f, __uint_as_float(o[4 * i + 1]) * f,
                                             __uint_as_float(o[4 * i + 2]) * f, __uint_as_float(o[4 * i + 3]) * f);
          }
          if constexpr (kHD == 64) {
            uint32_t rows = __ballot_sync(0xffffffffu, valid && bad != 0.f);
            for (; rows; rows &= rows - 1) {
              const int t = __ffs(rows) - 1;
              const int k1 = min(__shfl_sync(0xffffffffu, ke, t), nkbm * kRows), k0 = x.jb * kRows;
              const float2 acc = rows64::out_row(a, wm.q_base + row - lane + t, wm.k_base, h, k0, k0 + k1,
                                                 __shfl_sync(0xffffffffu, m_use, t));
              float* p = a.part_o + __shfl_sync(0xffffffffu, pu, t) * kHD + lane;
              p[0] = acc.x;
              p[32] = acc.y;
            }
          }
        }
      } else if (nkbm > 0) {
        const float inv = (kE4M3 ? a.v_descale : 1.f) / l;
        const int64_t orow = (int64_t)wm.q_base + row;
        // rows are stored by groups of four lanes (store_slice32)
        const int li = r & 3;
        const int64_t rstride = (int64_t)a.hq * kHD;
        __nv_bfloat16* const g0 = reinterpret_cast<__nv_bfloat16*>(a.out) + (orow - li) * rstride + h * kHD;
        float bad = 0.f;
#pragma unroll 1
        for (int c = 0; c < kHD / 32; ++c) {
          uint32_t o[32], w[16];
          ptx::tmem_ld32(tO + c * 32, o);
          ptx::tmem_ld_wait();
          ptx::reg_fence(o);
          if constexpr (kHD == 64)
#pragma unroll
            for (int i = 0; i < 32; ++i) bad = rows64::not_finite(o[i], bad);
          pack_scaled32(o, inv, w);
          store_slice32(w, g0 + 32 * c, rstride, wm.q_len - (row - li));
        }
        if constexpr (kHD == 64) {
          uint32_t rows = __ballot_sync(0xffffffffu, valid && bad != 0.f);
          if (rows) __syncwarp();  // (a row's first store may be another lane's)
          for (; rows; rows &= rows - 1) {
            const int t = __ffs(rows) - 1;
            const int32_t q_row = (int32_t)orow - lane + t;
            const float f = __shfl_sync(0xffffffffu, inv, t);
            const float2 acc = rows64::out_row(a, q_row, wm.k_base, h, 0, __shfl_sync(0xffffffffu, ke, t),
                                               __shfl_sync(0xffffffffu, m_use, t));
            rows64::store_row(static_cast<__nv_bfloat16*>(a.out) + (int64_t)q_row * rstride + h * kHD,
                              make_float2(acc.x * f, acc.y * f));
          }
        }
        if (valid && a.lse) a.lse[(int64_t)h * a.q_rows + orow] = (m_use + log2f(l)) * kLn2;
      }
    }
    if (!ok) set_abort(&bar->abort);
  }
  ptx::tc_fence_before();
  __syncthreads();
  if constexpr (kSplit) pdl_trigger();  // (the first warp to do so speaks for the CTA)
  if (warp == 9) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, kTmemCols);
  }
}

// Merge of the parts of each split item: a warp per (split item, half x, row),
// lanes first over the parts, then over the dimensions.  m in the base-2
// scaled units of the forward, so O = sum_p w_p O_p / sum_p w_p l_p with
// w_p = 2^(m_p - M), and LSE = (M + log2 L) ln 2, as the whole-item epilogue
// writes them.  Bound by reading the partials once; with a block of 128
// threads a row and two scalar loads a thread it took 12.3 us on two halves of
// the 8 x 16K prefill's last 56 items, 8.6 us now.
constexpr int kMaxParts = 32;
template <bool kTilePairs, int kHD>
__global__ void __launch_bounds__(128) fwd_split_merge_kernel(const AttnArgs a) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int r = (int)(i % a.part_rows), x = (int)((i / a.part_rows) & 1);
  const int64_t k = i / (2 * (int64_t)a.part_rows);
  if (k >= a.split_items) return;
  Unit un;
  decode_item<kTilePairs>(a, a.split_whole + k, un);
  if ((x ? un.nkb1 : un.nkb0) == 0) return;  // a tile pair without its second tile
  const Tile w = x ? un.w1 : un.w0;
  const int h = x ? un.h1 : un.h0;
  const int row = w.tile * kRows + r;
  if (row >= w.q_len) return;
  const int parts = a.split_parts;
  const int64_t stride = 2 * (int64_t)a.part_rows;                        // partial rows from part to part
  const int64_t p0 = (k * parts * 2 + x) * (int64_t)a.part_rows + r;      // part 0's
  float m = -INFINITY, l = 0.f;
  if (lane < parts) {
    const float2 ml = *reinterpret_cast<const float2*>(a.part_ml + (p0 + lane * stride) * 2);
    m = ml.x;
    l = ml.y;
  }
  float M = m;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  const float f = m == -INFINITY ? 0.f : exp2f(m - M);
  float L = f * l;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
  constexpr int kPer = kHD / 32;  // dimensions a lane
  float acc[kPer] = {};
#pragma unroll 4
  for (int p = 0; p < parts; ++p) {
    const float fp = __shfl_sync(0xffffffffu, f, p);
    if (fp == 0.f) continue;  // no key tile: O not written
    const float* src = a.part_o + (p0 + p * stride) * kHD + lane * kPer;
#pragma unroll
    for (int d = 0; d < kPer; ++d) acc[d] = fmaf(fp, src[d], acc[d]);
  }
  const int64_t orow = (int64_t)w.q_base + row;
  __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(a.out) + (orow * a.hq + h) * kHD + lane * kPer;
#pragma unroll
  for (int d = 0; d < kPer; d += 2)
    *reinterpret_cast<__nv_bfloat162*>(out + d) = __floats2bfloat162_rn(acc[d] / L, acc[d + 1] / L);
  if (lane == 0 && a.lse) a.lse[(int64_t)h * a.q_rows + orow] = (M + log2f(L)) * kLn2;
}

template <bool kE4M3, int kHD, bool kTilePairs>
cudaError_t launch_fwd_pair_t(const AttnArgs& a, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                              cudaStream_t st) {
  cudaError_t e;
  const bool split = a.split_items > 0;
  // e4m3 tile pairs always have a counter (they take no plan)
  constexpr bool kNeedsCounter = kTilePairs && kE4M3;
  auto kern = split ? fwd_pair_kernel<kTilePairs, kE4M3, true, kHD, false>
              : a.work_counter ? fwd_pair_kernel<kTilePairs, kE4M3, false, kHD, true>
                               : fwd_pair_kernel<kTilePairs, kE4M3, false, kHD, kNeedsCounter>;
  constexpr uint32_t smem = PairLayout<kE4M3, kHD>::SMEM;
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
    return e;
  const int64_t items = kTilePairs ? a.npairs * a.hq : a.nq * (a.hq / 2);
  if (items == 0) return cudaSuccess;
  if (split && (a.split_whole + a.split_items != items || !a.part_o || !a.part_ml || a.split_parts < 1 ||
                a.split_parts > kMaxParts))
    return cudaErrorInvalidValue;
  const int64_t n_units = split ? a.split_whole + a.split_parts * a.split_items : items;
  if (!split && (a.work_counter ? n_units >= (int64_t(1) << 30) : kNeedsCounter)) return cudaErrorInvalidValue;
  // persistent: one CTA per SM walks its share of the units
  const int64_t grid = n_units < sm_count() ? n_units : sm_count();
  if ((e = launch(split || a.dependent, kern, grid, kThreads, smem, st, tq, tk, tv, a, n_units)) != cudaSuccess ||
      !split)
    return e;
  const int64_t rows = a.split_items * 2 * a.part_rows;
  return launch(true, fwd_split_merge_kernel<kTilePairs, kHD>, (rows + 3) / 4, 128, 0, st, a);
}

}  // namespace

cudaError_t launch_fwd_pair(const AttnArgs& a, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                            cudaStream_t st) {
  if (a.pair_order)
    return a.dtype == ISM_E4M3 ? launch_fwd_pair_t<true, 128, true>(a, tq, tk, tv, st)
           : a.d == 64         ? launch_fwd_pair_t<false, 64, true>(a, tq, tk, tv, st)
                               : launch_fwd_pair_t<false, 128, true>(a, tq, tk, tv, st);
  return a.dtype == ISM_E4M3 ? launch_fwd_pair_t<true, 128, false>(a, tq, tk, tv, st)
         : a.d == 64         ? launch_fwd_pair_t<false, 64, false>(a, tq, tk, tv, st)
                             : launch_fwd_pair_t<false, 128, false>(a, tq, tk, tv, st);
}

}  // namespace tc
}  // namespace ism
