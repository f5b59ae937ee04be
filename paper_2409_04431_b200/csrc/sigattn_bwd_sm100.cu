// bf16 backward of sigmoid attention for sm_100a (Algorithm 2 of Appendix F.1, redesigned
// for Blackwell).  Per (batch*head, 128-key tile j) work item, looping over query tiles i:
//
//     S^T  = K_j Q_i^T                      (tensor memory region A, fp32)
//     P^T  = sigmoid(scale S^T + b ...)     (registers -> bf16 over region A)
//     dV_j += P^T dO_i                      (A operand from tensor memory)
//     dP^T = V_j dO_i^T                     (region B)
//     dS^T = P^T (1 - P^T) dP^T             (registers -> bf16, over region B and in shared memory)
//     dK_j += dS^T Q_i                      (A operand from tensor memory)
//     dQ_i  = dS K_j                        (region B again, then fp32 reduce-add to HBM)
//
// Everything is kept transposed (keys on the 128 TMEM lanes, queries along columns) so
// that P^T and dS^T can feed the dV and dK products straight from tensor memory; only dQ
// needs dS with queries as rows, and reads the shared-memory copy as an MN-major A operand.
// No row statistic of any kind is read or written: dS is a point-wise function of S and
// dP (Section 4 / Appendix F.1), and P is recomputed from Q and K alone.
//
// dK_j and dV_j stay in tensor memory across the whole query loop.  dQ_i is complete only
// after all key tiles have contributed, so each CTA adds its fp32 partial tile into a
// [B, H, N, D] fp32 workspace with TMA reduce-add; the workspace is zeroed before and
// converted to bf16 (times scale) after the main kernel: the two helper steps that
// survive from the paper's backward.  scale is also folded into dK's epilogue.
//
// Warp roles (see BwdRoles): activation groups of four warps (every thread owns one key row and a share of the
// tile's query columns), at D = 128 a dQ drain group, a TMA producer, an MMA issuer.
#include <atomic>

#include "launch.h"
#include "sigattn_internal.h"
#include "sigattn_activation.cuh"
#include "sm100_primitives.cuh"
#include "tensor_map.h"
#include "../../include/sigattn.h"

namespace sigattn {
namespace {

using namespace sm100;

constexpr int kT = 128;  // tile edge: keys per item (TMEM lanes) and queries per step

// Warp roles.  Narrow: two activation groups of four warps (64 query columns a thread) and a drain group.  Wide
// (D = 64): four activation groups (32 query columns a thread) that also drain dQ, and a thread that issues its adds.
// Four warps per scheduler instead of two cover the latency of the activation and feed the exponentials evenly where
// the warps take different paths; but 512 threads wait, drain and arrive where 256 and 128 did.  The launcher
// chooses (see there).  The 512 activation threads have 96 registers each: room for 32 columns and no more.
template <int D, bool WIDE>
struct BwdRoles {
  static_assert(D == 64 || !WIDE, "at D = 128 the step is bound by the products and the drain");
  static constexpr bool kDrainGroup = !WIDE;
  static constexpr int kGroups = WIDE ? 4 : 2;                 // activation groups
  static constexpr int kCols = kT / kGroups;                   // query columns of a thread
  static constexpr int kActThreads = 128 * kGroups;
  static constexpr int kDrainThreads = kDrainGroup ? 128 : kActThreads;
  static constexpr int kLoadWarp = 4 * kGroups + (kDrainGroup ? 4 : 0);
  static constexpr int kMmaWarp = kLoadWarp + 1;
  static constexpr int kThreads = 32 * (kMmaWarp + (kDrainGroup ? 1 : 2));
  static constexpr int kItemReaders = 1 + kActThreads + (kDrainGroup ? 128 : 1);   // threads that take every work item
  // first packed column of k-step ks (16 queries = 8 columns): a group packs its bf16 values over the first half
  // of its own columns
  __device__ static __forceinline__ uint32_t packed_col(int ks) {
    return (ks / (kCols / 16)) * kCols + (ks % (kCols / 16)) * 8;
  }
};
constexpr float kLog2eB = 1.4426950408889634f;

template <int D>
struct BwdSmem {
  static constexpr int kPanels = D / 64;
  static constexpr int kPanelBytes = kT * 128;
  static constexpr int kTileBytes = kPanels * kPanelBytes;  // a K, V, Q or dO tile
  // K, V buffers: at D = 64 two, so that the next item's first products do not wait for this item's results to be
  // stored (dV is staged in the V buffer, dK in the K buffer).  At D = 128 one; dK is staged where dS was, so that the
  // next K can be loaded as soon as the last dQ has read this one.
  static constexpr int kKvStages = (D == 64) ? 2 : 1;
  static constexpr int kKOff = 0;
  static constexpr int kVOff = kTileBytes;
  static constexpr int kKvBytes = 2 * kTileBytes;
  // Q stages: two at D = 128 (shared memory is full); three at D = 64, where S^T runs two steps ahead
  // (four, which would make stage and phase a mask and a shift, measured no faster)
  static constexpr int kQStages = (D == 64) ? 3 : 2;
  static constexpr int kQOff = kKvStages * kKvBytes;
  // dO stages.  With one stage the next tile's load starts when dV(i) has read this one, and dP^T(i+1) waits for it:
  // 700 to 1800 of a step's 3860 cycles at D = 64 (clock trace).  Three stages there; D = 128 has no room for more.
  static constexpr int kDoStages = (D == 64) ? 3 : 1;
  static constexpr int kDoOff = (2 * kKvStages + kQStages) * kTileBytes;
  static constexpr int kDsOff = (2 * kKvStages + kQStages + kDoStages) * kTileBytes;   // dS^T, 128 x 128 bf16 = two panels
  static constexpr int kDqOff = kDsOff + 2 * kPanelBytes;   // two fp32 staging boxes of 128 x 32
  static constexpr int kTotal = kDqOff + 2 * kPanelBytes;
  static constexpr int kDynBytes = kTotal + 1024;
};

struct BwdItem {
  int bh;       // (batch, key/value head) index: K_j, V_j, dK_j, dV_j
  int bh_q0;    // first of the `group` query heads that read this key/value head
  int j, i_begin;
  int n;        // query tiles per query head
  int steps;    // group * n, visited head by head; 0: no item is left
  int n_valid;  // rows of this sequence that count (N unless the batch is padded)
};

struct BwdBarriers {
  uint64_t k_full[2], v_full[2], k_empty[2], v_empty[2];
  uint64_t q_full[3], q_empty[3];
  uint64_t do_full[3], do_empty[3];
  // s_full, p_ready, dq_full, dq_empty: one per region of tensor memory that holds S^T / P^T (see BwdTmem);
  // a region's barriers flip once per use of that region
  uint64_t s_full[2], dp_full;
  uint64_t p_ready[2], ds_ready;
  uint64_t dq_full[2], dq_empty[2];
  uint64_t dv_full, dkv_full, dkv_empty;
  uint64_t ds_free;   // D = 128: dK has been stored from where dS goes
  uint64_t stage_full, stage_empty;   // wide: the dQ staging boxes between the activation groups and the storing thread
  // the TMA thread finds the next work item and hands it to the other roles through this two-slot ring
  uint64_t sched_full[2], sched_empty[2], sched_answer;
  BwdItem sched_item[2];
  __align__(16) uint32_t sched_response[4];
};

struct BwdParams {
  int BH, H, N;    // BH counts (batch, key/value head) pairs: the work items are per key/value head
  int H_kv, group; // heads of K, V and query heads per key/value head (H = H_kv * group)
  int n_tiles;    // query tiles: ceil(N / 128), N = rows of Q
  int n_tiles_k;  // key tiles: ceil(rows of K / 128)
  int pos0;       // position of query row 0 relative to key row 0 (see FwdParams of the forward)
  const int* seqlens;   // padded batch: valid length per batch entry (keys and queries), or nullptr
  // batch stored without padding (B = 1): sequence s owns rows [cu_seqlens[s], cu_seqlens[s + 1]);
  // bias_vec and dbias then hold one entry per (sequence, head)
  const int* cu_seqlens;
  int n_seqs;
  int dynamic;     // 1: work items are drawn, one thread block of the grid per item (see BwdSchedule)
  // Few (batch, key/value head) pairs (multi-query attention at a small batch): the query heads of a
  // group are split over n_sub work items of heads_per_sub heads each, which add their dK_j, dV_j
  // (bf16 TMA reduce-adds into the cleared outputs) instead of storing them.  n_sub = 1: off.
  int n_sub, heads_per_sub;
  // Few work items with one query head per key/value head (one long sequence, few heads): the query
  // tiles of a key tile are divided over two items (i_split = 2) that add their dK_j, dV_j likewise.
  int i_split;
  int dkv_add;   // 1: dK_j, dV_j are added (bf16 TMA reduce-adds) into outputs the caller cleared: several calls sum up
  int n_items;
  int head_group;  // (batch, key/value head) pairs whose items are handed out together
  float scale, scale_log2e, bias_log2e;
  const float* bias_vec;   // one bias per (batch, head) instead of the scalar, or nullptr
  float* dbias;            // receives sum dS per (batch, head), or nullptr
  const float* slopes;
  int* status;
};

// Ranks are ordered by decreasing cost; rounds alternate direction over the CTAs so that
// expensive and cheap items pair up (static stand-in for longest-first scheduling).
__device__ __forceinline__ int bwd_snake_rank(int round, int n_items) {
  const int g = gridDim.x;
  const int c = (round & 1) ? (g - 1 - static_cast<int>(blockIdx.x)) : static_cast<int>(blockIdx.x);
  const int rank = round * g + c;
  return rank < n_items ? rank : -1;
}

__device__ __forceinline__ int bwd_num_rounds(int n_items) { return (n_items + gridDim.x - 1) / gridDim.x; }

// Which item comes next.  Where the static order above does not sort by cost (batches without padding, where the cost
// follows the position of the key tile inside its own sequence, and heads handed out in groups) the items are drawn: the
// grid has one thread block per item; those that start take over the others in order (cluster launch control, as in the
// forward).  One thread per block, which has issued an item's last loads some steps before it ends, finds the
// next (an answer takes about 2200 cycles), decodes it and passes it on through the ring: the divisions and searches of
// decoding cost the other roles, above all the thread that issues the products, 600 to 1400 cycles between two items.
struct BwdSchedule {
  int turn, item, requests;
};
__device__ __forceinline__ void bwd_first_item(const BwdParams& p, BwdSchedule* s) {
  s->turn = 0;
  s->requests = 0;
  s->item = p.dynamic ? static_cast<int>(blockIdx.x) : bwd_snake_rank(0, p.n_items);
}
// The next one (s->item < 0: none is left).  false: a bounded wait expired.
__device__ __forceinline__ bool bwd_following_item(const BwdParams& p, BwdBarriers* bars, BwdSchedule* s, volatile int* cta_err) {
  if (p.dynamic) {
    mbar_arrive_expect_tx(smem_u32(&bars->sched_answer), 16);
    clc_try_cancel(smem_u32(bars->sched_response), smem_u32(&bars->sched_answer));
    if (!mbar_wait(smem_u32(&bars->sched_answer), s->requests & 1, cta_err, 76)) return false;
    ++s->requests;
    s->item = clc_block(smem_u32(bars->sched_response));
    fence_proxy_async_smem();   // the answer has been read before the next one is written there
    return true;
  }
  s->item = -1;
  const int rounds = bwd_num_rounds(p.n_items);
  while (s->item < 0 && ++s->turn < rounds) s->item = bwd_snake_rank(s->turn, p.n_items);
  return true;
}
// The ring: `number` counts the items of this thread block.
__device__ __forceinline__ bool bwd_hand_item(BwdBarriers* bars, uint32_t number, const BwdItem& w, volatile int* cta_err) {
  const uint32_t slot = number & 1, phase = (number >> 1) & 1;
  if (!mbar_wait(smem_u32(&bars->sched_empty[slot]), phase ^ 1, cta_err, 70)) return false;
  bars->sched_item[slot] = w;
  mbar_arrive(smem_u32(&bars->sched_full[slot]));
  return true;
}
// 1 when the slot holds an item, 0 when none is left, -1 when a bounded wait expired.  The activation threads keep the
// slot until the item is done and read its fields there, also at each step: their registers are full.  With the item
// copied (seven values, and a row's sequence, in every thread) the general instantiations at D = 64 spilled 32 to 56 bytes.
__device__ __forceinline__ int bwd_see_item(BwdBarriers* bars, uint32_t number, volatile int* cta_err) {
  const uint32_t slot = number & 1, phase = (number >> 1) & 1;
  if (!mbar_wait(smem_u32(&bars->sched_full[slot]), phase, cta_err, 71)) return -1;
  return bars->sched_item[slot].steps > 0 ? 1 : 0;
}
__device__ __forceinline__ void bwd_return_item(BwdBarriers* bars, uint32_t number) {
  mbar_arrive(smem_u32(&bars->sched_empty[number & 1]));
}
__device__ __forceinline__ int bwd_take_item(BwdBarriers* bars, uint32_t number, BwdItem* w, volatile int* cta_err) {
  const int more = bwd_see_item(bars, number, cta_err);
  if (more < 0) return more;
  *w = bars->sched_item[number & 1];
  bwd_return_item(bars, number);
  return more;
}

// GROUPED = false compiles the plain case (one query head per key/value head, no padded batch)
// without the head loop and without the per-sequence lengths; it is the benchmarked path.
// GROUPED = true serves grouped heads, padded batches and batches stored without padding.
// Sequence that owns `row` in a batch stored without padding: the largest s with cu[s] <= row.
__device__ __forceinline__ int bwd_seq_of_row(const int* __restrict__ cu, int n_seqs, int row) {
  int lo = 0, hi = n_seqs;   // cu[lo] <= row < cu[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(cu + mid) <= row) lo = mid; else hi = mid;
  }
  return lo;
}

template <bool CAUSAL, bool GROUPED>
__device__ __forceinline__ BwdItem decode_bwd_item(const BwdParams& p, int item) {
  BwdItem w;
  // Items are numbered group of heads by group of heads (see the launcher; one group = all heads), within a group by
  // ascending key tile = descending work when causal, then head, then part.
  const int parts = GROUPED ? (p.n_sub > 1 ? p.n_sub : p.i_split) : 1;
  int g0 = 0, r = item, per_tile = p.BH * parts;
  if (p.head_group < p.BH) {
    const int per_group = p.head_group * p.n_tiles_k * parts, gr = item / per_group;
    g0 = gr * p.head_group;
    r -= gr * per_group;
    per_tile = min(p.head_group, p.BH - g0) * parts;
  }
  w.j = r / per_tile;
  r -= w.j * per_tile;
  int of_parts = 0;
  if (GROUPED && parts > 1) {
    of_parts = r % parts;
    r /= parts;
  }
  w.bh = g0 + r;
  const int sub = (GROUPED && p.n_sub > 1) ? of_parts : 0;     // part of the query heads of a key/value head
  const int part = (GROUPED && p.i_split > 1) ? of_parts : 0;  // half of the query tiles
  w.bh_q0 = GROUPED ? (w.bh / p.H_kv) * p.H + (w.bh % p.H_kv) * p.group + sub * p.heads_per_sub : w.bh;
  // causal: the first query tile whose last row, at position 128 i + 127 + pos0, reaches key 128 j
  // padded batch: query tiles past the sequence's end are not visited at all
  const bool padded = GROUPED && p.seqlens != nullptr;
  w.n_valid = padded ? max(0, min(p.N, __ldg(p.seqlens + w.bh / p.H_kv))) : p.N;
  const int n_tiles_q = padded ? max(1, (w.n_valid + kT - 1) / kT) : p.n_tiles;
  // (a key tile that lies after every query still visits the last query tile, fully masked: zeros)
  w.i_begin = CAUSAL ? min(n_tiles_q - 1, max(0, (w.j * kT - p.pos0) / kT)) : 0;
  // a key tile wholly past the sequence's end needs one (fully masked) query tile to write its zeros
  if (padded && w.j * kT >= w.n_valid) w.i_begin = n_tiles_q - 1;
  w.n = n_tiles_q - w.i_begin;
  if (GROUPED && p.cu_seqlens != nullptr) {
    // batch without padding: the queries that see this key tile run from the start of its first
    // key's sequence (causal: from the first key itself) to the end of its last key's sequence
    const int k_first = w.j * kT, k_last = min(p.N, k_first + kT) - 1;
    const int q_lo = CAUSAL ? k_first : __ldg(p.cu_seqlens + bwd_seq_of_row(p.cu_seqlens, p.n_seqs, k_first));
    const int q_hi = __ldg(p.cu_seqlens + bwd_seq_of_row(p.cu_seqlens, p.n_seqs, k_last) + 1);
    // (offsets that do not rise from 0 to N give wrong results, but the clamps keep every loop bounded)
    w.i_begin = max(0, min(p.n_tiles - 1, q_lo / kT));
    w.n = max(1, min(p.n_tiles, (q_hi + kT - 1) / kT) - w.i_begin);
  }
  if (GROUPED && p.i_split > 1) {
    const int first_half = (w.n + 1) / 2;
    if (part == 0) {
      w.n = first_half;
    } else if (w.n > first_half) {
      w.i_begin += first_half;
      w.n -= first_half;
    } else {
      // a single query tile cannot be divided (the last key tile of a causal call): the second item
      // visits the query tile before it, which the mask blanks completely, and adds zeros
      w.i_begin = max(0, w.i_begin - 1);
      w.n = 1;
    }
  }
  w.steps = GROUPED ? p.heads_per_sub * w.n : w.n;
  return w;
}

// TMEM column map (fp32 columns).
// D = 128: region A = S^T / P^T, region B = dP^T / dS^T / dQ, then dV and dK: 4 x 128 columns, tensor memory
// is full.  S^T(i+1) has to wait for dV(i), which reads P^T(i) from A, and dP^T(i+1) for the drain of dQ(i).
// D = 64: dV and dK take 64 columns each and 128 are left over.  They make a second region A: steps
// alternate between A0 and A1, S^T runs two steps ahead of the activation, and dQ(i) is written over the
// first 64 columns of the step's own region A (its P^T has been consumed by dV(i), which the same thread
// issued earlier) so that region B is free for dP^T(i+1) at once.  S^T(i+2) waits for the drain of dQ(i).
template <int D>
struct BwdTmem {
  static constexpr bool kTwoA = (D == 64);
  static constexpr uint32_t kB = 128;
  static constexpr uint32_t kDv = 256;
  static constexpr uint32_t kDk = 256 + D;
  // region A of (global) step `step`, its index, and how often that region has been used before
  __device__ static __forceinline__ uint32_t a_col(uint32_t step) { return (kTwoA && (step & 1)) ? 384u : 0u; }
  __device__ static __forceinline__ uint32_t r_index(uint32_t step) { return kTwoA ? (step & 1) : 0u; }
  __device__ static __forceinline__ uint32_t r_use(uint32_t step) { return kTwoA ? (step >> 1) : step; }
  // where dQ of that step is accumulated
  __device__ static __forceinline__ uint32_t dq_col(uint32_t step) { return kTwoA ? a_col(step) : kB; }
};

// ------------------------------------------------------------------ producer

template <int D, bool CAUSAL, bool GROUPED>
__device__ void bwd_load_role(const BwdParams& p, const CUtensorMap* tmQ, const CUtensorMap* tmK,
                              const CUtensorMap* tmV, const CUtensorMap* tmDo, uint32_t smem_base,
                              BwdBarriers* bars, volatile int* cta_err) {
  using L = BwdSmem<D>;
  uint32_t q_cnt = 0, do_cnt = 0, item_cnt = 0;
  auto load_tile = [&](const CUtensorMap* tm, uint32_t dst, uint32_t bar, int row, int bh) {
#pragma unroll
    for (int pn = 0; pn < L::kPanels; ++pn) tma_load_3d(dst + pn * L::kPanelBytes, tm, bar, pn * 64, row, bh);
  };
  auto load_q = [&](int i, int bh) -> bool {
    const uint32_t st = q_cnt % L::kQStages, ph = (q_cnt / L::kQStages) & 1;
    if (!mbar_wait(smem_u32(&bars->q_empty[st]), ph ^ 1, cta_err, 40)) return false;
    const uint32_t bar = smem_u32(&bars->q_full[st]);
    mbar_arrive_expect_tx(bar, L::kTileBytes);
    load_tile(tmQ, smem_base + L::kQOff + st * L::kTileBytes, bar, i * kT, bh);
    ++q_cnt;
    return true;
  };
  auto load_do = [&](int i, int bh) -> bool {
    const uint32_t st = do_cnt % L::kDoStages, ph = (do_cnt / L::kDoStages) & 1;
    if (!mbar_wait(smem_u32(&bars->do_empty[st]), ph ^ 1, cta_err, 41)) return false;
    const uint32_t bar = smem_u32(&bars->do_full[st]);
    mbar_arrive_expect_tx(bar, L::kTileBytes);
    load_tile(tmDo, smem_base + L::kDoOff + st * L::kTileBytes, bar, i * kT, bh);
    ++do_cnt;
    return true;
  };
  BwdSchedule sched;
  bwd_first_item(p, &sched);
  for (uint32_t number = 0;; ++number) {
    BwdItem w;
    w.steps = 0;
    if (sched.item >= 0) w = decode_bwd_item<CAUSAL, GROUPED>(p, sched.item);
    if (!bwd_hand_item(bars, number, w, cta_err)) return;
    if (sched.item < 0) break;
    auto load_kv = [&]() -> bool {
      const uint32_t st = item_cnt % L::kKvStages, ph = (item_cnt / L::kKvStages) & 1, dst = smem_base + st * L::kKvBytes;
      if (!mbar_wait(smem_u32(&bars->k_empty[st]), ph ^ 1, cta_err, 42)) return false;
      mbar_arrive_expect_tx(smem_u32(&bars->k_full[st]), L::kTileBytes);
      load_tile(tmK, dst + L::kKOff, smem_u32(&bars->k_full[st]), w.j * kT, w.bh);
      if (!mbar_wait(smem_u32(&bars->v_empty[st]), ph ^ 1, cta_err, 43)) return false;
      mbar_arrive_expect_tx(smem_u32(&bars->v_full[st]), L::kTileBytes);
      load_tile(tmV, dst + L::kVOff, smem_u32(&bars->v_full[st]), w.j * kT, w.bh);
      ++item_cnt;
      return true;
    };
    // They can only be loaded when the item before is done: at least from L2 then (D = 128, whole backward, us, without /
    // with: 120 documents in 16384 rows 244 / 240, B4 H16 N1024 causal ALiBi 80.4 / 79.5; longer items the same).
    if (L::kKvStages == 1) {
#pragma unroll
      for (int pn = 0; pn < L::kPanels; ++pn) {
        tma_prefetch_3d(tmK, pn * 64, w.j * kT, w.bh);
        tma_prefetch_3d(tmV, pn * 64, w.j * kT, w.bh);
      }
    }
    // With one K, V buffer the first Q and dO tiles can be loaded earlier than K and V, with two later.
    if (L::kKvStages > 1 && !load_kv()) return;
    if (!load_q(w.i_begin, w.bh_q0)) return;
    if (!load_do(w.i_begin, w.bh_q0)) return;
    if (L::kKvStages == 1 && !load_kv()) return;
    // The remaining steps, head by head.  With two regions A (D = 64) S^T runs a step further ahead than
    // dP^T, so Q stays one tile ahead of dO: dO(s) can only be loaded after dV(s-1), and S^T(s+1) is issued
    // before that product's inputs exist.
    constexpr int lead = BwdTmem<D>::kTwoA ? 1 : 0;
    auto load_step = [&](int s, bool is_q) -> bool {
      const int g = GROUPED ? s / w.n : 0;
      const int i = w.i_begin + (s - g * w.n), bh = w.bh_q0 + g;
      return is_q ? load_q(i, bh) : load_do(i, bh);
    };
    for (int q_next = 1, do_next = 1; do_next < w.steps; ++do_next) {
      for (; q_next < w.steps && q_next <= do_next + lead; ++q_next)
        if (!load_step(q_next, true)) return;
      if (!load_step(do_next, false)) return;
    }
    // (asked for only now: with the request at the item's start the answer costs nothing, but items go to blocks that are
    // far from ready for them: B4 H32 H_kv8 N2048 D128 causal 468 -> 563 us, 16 documents in 16384 rows 508 -> 555)
    if (!bwd_following_item(p, bars, &sched, cta_err)) return;
  }
}

// ------------------------------------------------------------------ MMA issuer

// Run by one thread that elect.sync chose: with a test of the thread index instead the compiler does not know that
// a single thread is active, and every product costs the thread more.  Measured, whole backward, us:
// B8 H12 N4096 D64 1540 -> 1385, B8 H16 N2048 D64 causal ALiBi 353 -> 331, B2 H16 N4096 D128 causal 389 -> 387.
// (The role run by the whole warp with an election per batch of products: 1405, 339, 392.)
template <int D, bool WIDE>
__device__ void bwd_mma_role(uint32_t smem_base, uint32_t tmem, BwdBarriers* bars,
                             volatile int* cta_err) {
  using L = BwdSmem<D>;
  using TM = BwdTmem<D>;
  constexpr uint32_t kIdescSt = make_idesc_bf16(kT, kT, 0, 0);   // S^T, dP^T : K-major x K-major
  constexpr uint32_t kIdescAcc = make_idesc_bf16(kT, D, 0, 1);   // dV, dK   : (TMEM | K-major) x MN-major
  constexpr uint32_t kIdescDq = make_idesc_bf16(kT, D, 1, 1);    // dQ       : MN-major x MN-major
  const uint32_t sK = smem_base + L::kKOff, sV = smem_base + L::kVOff, sDo = smem_base + L::kDoOff,
                 sDs = smem_base + L::kDsOff;
  uint32_t q_cnt = 0, do_cnt = 0, item_cnt = 0, step_cnt = 0;

  // [128 x 128] = X[128 x D] * Y[128 x D]^T, both K-major
  auto issue_kk = [&](uint32_t d_col, uint64_t x_desc, uint64_t y_desc) {
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
      const uint32_t off = (ks >> 2) * L::kPanelBytes + (ks & 3) * 32;
      umma_ss(tmem + d_col, desc_advance(x_desc, off), desc_advance(y_desc, off), kIdescSt, ks > 0);
    }
  };
  // Descriptors are built once; each k-step only advances the start address.
  const uint64_t dK_k0 = make_smem_desc_sw128(sK, 16, 1024);                // K_j, K-major (S^T)
  const uint64_t dV_k0 = make_smem_desc_sw128(sV, 16, 1024);                // V_j, K-major (dP^T)
  const uint64_t dDo_k0 = make_smem_desc_sw128(sDo, 16, 1024);               // dO_i, K-major (dP^T)
  const uint64_t dDo_mn0 = make_smem_desc_sw128(sDo, L::kPanelBytes, 1024);  // dO_i, MN-major (dV)
  const uint64_t dK_mn0 = make_smem_desc_sw128(sK, L::kPanelBytes, 1024);   // K_j, MN-major (dQ)
  const uint64_t dDs_mn = make_smem_desc_sw128(sDs, L::kPanelBytes, 1024);  // dS^T, MN-major (dQ)
  // Stage 0 of Q; the other stages are reached by advancing the start address (an array indexed by the
  // stage at run time would live in local memory, and this thread pays for every load in full)
  const uint64_t dQ_k0 = make_smem_desc_sw128(smem_base + L::kQOff, 16, 1024);                 // Q_i, K-major (S^T)
  const uint64_t dQ_mn0 = make_smem_desc_sw128(smem_base + L::kQOff, L::kPanelBytes, 1024);    // Q_i, MN-major (dK)
  auto q_stage = [](uint32_t cnt) -> uint32_t { return cnt % L::kQStages; };
  auto q_phase = [](uint32_t cnt) -> uint32_t { return (cnt / L::kQStages) & 1; };
  auto do_stage = [](uint32_t cnt) -> uint32_t { return cnt % L::kDoStages; };
  auto do_phase = [](uint32_t cnt) -> uint32_t { return (cnt / L::kDoStages) & 1; };
  auto kv_off = [&]() -> uint32_t { return (item_cnt % L::kKvStages) * L::kKvBytes; };   // this item's buffer
  // S^T of global step `step` from the Q tile with running number `qn`.  D = 64: the step's region A last
  // held dQ of two steps earlier, which the drain group must have read.
  auto issue_s = [&](uint32_t step, uint32_t qn, int where) -> bool {
    if (!mbar_wait(smem_u32(&bars->q_full[q_stage(qn)]), q_phase(qn), cta_err, where)) return false;
    if (TM::kTwoA &&
        !mbar_wait(smem_u32(&bars->dq_empty[TM::r_index(step)]), (TM::r_use(step) & 1) ^ 1, cta_err, where + 20))
      return false;
    tc_fence_after_sync();
    issue_kk(TM::a_col(step), desc_advance(dK_k0, kv_off()), desc_advance(dQ_k0, q_stage(qn) * L::kTileBytes));
    umma_commit(smem_u32(&bars->s_full[TM::r_index(step)]));
    return true;
  };
  // dP^T of global step `step`.  D = 128: region B last held dQ of the step before.
  auto issue_dp = [&](uint32_t step, int where) -> bool {
    if (!mbar_wait(smem_u32(&bars->do_full[do_stage(do_cnt)]), do_phase(do_cnt), cta_err, where)) return false;
    if (!TM::kTwoA &&
        !mbar_wait(smem_u32(&bars->dq_empty[0]), (step & 1) ^ 1, cta_err, where + 20))
      return false;
    tc_fence_after_sync();
    issue_kk(TM::kB, desc_advance(dV_k0, kv_off()), desc_advance(dDo_k0, do_stage(do_cnt) * L::kTileBytes));
    umma_commit(smem_u32(&bars->dp_full));
    return true;
  };

  BwdItem w;
  if (bwd_take_item(bars, 0, &w, cta_err) < 0) return;
  int next_steps = w.steps;
  while (next_steps > 0) {
    const int steps = next_steps;
    const uint64_t dK_mn = desc_advance(dK_mn0, kv_off());

    // prologue: S^T(0), dP^T(0) and, with two regions A, S^T(1)
    const uint32_t kv_stage = item_cnt % L::kKvStages, kv_phase = (item_cnt / L::kKvStages) & 1;
    if (!mbar_wait(smem_u32(&bars->k_full[kv_stage]), kv_phase, cta_err, 50)) return;
    if (!issue_s(step_cnt, q_cnt, 51)) return;
    if (!mbar_wait(smem_u32(&bars->v_full[kv_stage]), kv_phase, cta_err, 49)) return;
    if (!issue_dp(step_cnt, 52)) return;
    if (TM::kTwoA && steps > 1 && !issue_s(step_cnt + 1, q_cnt + 1, 53)) return;

    for (int it = 0; it < steps; ++it) {
      const uint32_t st = q_stage(q_cnt), reg = TM::r_index(step_cnt);
      // dV += P^T dO_i
      if (!mbar_wait(smem_u32(&bars->p_ready[reg]), TM::r_use(step_cnt) & 1, cta_err, 54)) return;
      if (it == 0 && !mbar_wait(smem_u32(&bars->dkv_empty), (item_cnt & 1) ^ 1, cta_err, 55)) return;
      tc_fence_after_sync();
      const uint64_t dDo_mn = desc_advance(dDo_mn0, do_stage(do_cnt) * L::kTileBytes);
#pragma unroll
      for (int ks = 0; ks < kT / 16; ++ks) {
        umma_ts(tmem + TM::kDv, tmem + TM::a_col(step_cnt) + BwdRoles<D, WIDE>::packed_col(ks),
                desc_advance(dDo_mn, ks * 2048), kIdescAcc, (it > 0 || ks > 0));
      }
      umma_commit(smem_u32(&bars->do_empty[do_stage(do_cnt)]));
      ++do_cnt;
      // one region A: S^T of the next query tile goes where P^T was
      if (!TM::kTwoA && it + 1 < steps && !issue_s(step_cnt + 1, q_cnt + 1, 56)) return;
      if (it + 1 == steps) {
        umma_commit(smem_u32(&bars->dv_full));
        if (bwd_take_item(bars, item_cnt + 1, &w, cta_err) < 0) return;
        next_steps = w.steps;
      }
      // dK += dS^T Q_i with dS^T read from region B of tensor memory (the activation groups
      // leave a bf16 copy there, over the dP^T columns they have consumed), then dQ_i = dS K_j,
      // which overwrites region B (D = 128) or the head of the step's region A (D = 64): MMAs of
      // one thread execute in issue order.
      if (!mbar_wait(smem_u32(&bars->ds_ready), step_cnt & 1, cta_err, 57)) return;
      tc_fence_after_sync();
      const uint64_t q_mn = desc_advance(dQ_mn0, st * L::kTileBytes);
#pragma unroll
      for (int ks = 0; ks < kT / 16; ++ks) {
        umma_ts(tmem + TM::kDk, tmem + TM::kB + BwdRoles<D, WIDE>::packed_col(ks), desc_advance(q_mn, ks * 2048),
                kIdescAcc, (it > 0 || ks > 0));
      }
#pragma unroll
      for (int ks = 0; ks < kT / 16; ++ks) {
        umma_ss(tmem + TM::dq_col(step_cnt), desc_advance(dDs_mn, ks * 2048), desc_advance(dK_mn, ks * 2048),
                kIdescDq, ks > 0);
      }
      umma_commit(smem_u32(&bars->dq_full[reg]));
      umma_commit(smem_u32(&bars->q_empty[st]));
      // dP^T of the next query tile, then (two regions A) S^T of the one after it
      if (it + 1 < steps && !issue_dp(step_cnt + 1, 58)) return;
      if (TM::kTwoA && it + 2 < steps && !issue_s(step_cnt + 2, q_cnt + 2, 59)) return;
      ++q_cnt;
      ++step_cnt;
    }
    // (the commit that the epilogue waits for comes last: after a block's last item nothing waits for k_empty, and no
    // arrival may be on its way when the block ends)
    if (L::kKvStages == 1) umma_commit(smem_u32(&bars->k_empty[0]));
    umma_commit(smem_u32(&bars->dkv_full));
    ++item_cnt;
  }
}

// ------------------------------------------------------------------ activation groups

// Group `wg`'s columns of one row of a [128 x D] fp32 accumulator -> bf16 (times `mul`) -> swizzled staging tile.
template <int D, bool WIDE>
__device__ __forceinline__ void bwd_store_acc_rows(uint32_t t_acc, uint8_t* stage, int tid, float mul, int wg) {
  using L = BwdSmem<D>;
  constexpr int kShare = D / BwdRoles<D, WIDE>::kGroups, kRun = kShare < 32 ? kShare : 32;   // columns, at a time
#pragma unroll 1
  for (int c = wg * kShare; c < (wg + 1) * kShare; c += kRun) {
    uint32_t o[kRun];
    if constexpr (kRun == 32) tmem_ld32(t_acc + c, o); else tmem_ld16(t_acc + c, o);
    tmem_wait_ld();
    uint8_t* panel = stage + (c >> 6) * L::kPanelBytes + tid * 128;
#pragma unroll
    for (int g = 0; g < kRun / 8; ++g) {
      uint4 val;
      val.x = pack_bf16x2(mul * __uint_as_float(o[8 * g + 0]), mul * __uint_as_float(o[8 * g + 1]));
      val.y = pack_bf16x2(mul * __uint_as_float(o[8 * g + 2]), mul * __uint_as_float(o[8 * g + 3]));
      val.z = pack_bf16x2(mul * __uint_as_float(o[8 * g + 4]), mul * __uint_as_float(o[8 * g + 5]));
      val.w = pack_bf16x2(mul * __uint_as_float(o[8 * g + 6]), mul * __uint_as_float(o[8 * g + 7]));
      *reinterpret_cast<uint4*>(panel + (((((c & 63) >> 3) + g) ^ (tid & 7)) * 16)) = val;
    }
  }
}

// What a thread's key row needs to know about the item's query head g.  Batch without padding: the queries [q_lo, q_hi)
// that see the key (its own sequence, from the key itself on when causal), and the sequence's bias.
struct BwdRow {
  float slope_log2e, bias_log2e;
  int q_lo, q_hi;
};
template <bool CAUSAL, bool ALIBI, bool RAGGED>
__device__ __forceinline__ BwdRow bwd_row(const BwdParams& p, const BwdItem& w, int tid, int g) {
  const int key = w.j * kT + tid, bh_q = w.bh_q0 + g;
  BwdRow r;
  r.slope_log2e = ALIBI ? __ldg(p.slopes + bh_q % p.H) * kLog2eB : 0.0f;
  r.bias_log2e = p.bias_log2e;
  r.q_lo = r.q_hi = 0;
  if (!RAGGED) {
    if (p.bias_vec) r.bias_log2e = __ldg(p.bias_vec + bh_q) * kLog2eB;
  } else if (key < p.N) {
    const int seq = bwd_seq_of_row(p.cu_seqlens, p.n_seqs, key);
    r.q_lo = CAUSAL ? key : __ldg(p.cu_seqlens + seq);
    r.q_hi = __ldg(p.cu_seqlens + seq + 1);
    if (p.bias_vec) r.bias_log2e = __ldg(p.bias_vec + seq * p.H + bh_q) * kLog2eB;
  }
  return r;
}

// KIND: 0 plain, 1 general (grouped heads, padded batch), 2 general plus a batch stored without padding
template <int D, bool CAUSAL, bool ALIBI, bool DBIAS, int KIND, bool WIDE>
__device__ void bwd_act_role(const BwdParams& p, const CUtensorMap* tmDk, const CUtensorMap* tmDv,
                             int wg, uint8_t* smem, uint32_t smem_base, uint32_t tmem, BwdBarriers* bars,
                             volatile int* cta_err) {
  using L = BwdSmem<D>;
  using TM = BwdTmem<D>;
  using R = BwdRoles<D, WIDE>;
  constexpr bool GROUPED = KIND >= 1;
  constexpr int kCols = R::kCols;
  const int tid = threadIdx.x & 127;  // key row within the tile
  const uint32_t lane_off = static_cast<uint32_t>(((threadIdx.x >> 5) & 3) * 32) << 16;
  uint32_t step_cnt = 0, item_cnt = 0;

  // Without a drain group: the dQ tile of global step `step`, 16 of its 64 columns per group, to the two staging
  // boxes, from where one thread of another warp adds it to the fp32 accumulator (with barriers among the 512 threads
  // instead a drain cost 1000 of a step's 3520 cycles).  Done after the P phase of the following step, by when the
  // products have completed it.
  auto drain = [&](uint32_t step) -> bool {
    const uint32_t reg = TM::r_index(step);
    if (!mbar_wait(smem_u32(&bars->dq_full[reg]), TM::r_use(step) & 1, cta_err, 70 + wg)) return false;
    tc_fence_after_sync();
    uint32_t o[16];
    tmem_ld16(tmem + TM::dq_col(step) + lane_off + wg * 16, o);
    tmem_wait_ld();
    tc_fence_before_sync();
    mbar_arrive(smem_u32(&bars->dq_empty[reg]));
    if (!mbar_wait(smem_u32(&bars->stage_empty), (step & 1) ^ 1, cta_err, 74)) return false;
    const uint32_t box = smem_base + L::kDqOff + (wg >> 1) * L::kPanelBytes + tid * 128;
#pragma unroll
    for (int e = 0; e < 4; ++e) st_shared_v4(box + ((((wg & 1) * 4 + e) ^ (tid & 7)) * 16), o + 4 * e);
    fence_proxy_async_smem();
    mbar_arrive(smem_u32(&bars->stage_full));
    return true;
  };

  constexpr bool ragged = (KIND == 2);
  auto item = [&]() -> const BwdItem& { return bars->sched_item[item_cnt & 1]; };
  bool release = false;   // the results that this thread stored may not have left their staging tile yet
  int more = bwd_see_item(bars, 0, cta_err);
  if (more < 0) return;
  BwdRow row;
  if (more) row = bwd_row<CAUSAL, ALIBI, ragged>(p, item(), tid, 0);
  while (more) {
    for (int g = 0; g < (GROUPED ? p.heads_per_sub : 1); ++g) {   // the query heads that read this key/value head
    if (g > 0) row = bwd_row<CAUSAL, ALIBI, ragged>(p, item(), tid, g);
    const float slope_log2e = row.slope_log2e, bias_log2e = row.bias_log2e;
    const int q_lo = row.q_lo, q_hi = row.q_hi;
    float ds_sum = 0.0f;   // this thread's share of sum dS over the head's tiles (the bias gradient)

    const int i_first = item().i_begin, i_end = i_first + item().n;
    for (int i = i_first; i < i_end; ++i) {
      const BwdItem& w = item();
      // this thread's key index minus the position of the tile's first query
      const float col_rel = static_cast<float>((w.j - i) * kT + tid - p.pos0);
      // the mask cuts through the tile unless even its first query sits at or after the last key:
      // the first tile of the loop, and with pos0 not a multiple of 128 also the second
      bool diag = CAUSAL && (i * kT + p.pos0 < w.j * kT + kT - 1);
      // queries [mask_lo, mask_hi) of the tile keep their weight for this thread's key
      float mask_lo = CAUSAL ? col_rel : -1.0f, mask_hi = 1.0e9f;
      if (GROUPED && p.seqlens != nullptr) {
        mask_hi = static_cast<float>(w.n_valid - i * kT);
        if (w.j * kT + tid >= w.n_valid) mask_hi = -1.0f;   // a key past the end: the whole row
        diag = diag || (w.j + 1) * kT > w.n_valid || (i + 1) * kT > w.n_valid;
      }
      if (ragged) {
        mask_lo = static_cast<float>(q_lo - i * kT);
        mask_hi = static_cast<float>(q_hi - i * kT);
        // the tile is not wholly inside the queries of some key of this warp (decided by the warp: threads that
        // disagree would run the masked and the plain evaluation one after the other, 5200 cycles instead of 2200)
        diag = __any_sync(0xffffffffu, i * kT < q_lo || (i + 1) * kT > q_hi);
      }
      float pp[kCols / 32][32];
      if (!mbar_wait(smem_u32(&bars->s_full[TM::r_index(step_cnt)]), TM::r_use(step_cnt) & 1, cta_err, 60 + wg))
        return;
      tc_fence_after_sync();
#pragma unroll
      for (int c = 0; c < kCols / 32; ++c) {
        const int gc = wg * (kCols / 32) + c;  // 32-query chunk of the tile
        uint32_t s[32], pk[16];
        tmem_ld32(tmem + TM::a_col(step_cnt) + lane_off + gc * 32, s);
        tmem_wait_ld();
        float(&ppc)[32] = pp[c];
        if (GROUPED && diag)
          bwd_sigmoid_chunk<2, ALIBI, CAUSAL, ragged>(s, pk, ppc, p.scale_log2e, bias_log2e, slope_log2e, col_rel, gc * 32,
                                                      mask_lo, mask_hi);
        else if (CAUSAL && diag)
          bwd_sigmoid_chunk<1, ALIBI, CAUSAL, ragged>(s, pk, ppc, p.scale_log2e, bias_log2e, slope_log2e, col_rel, gc * 32,
                                                      col_rel, 0.0f);
        else
          bwd_sigmoid_chunk<0, ALIBI, CAUSAL, ragged>(s, pk, ppc, p.scale_log2e, bias_log2e, slope_log2e, col_rel, gc * 32,
                                                      0.0f, 0.0f);
        tmem_st16(tmem + TM::a_col(step_cnt) + lane_off + wg * kCols + c * 16, pk);
      }
      tmem_wait_st();
      tc_fence_before_sync();
      mbar_arrive(smem_u32(&bars->p_ready[TM::r_index(step_cnt)]));
      if (release) {   // (one thread a result)
        tma_wait_group_read<0>();
        const uint32_t st = (item_cnt - 1) % L::kKvStages;
        mbar_arrive(smem_u32(wg == 0 ? &bars->v_empty[st] : L::kKvStages == 1 ? &bars->ds_free : &bars->k_empty[st]));
        release = false;
      }
      if constexpr (!R::kDrainGroup) {
        if ((g > 0 || i > i_first) && !drain(step_cnt - 1)) return;
      }

      // dS^T = P (1 - P) dP^T -> bf16 -> shared memory [key][query], 128-byte swizzle
      if (!mbar_wait(smem_u32(&bars->dp_full), step_cnt & 1, cta_err, 62 + wg)) return;
      if (L::kKvStages == 1 && g == 0 && i == i_first &&
          !mbar_wait(smem_u32(&bars->ds_free), (item_cnt & 1) ^ 1, cta_err, 68))
        return;
      tc_fence_after_sync();
      const uint32_t ds_row = smem_base + L::kDsOff + (wg * kCols >> 6) * L::kPanelBytes + tid * 128;
#pragma unroll
      for (int c = 0; c < kCols / 16; ++c) {  // 16 queries at a time
        uint32_t dp[16];
        tmem_ld16(tmem + TM::kB + lane_off + wg * kCols + c * 16, dp);
        tmem_wait_ld();
        uint32_t ds[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float* f = pp[c >> 1] + (c & 1) * 16 + 2 * e;
          const float ds0 = f[0] * __uint_as_float(dp[2 * e]), ds1 = f[1] * __uint_as_float(dp[2 * e + 1]);
          if (DBIAS) ds_sum += ds0 + ds1;
          ds[e] = pack_bf16x2(ds0, ds1);
        }
        // one copy to shared memory (A operand of dQ, MN-major) ...
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const int chunk = ((wg * kCols & 63) >> 3) + c * 2 + g;
          st_shared_v4(ds_row + ((chunk ^ (tid & 7)) * 16), ds + 4 * g);
        }
        // ... and one to tensor memory (A operand of dK), over dP^T columns already consumed
        tmem_st8(tmem + TM::kB + lane_off + wg * kCols + c * 8, ds);
      }
      tmem_wait_st();
      tc_fence_before_sync();   // the dP^T reads above precede the dQ MMA that overwrites region B
      fence_proxy_async_smem();
      mbar_arrive(smem_u32(&bars->ds_ready));
      ++step_cnt;
    }

    const int bh_q = DBIAS ? item().bh_q0 + g : 0;
    if (DBIAS && ragged) {   // keys of one warp may belong to different sequences: one atomic per key
      if (q_hi > q_lo)
        atomicAdd(p.dbias + bwd_seq_of_row(p.cu_seqlens, p.n_seqs, item().j * kT + tid) * p.H + bh_q, ds_sum);
    } else if (DBIAS) {   // sum over the warp, one atomic per warp, item and query head
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) ds_sum += __shfl_xor_sync(0xffffffffu, ds_sum, off);
      if ((threadIdx.x & 31) == 0) atomicAdd(p.dbias + bh_q, ds_sum);
    }
    }   // query heads

    // Epilogue.  While the last dK and dQ are computed, the next item is looked up and dV, complete before them, is
    // converted and stored from the V buffer; then scale * dK, from the K buffer (D = 128: from where dS was).  The
    // buffers go back once the stores have read them: with two of them after the next P phase, by when they have.
    // Waited for at once, with both results converted after the last product and the next item looked up then, the
    // threads stood 5000 to 6000 cycles between two items (clock traces).  Whole backward, us, that way / this way (both
    // with the polls of all waits unrolled, see mbar_wait_limit):
    // B16 H12 N577 D64 94.5 / 90.3, B16 H16 N512 D64 causal 82.9 / 79.0, B16 H8 padded N1500 D64 225.7 / 216.9,
    // 60 documents in 16384 rows D64 223 / 208.5, B4 H16 N1024 D128 causal ALiBi 87.8 / 80.0,
    // B2 H16 N4096 D128 causal 428 / 418.
    const int done_row = item().j * kT, done_bh = item().bh;
    const uint32_t done = item_cnt & 1, kv_stage = item_cnt % L::kKvStages;
    bwd_return_item(bars, item_cnt);
    ++item_cnt;
    more = bwd_see_item(bars, item_cnt, cta_err);
    if (more < 0) return;
    if (more) row = bwd_row<CAUSAL, ALIBI, ragged>(p, item(), tid, 0);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const bool is_dv = r == 0;
      if (!mbar_wait(smem_u32(is_dv ? &bars->dv_full : &bars->dkv_full), done, cta_err, is_dv ? 66 : 64)) return;
      tc_fence_after_sync();
      uint8_t* stage = smem + (is_dv ? kv_stage * L::kKvBytes + L::kVOff
                                     : L::kKvStages == 1 ? L::kDsOff : kv_stage * L::kKvBytes + L::kKOff);
      bwd_store_acc_rows<D, WIDE>(tmem + (is_dv ? TM::kDv : TM::kDk) + lane_off, stage, tid, is_dv ? 1.0f : p.scale, wg);
      if (!is_dv) {
        tc_fence_before_sync();
        mbar_arrive(smem_u32(&bars->dkv_empty));
      }
      fence_proxy_async_smem();
      named_barrier_sync<1, R::kActThreads>();
      if (tid == 0 && wg == r) {
        const CUtensorMap* tm = is_dv ? tmDv : tmDk;
#pragma unroll
        for (int pn = 0; pn < L::kPanels; ++pn)
          if (GROUPED && (p.n_sub > 1 || p.i_split > 1 || p.dkv_add))   // the parts (or successive calls) add their shares
            tma_reduce_add_3d(tm, smem_u32(stage + pn * L::kPanelBytes), pn * 64, done_row, done_bh);
          else
            tma_store_3d(tm, smem_u32(stage + pn * L::kPanelBytes), pn * 64, done_row, done_bh);
        tma_commit_group();
        release = true;
      }
      if constexpr (!R::kDrainGroup) {
        if (is_dv && !drain(step_cnt - 1)) return;
      }
    }
    if (L::kKvStages == 1 && tid == 0 && wg == 0) {   // the next V is waited for
      tma_wait_group_read<0>();
      mbar_arrive(smem_u32(&bars->v_empty[0]));
      release = false;
    }
  }
  if (tid == 0) tma_wait_group<0>();
}

// ------------------------------------------------------------------ dQ drain group

template <int D, bool GROUPED>
__device__ void bwd_drain_role(const BwdParams& p, const CUtensorMap* tmW, uint8_t* smem, uint32_t tmem,
                               BwdBarriers* bars, volatile int* cta_err) {
  using L = BwdSmem<D>;
  using TM = BwdTmem<D>;
  const int tid = threadIdx.x & 127;  // query row within the tile
  const uint32_t lane_off = static_cast<uint32_t>(((threadIdx.x >> 5) & 3) * 32) << 16;
  uint32_t step_cnt = 0;
  for (uint32_t number = 0;; ++number) {
    BwdItem w;
    if (bwd_take_item(bars, number, &w, cta_err) <= 0) break;
    for (int s = 0; s < w.steps; ++s) {
      const int g = GROUPED ? s / w.n : 0, it = s - g * w.n;   // query head within the group, query tile
      const int row0 = (w.i_begin + it) * kT, bh_q = w.bh_q0 + g;
      const uint32_t reg = TM::r_index(step_cnt), dq_col = TM::dq_col(step_cnt);
      if (!mbar_wait(smem_u32(&bars->dq_full[reg]), TM::r_use(step_cnt) & 1, cta_err, 70)) return;
      ++step_cnt;
      tc_fence_after_sync();
      // 64 columns per round: both staging boxes are filled from registers, so region B is
      // released right after the last TMEM read instead of after the last reduce-add.
#pragma unroll 1
      for (int r = 0; r < D / 64; ++r) {
        uint32_t o0[32], o1[32];
        tmem_ld32(tmem + dq_col + lane_off + r * 64, o0);
        tmem_ld32(tmem + dq_col + lane_off + r * 64 + 32, o1);
        tmem_wait_ld();
        if (r == D / 64 - 1) {
          tc_fence_before_sync();
          mbar_arrive(smem_u32(&bars->dq_empty[reg]));
        }
        // both staging boxes must have been read by the reduce-adds issued earlier
        if (tid == 0) tma_wait_group_read<0>();
        named_barrier_sync<3, 128>();
        uint8_t* row0p = smem + L::kDqOff + tid * 128;
        uint8_t* row1p = row0p + L::kPanelBytes;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          *reinterpret_cast<uint4*>(row0p + ((g ^ (tid & 7)) * 16)) =
              make_uint4(o0[4 * g + 0], o0[4 * g + 1], o0[4 * g + 2], o0[4 * g + 3]);
          *reinterpret_cast<uint4*>(row1p + ((g ^ (tid & 7)) * 16)) =
              make_uint4(o1[4 * g + 0], o1[4 * g + 1], o1[4 * g + 2], o1[4 * g + 3]);
        }
        fence_proxy_async_smem();
        named_barrier_sync<3, 128>();
        if (tid == 0) {
          tma_reduce_add_3d(tmW, smem_u32(smem + L::kDqOff), r * 64, row0, bh_q);
          tma_reduce_add_3d(tmW, smem_u32(smem + L::kDqOff + L::kPanelBytes), r * 64 + 32, row0, bh_q);
          tma_commit_group();
        }
      }
    }
  }
  if (tid == 0) tma_wait_group<0>();
}

// Wide: one thread adds the staged dQ tiles to the fp32 accumulator.
template <int D>
__device__ void bwd_store_role(const BwdParams& p, const CUtensorMap* tmW, uint32_t smem_base, BwdBarriers* bars,
                               volatile int* cta_err) {
  using L = BwdSmem<D>;
  uint32_t step_cnt = 0;
  for (uint32_t number = 0;; ++number) {
    BwdItem w;
    if (bwd_take_item(bars, number, &w, cta_err) <= 0) break;
    int it = 0, bh_q = w.bh_q0;
    for (int s = 0; s < w.steps; ++s, ++step_cnt) {
      if (!mbar_wait(smem_u32(&bars->stage_full), step_cnt & 1, cta_err, 75)) return;
      tma_reduce_add_3d(tmW, smem_base + L::kDqOff, 0, (w.i_begin + it) * kT, bh_q);
      tma_reduce_add_3d(tmW, smem_base + L::kDqOff + L::kPanelBytes, 32, (w.i_begin + it) * kT, bh_q);
      tma_commit_group();
      tma_wait_group_read<0>();
      mbar_arrive(smem_u32(&bars->stage_empty));
      if (++it == w.n) {   // the next query head of the group
        it = 0;
        ++bh_q;
      }
    }
  }
  tma_wait_group<0>();
}

// ------------------------------------------------------------------ kernels

template <int D, bool CAUSAL, bool ALIBI, bool DBIAS, int KIND, bool WIDE>
__global__ void __launch_bounds__(BwdRoles<D, WIDE>::kThreads, 1)
sigattn_bwd_bf16_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmDo,
                        const __grid_constant__ CUtensorMap tmDk, const __grid_constant__ CUtensorMap tmDv,
                        const __grid_constant__ CUtensorMap tmW, const BwdParams p) {
  using R = BwdRoles<D, WIDE>;
  constexpr bool GROUPED = KIND >= 1;
  extern __shared__ uint8_t smem_raw[];
  __shared__ BwdBarriers bars;
  __shared__ uint32_t tmem_base_slot;
  __shared__ int cta_err;

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem_base = smem_u32(smem);
  const int warp = threadIdx.x >> 5;

  if (threadIdx.x == 0) {
    cta_err = 0;
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&bars.k_full[s]), 1);
      mbar_init(smem_u32(&bars.v_full[s]), 1);
      mbar_init(smem_u32(&bars.k_empty[s]), 1);
      mbar_init(smem_u32(&bars.v_empty[s]), 1);
    }
    for (int s = 0; s < 3; ++s) {
      mbar_init(smem_u32(&bars.q_full[s]), 1);
      mbar_init(smem_u32(&bars.q_empty[s]), 1);
      mbar_init(smem_u32(&bars.do_full[s]), 1);
      mbar_init(smem_u32(&bars.do_empty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&bars.s_full[s]), 1);
      mbar_init(smem_u32(&bars.p_ready[s]), R::kActThreads);
      mbar_init(smem_u32(&bars.dq_full[s]), 1);
      mbar_init(smem_u32(&bars.dq_empty[s]), R::kDrainThreads);
    }
    mbar_init(smem_u32(&bars.dp_full), 1);
    mbar_init(smem_u32(&bars.ds_ready), R::kActThreads);
    mbar_init(smem_u32(&bars.dv_full), 1);
    mbar_init(smem_u32(&bars.dkv_full), 1);
    mbar_init(smem_u32(&bars.ds_free), 1);
    mbar_init(smem_u32(&bars.stage_full), R::kActThreads);
    mbar_init(smem_u32(&bars.stage_empty), 1);
    mbar_init(smem_u32(&bars.dkv_empty), R::kActThreads);
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&bars.sched_full[s]), 1);
      mbar_init(smem_u32(&bars.sched_empty[s]), BwdRoles<D, WIDE>::kItemReaders);
    }
    mbar_init(smem_u32(&bars.sched_answer), 1);
    fence_mbar_init();
  }
  if (warp == R::kLoadWarp && elect_one()) {
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
    tma_prefetch_desc(&tmDo);
    tma_prefetch_desc(&tmDk);
    tma_prefetch_desc(&tmDv);
    tma_prefetch_desc(&tmW);
  }
  if (warp == R::kMmaWarp) {
    tmem_alloc(smem_u32(&tmem_base_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_base_slot;
  grid_dependency_wait();
  grid_dependency_trigger();

  if (warp == R::kLoadWarp) {
    if ((threadIdx.x & 31) == 0) bwd_load_role<D, CAUSAL, GROUPED>(p, &tmQ, &tmK, &tmV, &tmDo, smem_base, &bars, &cta_err);
    __syncwarp();
  } else if (warp == R::kMmaWarp) {
    if (elect_one()) bwd_mma_role<D, WIDE>(smem_base, tmem, &bars, &cta_err);
    __syncwarp();
  } else if (warp < 4 * R::kGroups) {
    bwd_act_role<D, CAUSAL, ALIBI, DBIAS, KIND, WIDE>(p, &tmDk, &tmDv, warp >> 2, smem, smem_base, tmem, &bars, &cta_err);
  } else if constexpr (R::kDrainGroup) {
    bwd_drain_role<D, GROUPED>(p, &tmW, smem, tmem, &bars, &cta_err);
  } else {
    if (elect_one()) bwd_store_role<D>(p, &tmW, smem_base, &bars, &cta_err);
    __syncwarp();
  }

  tc_fence_before_sync();
  __syncthreads();
  if (cta_err != 0) {
    if (threadIdx.x == 0) atomicExch(p.status, 200 + cta_err);
    __nanosleep(100000);
  }
  if (warp == R::kMmaWarp) tmem_dealloc(tmem, 512);
}

// dQ (bf16) = scale * workspace (fp32): the conversion step that follows the main kernel.
__global__ void __launch_bounds__(256)
sigattn_bwd_convert_dq_kernel(const float4* __restrict__ ws, uint2* __restrict__ dq, size_t n_vec4, float scale) {
  grid_dependency_wait();
  grid_dependency_trigger();
  const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n_vec4; i += stride) {
    const float4 v = ws[i];
    uint2 o;
    o.x = pack_bf16x2(scale * v.x, scale * v.y);
    o.y = pack_bf16x2(scale * v.z, scale * v.w);
    dq[i] = o;
  }
}

// The same conversion with the temperature gradient on the side.  With the logits e^t * scale * q k + b
// (the learnable temperature of Section 5 and Appendix G.2.2; the caller passes scale * e^t as the
// scale), dL/dt = sum_ij dS_ij * scale' q_i k_j = sum_i <q_i, dQ_i>, because dQ_i = scale' sum_j dS_ij k_j:
// a reduction of what this pass streams anyway.  grid = (blocks per head, B*H); every block reduces its
// slice of one head and adds it to dtemp[b*H + h] (fp32 atomics: the last bits depend on the order).
__global__ void __launch_bounds__(256)
sigattn_bwd_convert_dq_dtemp_kernel(const float4* __restrict__ ws, const uint2* __restrict__ q, uint2* __restrict__ dq,
                                    size_t vec4_per_head, float scale, float* __restrict__ dtemp) {
  const size_t base = static_cast<size_t>(blockIdx.y) * vec4_per_head;
  const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
  float sum = 0.0f;
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < vec4_per_head; i += stride) {
    const float4 v = ws[base + i];
    const uint2 qq = q[base + i];
    const float g0 = scale * v.x, g1 = scale * v.y, g2 = scale * v.z, g3 = scale * v.w;
    dq[base + i] = make_uint2(pack_bf16x2(g0, g1), pack_bf16x2(g2, g3));
    sum = fmaf(g0, __uint_as_float(qq.x << 16), sum);
    sum = fmaf(g1, __uint_as_float(qq.x & 0xffff0000u), sum);
    sum = fmaf(g2, __uint_as_float(qq.y << 16), sum);
    sum = fmaf(g3, __uint_as_float(qq.y & 0xffff0000u), sum);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  __shared__ float warp_sums[8];
  if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    float total = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) total += warp_sums[w];
    atomicAdd(dtemp + blockIdx.y, total);
  }
}

// Sequence-length normalisation, O = r (P V) with one factor per query row: the whole backward
// is the plain one on r_i dO_i.  This pass writes bf16(r_i dO_i) for every row ([B*H, N, D]
// row-major, 8 elements per thread); the main kernel then reads it in place of dO.
__device__ __forceinline__ uint32_t scale_bf16x2(uint32_t x, float r) {
  return pack_bf16x2(r * __uint_as_float(x << 16), r * __uint_as_float(x & 0xffff0000u));
}

__global__ void __launch_bounds__(256)
sigattn_bwd_scale_rows_kernel(const uint4* __restrict__ d_o, const float* __restrict__ row_scale,
                              uint4* __restrict__ out, size_t n_vec8, int N, int vec_per_row) {
  const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n_vec8; i += stride) {
    const float r = __ldg(row_scale + static_cast<int>((i / vec_per_row) % N));
    const uint4 x = d_o[i];
    out[i] = make_uint4(scale_bf16x2(x.x, r), scale_bf16x2(x.y, r), scale_bf16x2(x.z, r), scale_bf16x2(x.w, r));
  }
}

// What the items in work at a time may touch of Q, dO and the dQ accumulator.
constexpr size_t kBwdL2Share = 64u << 20;

template <int D, bool CAUSAL, bool ALIBI, bool DBIAS, int KIND, bool WIDE>
int launch_bwd_variant(const CUtensorMap* maps, const BwdParams& bp, int num_sms, cudaStream_t stream,
                       cudaError_t* cuda_err) {
  auto kernel = sigattn_bwd_bf16_kernel<D, CAUSAL, ALIBI, DBIAS, KIND, WIDE>;
  // The shared-memory opt-in is a per-device attribute of the kernel: one bit per device ordinal
  // (a process may drive several GPUs); ordinals past 63 simply set it on every launch.
  static std::atomic<unsigned long long> configured{0};
  int dev = 0;
  *cuda_err = cudaGetDevice(&dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  const unsigned long long bit = (dev >= 0 && dev < 64) ? (1ull << dev) : 0ull;
  if ((configured.load(std::memory_order_relaxed) & bit) == 0) {
    *cuda_err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdSmem<D>::kDynBytes);
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
    configured.fetch_or(bit, std::memory_order_relaxed);
  }
  const int grid = (bp.dynamic || bp.n_items < num_sms) ? bp.n_items : num_sms;
  *cuda_err = launch_after(kernel, dim3(grid), BwdRoles<D, WIDE>::kThreads, BwdSmem<D>::kDynBytes, stream, 0, maps[0], maps[1],
                           maps[2], maps[3], maps[4], maps[5], maps[6], bp);
  return *cuda_err == cudaSuccess ? SIGATTN_OK : SIGATTN_ERR_CUDA;
}

}  // namespace

namespace {
thread_local cudaEvent_t t_ev_start = nullptr;
thread_local cudaEvent_t t_ev_stop = nullptr;
}  // namespace

void set_bwd_timing_events(cudaEvent_t start, cudaEvent_t stop) {
  t_ev_start = start;
  t_ev_stop = stop;
}

int launch_acc_to_bf16(const float* acc, void* out, size_t n, float mul, cudaStream_t stream,
                       unsigned long long* launches, cudaError_t* cuda_err) {
  int dev = 0, num_sms = 0;
  *cuda_err = cudaGetDevice(&dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  *cuda_err = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  const size_t n_vec4 = n / 4;
  const size_t want = n_vec4 / 256 + 1, cap = static_cast<size_t>(num_sms) * 8;
  *cuda_err = launch_after(sigattn_bwd_convert_dq_kernel, dim3(static_cast<unsigned>(want < cap ? want : cap)), 256, 0, stream, 0,
                           reinterpret_cast<const float4*>(acc), static_cast<uint2*>(out), n_vec4, mul);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  *launches += 1;
  return SIGATTN_OK;
}

size_t bwd_bf16_workspace_bytes(int B, int H, int N, int D) {
  return static_cast<size_t>(B) * H * N * D * sizeof(float);
}

int launch_bwd_bf16(const void* q, const void* k, const void* v, const void* d_o, void* dq, void* dk, void* dv,
                    const Problem& p, void* workspace, int* status, cudaStream_t stream,
                    unsigned long long* launches, cudaError_t* cuda_err) {
  if (short_bwd_serves(p)) {
    const bool timed = (t_ev_start != nullptr && t_ev_stop != nullptr);
    if (timed) cudaEventRecord(t_ev_start, stream);
    const int rc = launch_short_bwd_bf16(q, k, v, d_o, dq, dk, dv, p, status, stream, launches, cuda_err);
    if (timed && rc == SIGATTN_OK) cudaEventRecord(t_ev_stop, stream);
    return rc;
  }
  int dev = 0, num_sms = 0;
  *cuda_err = cudaGetDevice(&dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  *cuda_err = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;

  const uint64_t BH = static_cast<uint64_t>(p.B) * p.H;             // query heads: Q, dO, the dQ accumulator
  const uint64_t BH_kv = static_cast<uint64_t>(p.B) * p.kv_heads();  // K, V, dK, dV
  CUtensorMap maps[7];
  // with factors per query row the main kernel reads r dO, staged in the dq buffer: nothing
  // writes dq before the conversion step at the end, which reads only the workspace
  const void* ptrs[6] = {q, k, v, p.row_scale != nullptr ? dq : d_o, dk, dv};
  for (int i = 0; i < 6; ++i) {
    const uint64_t heads = (i == 0 || i == 3) ? BH : BH_kv;
    const uint64_t rows = (i == 0 || i == 3) ? p.N : p.key_rows();
    if (make_map_3d(&maps[i], ptrs[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, heads, rows, p.D, kT, 64) != 0) {
      *cuda_err = cudaErrorInvalidValue;
      return SIGATTN_ERR_CUDA;
    }
  }
  if (make_map_3d(&maps[6], workspace, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, BH, p.N, p.D, kT, 32) != 0) {
    *cuda_err = cudaErrorInvalidValue;
    return SIGATTN_ERR_CUDA;
  }
  BwdParams bp;
  bp.BH = static_cast<int>(BH_kv);
  bp.H = p.H;
  bp.H_kv = p.kv_heads();
  bp.group = p.H / p.kv_heads();
  bp.N = p.N;
  bp.n_tiles = (p.N + kT - 1) / kT;
  bp.n_tiles_k = (p.key_rows() + kT - 1) / kT;
  bp.pos0 = p.query_pos0();
  // Grouped heads with few (batch, key/value head) pairs: split a group's query heads over several
  // work items (the smallest divisor of the group size that yields two items per SM, if any).
  bp.n_sub = 1;
  if (bp.group > 1 && p.seqlens == nullptr && p.cu_seqlens == nullptr) {
    const long long base_items = static_cast<long long>(bp.n_tiles_k) * bp.BH;
    // at most four parts: every part adds one bf16 rounding to dK, dV (sixteen parts measured a
    // relative error of 5.5e-3, four stay near 3e-3)
    for (int d = 1; d <= bp.group && d <= 4; ++d) {
      if (bp.group % d != 0) continue;
      bp.n_sub = d;
      if (base_items * d >= 2ll * num_sms) break;
    }
  }
  bp.heads_per_sub = bp.group / bp.n_sub;
  // One query head per key/value head and at most one round of items: the first key tiles, which
  // meet every query tile, set the time.  Divide the query tiles of every key tile over two items
  // (two shares add up the same in either order, so dK, dV stay bit-reproducible).
  bp.i_split = 1;
  {
    const long long base_items = static_cast<long long>(bp.n_tiles_k) * bp.BH;
    const bool square = p.key_rows() == p.N && p.query_pos0() == 0;
    if (bp.group == 1 && square && p.seqlens == nullptr && p.cu_seqlens == nullptr && bp.n_tiles >= 4 &&
        (2 * base_items <= num_sms || (p.causal && base_items <= num_sms && bp.n_tiles >= 16)))
      bp.i_split = 2;
  }
  bp.dkv_add = p.acc_only == 2 ? 1 : 0;
  bp.n_items = bp.n_tiles_k * bp.BH * bp.n_sub * bp.i_split;
  bp.scale = p.scale;
  bp.scale_log2e = p.scale * kLog2eB;
  bp.bias_log2e = p.bias * kLog2eB;
  bp.bias_vec = p.bias_vec;
  bp.dbias = p.dbias;
  bp.slopes = p.slopes;
  bp.seqlens = p.seqlens;
  bp.cu_seqlens = p.cu_seqlens;
  bp.n_seqs = p.n_seqs;
  bp.status = status;

  const size_t n_elems = static_cast<size_t>(BH) * p.N * p.D;
  if ((bp.n_sub > 1 || bp.i_split > 1) && !bp.dkv_add) {   // dK, dV are summed over the parts: clear them first
    const size_t kv_bytes = static_cast<size_t>(BH_kv) * p.key_rows() * p.D * 2;
    *cuda_err = cudaMemsetAsync(dk, 0, kv_bytes, stream);
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
    *cuda_err = cudaMemsetAsync(dv, 0, kv_bytes, stream);
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  }
  // step 1: clear the fp32 dQ accumulator (and the bias gradient, which the kernel adds into);
  // with acc_only the accumulator is the caller's running sum over key/value shards: not cleared
  if (!p.acc_only) {
    *cuda_err = cudaMemsetAsync(workspace, 0, n_elems * sizeof(float), stream);
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  }
  if (p.dbias != nullptr) {
    const size_t n_bias = p.cu_seqlens != nullptr ? static_cast<size_t>(p.n_seqs) * p.H : BH;
    *cuda_err = cudaMemsetAsync(p.dbias, 0, n_bias * sizeof(float), stream);
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  }

  // Which heads are in work at a time.  Every item of a head reads the head's Q and dO and adds to its fp32 dQ
  // (8 N D bytes a head), so what all running items touch should stay in L2 (126 MB): heads are handed out in groups
  // of about 64 MB, drawn dynamically (the costs then fall group by group).  Long sequences run at the power limit,
  // where every byte that does not go to HBM is time.  Whole backward in a sustained loop, us, all heads at once /
  // groups of 128, 64, 32, 16 MB:
  //   B1 H32 N16384 D128 causal (512 MB)   7250 / 6040  5960  5970  6040
  //   B8 H12 N4096 D64 (192 MB)            1640 / 1410  1320  1305  1305
  //   B8 H16 N2048 D64 causal ALiBi (128)   322 /        310   311   314
  //   B2 H16 N4096 D128 causal (128)        455 /        441   444   445
  // A padded batch touches less than its shape says, and its items' costs differ: groups pay from about three times
  // that on (lengths N/4 to N, D64: B32 H16 N2500, 625 MB, 2300 -> 1970; B32 H8 N1500, 187 MB, 495 -> 505).
  // (Packed documents have their own locality: the key tiles in work belong to a few documents.)
  const size_t head_bytes = static_cast<size_t>(bp.group) * p.N * p.D * 8;
  bp.head_group = bp.BH;
  if (p.cu_seqlens == nullptr && head_bytes * bp.BH > (p.seqlens != nullptr ? 3 * kBwdL2Share : kBwdL2Share)) {
    const size_t heads = kBwdL2Share / head_bytes;
    if (heads < static_cast<size_t>(bp.BH)) bp.head_group = heads < 1 ? 1 : static_cast<int>(heads);
  }
  bp.dynamic = p.cu_seqlens != nullptr || bp.head_group < bp.BH;
  if (p.row_scale != nullptr) {
    const size_t n_vec8 = n_elems / 8;
    const size_t want = n_vec8 / 256 + 1, cap = static_cast<size_t>(num_sms) * 8;
    sigattn_bwd_scale_rows_kernel<<<static_cast<int>(want < cap ? want : cap), 256, 0, stream>>>(
        static_cast<const uint4*>(d_o), p.row_scale, static_cast<uint4*>(dq), n_vec8, p.N, p.D / 8);
    *cuda_err = cudaGetLastError();
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
    *launches += 1;
  }

  // step 2: main kernel
  const bool timed = (t_ev_start != nullptr && t_ev_stop != nullptr);
  if (timed) cudaEventRecord(t_ev_start, stream);
  int rc;
  const bool alibi = p.slopes != nullptr;
  // the bias gradient costs the activation groups a running sum (4-5 % of the kernel), so it
  // is compiled in only where it is asked for; likewise the loop over a group's query heads and
  // the per-sequence lengths (kind 1) and the lookups of a batch without padding (kind 2)
  // Wide or narrow at D = 64 (see BwdRoles).  Short sequences have b = -log n near the common path's limit, so many warps
  // take both activation paths, and their items have few steps, few of them unmasked; there four groups pay.  Elsewhere
  // the other work of those groups costs more.  The line is drawn by the length a typical row sees, where the two cross
  // (whole backward, us, narrow / wide; lengths of padded batches N/4 to N, packed documents in 16384 rows):
  //   no mask, B16 H12:        N300 43.0 / 41.0, 385 62.7 / 64.4, 577 86.6 / 87.5, 1100 225 / 237, 2048 347 / 371
  //     ALiBi:                 N260 41.3 / 42.6, 350 42.8 / 43.0, 577 88.2 / 94.1, 1025 245 / 255
  //     H16 H_kv4:             N300 70.4 / 63.5, 400 98.2 / 90.9, 600 137 / 140, 1500 270 / 290
  //     the same with ALiBi:   N200 48.6 / 43.1, 385 106 / 102, 520 151 / 156, 1025 344 / 355
  //   causal, H16:             N300 53.8 / 53.2, 512 79.2 / 75.7, 700 66.2 / 63.7, 850 75.0 / 76.4, 1024 89 / 92, 2048 272 / 280
  //     ALiBi:                 N300 51.9 / 49.2, 512 72.4 / 71.5, 850 74.8 / 76.1, 2048 280 / 290
  //     H_kv4:                 N300 62.5 / 59.4, 512 51.9 / 49.7, 577 108 / 113, 1000 94.6 / 98.6, 2000 137 / 145, 3000 309 / 333
  //     query tiles divided:   B1 H2 N500 19.2 / 19.2, 700 19.4 / 21.1, 2000 27.5 / 29.6
  //   padded, H8:              N400 51.2 / 49.2, 800 100 / 94, 1000 115 / 118, 1500 203 / 208, 2700 303 / 311
  //     causal:                N400 47.8 / 47.3, 800 83.8 / 77.9, 1200 132 / 140, 1500 146 / 139, 1800 94.1 / 93.4, 2500 168 / 176
  //     ALiBi without a mask:  N200 30.7 / 30.2, 400 55.3 / 53.3, 577 72 / 73, 1250 226 / 237
  //   packed, causal, H16:     120 documents 178 / 162, 60 218 / 186, 20 317 / 299, 14 320 / 310, 12 346 / 343, 10 404 / 404, 8 490 / 499
  //     H_kv4:                 60 229 / 205, 20 454 / 444, 14 337 / 324, 12 383 / 388, 8 500 / 504;  no mask 60 298 / 252, 12 570 / 579
  //     ALiBi without a mask:  60 297 / 272, 20 608 / 596, 16 525 / 527, 12 669 / 680
  const int typical_rows = p.cu_seqlens != nullptr ? p.N / p.n_seqs
                           : p.seqlens != nullptr  ? p.N / 2
                           : p.causal              ? p.N / 3 * 2 : p.N;
  const bool alibi_no_mask = alibi && !p.causal;
  const int wide_rows = p.cu_seqlens != nullptr            ? (alibi_no_mask ? 900 : 1280)
                        : p.seqlens != nullptr             ? (alibi_no_mask ? 250 : 450)
                        : bp.group > 1                     ? (p.causal ? 360 : 480)
                        : alibi_no_mask || bp.i_split > 1  ? 0
                                                           : (p.causal ? 500 : 320);
  const bool wide = p.D == 64 && typical_rows <= wide_rows;
  // (plain calls with ALiBi and no mask never take the wide shape: it is not compiled for them)
#define SIGATTN_BWD_SHAPE(DD, CC, AA, BB, KK)                                                              \
  (wide ? launch_bwd_variant<DD, CC, AA, BB, KK, DD == 64 && !(KK == 0 && AA && !CC)>(maps, bp, num_sms, stream, cuda_err) \
        : launch_bwd_variant<DD, CC, AA, BB, KK, false>(maps, bp, num_sms, stream, cuda_err))
#define SIGATTN_BWD_KIND(DD, CC, AA, KK)                                                                   \
  ((p.dbias != nullptr) ? SIGATTN_BWD_SHAPE(DD, CC, AA, true, KK) : SIGATTN_BWD_SHAPE(DD, CC, AA, false, KK))
#define SIGATTN_BWD_CASE(DD, CC, AA)                                                                       \
  rc = (bp.cu_seqlens != nullptr)                  ? SIGATTN_BWD_KIND(DD, CC, AA, 2)                        \
       : (bp.group > 1 || bp.seqlens != nullptr || bp.i_split > 1 || bp.dkv_add) ? SIGATTN_BWD_KIND(DD, CC, AA, 1) \
                                                   : SIGATTN_BWD_KIND(DD, CC, AA, 0)
  if (p.D == 128) {
    if (p.causal) { if (alibi) SIGATTN_BWD_CASE(128, true, true); else SIGATTN_BWD_CASE(128, true, false); }
    else          { if (alibi) SIGATTN_BWD_CASE(128, false, true); else SIGATTN_BWD_CASE(128, false, false); }
  } else {
    if (p.causal) { if (alibi) SIGATTN_BWD_CASE(64, true, true); else SIGATTN_BWD_CASE(64, true, false); }
    else          { if (alibi) SIGATTN_BWD_CASE(64, false, true); else SIGATTN_BWD_CASE(64, false, false); }
  }
#undef SIGATTN_BWD_CASE
#undef SIGATTN_BWD_KIND
#undef SIGATTN_BWD_SHAPE
  if (rc != SIGATTN_OK) return rc;
  if (timed) cudaEventRecord(t_ev_stop, stream);
  *launches += 1;

  if (p.acc_only) return SIGATTN_OK;   // the owner of the accumulator converts once every shard has added

  // step 3: dQ = scale * accumulator, as bf16 (and, on request, the temperature gradient from the same pass)
  const size_t n_vec4 = n_elems / 4;  // D is a multiple of 64
  if (p.dtemp != nullptr) {
    *cuda_err = cudaMemsetAsync(p.dtemp, 0, BH * sizeof(float), stream);
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
    const size_t per_head = static_cast<size_t>(p.N) * p.D / 4;
    const size_t want = per_head / 256 + 1, cap = (static_cast<size_t>(num_sms) * 8 + BH - 1) / BH;
    dim3 grid(static_cast<unsigned>(want < cap ? want : (cap < 1 ? 1 : cap)), static_cast<unsigned>(BH));
    sigattn_bwd_convert_dq_dtemp_kernel<<<grid, 256, 0, stream>>>(static_cast<const float4*>(workspace),
                                                                  static_cast<const uint2*>(q), static_cast<uint2*>(dq),
                                                                  per_head, p.scale, p.dtemp);
    *cuda_err = cudaGetLastError();
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
    *launches += 1;
    return SIGATTN_OK;
  }
  const int blocks = static_cast<int>(n_vec4 / 256 + 1 < static_cast<size_t>(num_sms) * 8 ? n_vec4 / 256 + 1
                                                                                            : static_cast<size_t>(num_sms) * 8);
  *cuda_err = launch_after(sigattn_bwd_convert_dq_kernel, dim3(blocks), 256, 0, stream, 0, static_cast<const float4*>(workspace),
                           static_cast<uint2*>(dq), n_vec4, p.scale);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  *launches += 1;
  return SIGATTN_OK;
}

}  // namespace sigattn
