// bf16 backward for short sequences, D = 64 and N <= 256: one thread block computes a whole (batch, head).
//
// Per head at most two key tiles j and two query tiles i of 128 rows, visited in the order (j, i) = (0,0), (0,1),
// (1,0), (1,1) (causal: without (1,0)); the products of a step are those of the general kernel,
//
//     S^T = K_j Q_i^T -> P^T;  dV_j += P^T dO_i;  dP^T = V_j dO_i^T;  dS^T = P^T (1 - P^T) dP^T;
//     dK_j += dS^T Q_i;  dQ_i += dS K_j
//
// but dQ stays in tensor memory as well (S^T and dP^T 128 columns each, dV, dK, dQ_0, dQ_1 64 each: all 512), so
// there is no fp32 accumulator in global memory: nothing to clear, no reduce-adds, no drain, no conversion pass.
// Each input is read once and each gradient written once.
//
// The steps of all heads of a thread block form one stream.  Q_0 and dO_0 have two buffers each, K_0 and V_0 are
// free after half a head, and the others are needed last, so the next head's first products run while this head's
// last step is evaluated.  The accumulators of a finished key tile (and of the head) are converted after the P
// phase of the following step, when the products that complete them have had time to run.  Only what counts is
// evaluated: query columns and key quarters in units of 32.
//
// Sixteen activation warps (32 columns a thread; four per scheduler hide the chain's latency); the epilogues are
// theirs too, so registers allow them.  What bounds it: the activation phases of a step (P, then dS) and the wait
// for the next S^T between them (at B32 H12 N197 43 % of the issue slots, 29 % of the MUFU pipe and 17 % of the tensor
// pipe are in use).  Measured when it was new, whole backward, us, clear + general kernel + conversion / this: B32 H12 N197
// 61.8 / 36.9, N64 28.7 / 12.7, N128 32.8 / 16.5, N256 74.2 / 43.2; causal B64 H16 N200 143 / 84.6; B1 H12 N50 13.6 / 7.2,
// N197 19.5 / 15.2.  Now, one call after the other: 32.5, 9.6, 13.0, 36.2; 74.2; 7.5, 12.6.
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

constexpr int kSbD = 64;
constexpr int kSbT = 128;                     // rows of a tile
constexpr int kSbMaxN = 256;
constexpr int kSbActWarps = 16;
constexpr int kSbActThreads = 32 * kSbActWarps;
constexpr int kSbThreads = kSbActThreads + 64;
constexpr int kSbLoadWarp = kSbActWarps;
constexpr int kSbMmaWarp = kSbActWarps + 1;
constexpr int kSbTileBytes = kSbT * 128;      // 128 rows of 64 bf16
constexpr int kSbSlots = 10;                  // operand tiles
// shared memory: operand tiles; dS^T (two panels of 64 queries); dV, dK staging
constexpr int kSbDs = kSbSlots * kSbTileBytes;
constexpr int kSbStage = kSbDs + 2 * kSbTileBytes;
constexpr int kSbDynBytes = kSbStage + 2 * kSbTileBytes + 1024;
// tensor memory
constexpr uint32_t kSbA = 0, kSbB = 128, kSbDv = 256, kSbDk = 320, kSbDq = 384;
constexpr float kSbLog2e = 1.4426950408889634f;

struct ShortBwdBarriers {
  uint64_t full[kSbSlots], empty[kSbSlots];
  uint64_t s_full, p_ready, dp_full, ds_ready, acc_full, acc_empty;
};

struct ShortBwdParams {
  int H, N, n_tiles, n_heads;
  float scale, scale_log2e, bias_log2e;
  const float* bias_vec;   // one bias per (batch, head), or nullptr
  const float* slopes;
  int* status;
};

// Operand tiles and where head number `h` (of this thread block) keeps them.  With two tiles Q_0 and dO_0
// alternate between two slots; with one tile all four operands do.
enum ShortTile { kQ0, kDo0, kK0, kV0, kQ1, kDo1, kK1, kV1 };
__device__ __forceinline__ uint32_t short_slot(int tile, uint32_t h, bool one_tile) {
  const uint32_t odd = h & 1;
  switch (tile) {
    case kQ0: return odd;
    case kDo0: return 2 + odd;
    case kK0: return one_tile ? 4 + 4 * odd : 4;
    case kV0: return one_tile ? 5 + 4 * odd : 5;
    case kQ1: return 6;
    case kDo1: return 7;
    case kK1: return 8;
    default: return 9;
  }
}
// Parity of that slot's use (its use number, modulo two).
__device__ __forceinline__ uint32_t short_use(int tile, uint32_t h, bool one_tile) {
  return ((one_tile || tile == kQ0 || tile == kDo0) ? h >> 1 : h) & 1;
}

// Rows of tile t that count, rounded up to 32.
__device__ __forceinline__ int short_live(const ShortBwdParams& p, int t) {
  return (min(kSbT, p.N - t * kSbT) + 31) & ~31;
}

// The step stream: head by head, key tile by key tile.
struct ShortStep {
  uint32_t h;    // number of the head within this thread block
  int head;      // (batch, head), or >= n_heads past the end
  int j, i;
};
template <bool CAUSAL>
__device__ __forceinline__ ShortStep short_next(ShortStep s, int n_tiles) {
  if (++s.i == n_tiles) {
    if (++s.j == n_tiles) {
      s.j = 0;
      ++s.h;
      s.head += gridDim.x;
    }
    s.i = CAUSAL ? s.j : 0;
  }
  return s;
}

template <bool CAUSAL, bool ALIBI>
__global__ void __launch_bounds__(kSbThreads, 1)
sigattn_short_bwd_bf16_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                              const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmDo,
                              const __grid_constant__ CUtensorMap tmDq, const __grid_constant__ CUtensorMap tmDk,
                              const __grid_constant__ CUtensorMap tmDv, const ShortBwdParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ ShortBwdBarriers bars;
  __shared__ uint32_t tmem_base_slot;
  __shared__ int cta_err_slot;
  volatile int* cta_err = &cta_err_slot;

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem_base = smem_u32(smem);
  const int warp = threadIdx.x >> 5;
  const int n_tiles = p.n_tiles;
  const bool one_tile = n_tiles == 1;

  if (threadIdx.x == 0) {
    cta_err_slot = 0;
    for (int s = 0; s < kSbSlots; ++s) {
      mbar_init(smem_u32(&bars.full[s]), 1);
      mbar_init(smem_u32(&bars.empty[s]), 1);
    }
    mbar_init(smem_u32(&bars.s_full), 1);
    mbar_init(smem_u32(&bars.p_ready), kSbActThreads);
    mbar_init(smem_u32(&bars.dp_full), 1);
    mbar_init(smem_u32(&bars.ds_ready), kSbActThreads);
    mbar_init(smem_u32(&bars.acc_full), 1);
    mbar_init(smem_u32(&bars.acc_empty), kSbActThreads);
    fence_mbar_init();
  }
  if (warp == kSbLoadWarp && elect_one()) {
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
    tma_prefetch_desc(&tmDo);
    tma_prefetch_desc(&tmDq);
    tma_prefetch_desc(&tmDk);
    tma_prefetch_desc(&tmDv);
  }
  if (warp == kSbMmaWarp) {
    tmem_alloc(smem_u32(&tmem_base_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_base_slot;
  grid_dependency_wait();
  grid_dependency_trigger();

  if (warp == kSbLoadWarp) {
    if (elect_one()) {
      bool ok = true;
      uint32_t h = 0;
      for (int head = blockIdx.x; ok && head < p.n_heads; head += gridDim.x, ++h) {
        // in the order of first use: S^T(0,0), dP^T(0,0), then the second query tile, then the second key tile
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          constexpr int kOrder[8] = {kQ0, kK0, kDo0, kV0, kQ1, kDo1, kK1, kV1};
          const int tile = kOrder[e];
          if (!ok || (one_tile && e >= 4)) break;
          const uint32_t slot = short_slot(tile, h, one_tile);
          ok = mbar_wait(smem_u32(&bars.empty[slot]), short_use(tile, h, one_tile) ^ 1, cta_err, 10);
          if (!ok) break;
          const uint32_t bar = smem_u32(&bars.full[slot]);
          mbar_arrive_expect_tx(bar, kSbTileBytes);
          const CUtensorMap* tm = (tile == kQ0 || tile == kQ1) ? &tmQ
                                  : (tile == kK0 || tile == kK1) ? &tmK
                                  : (tile == kV0 || tile == kV1) ? &tmV : &tmDo;
          tma_load_3d(smem_base + slot * kSbTileBytes, tm, bar, 0, e >= 4 ? kSbT : 0, head);
        }
      }
    }
    __syncwarp();
  } else if (warp == kSbMmaWarp) {
    if (elect_one()) {
      constexpr uint32_t kIdescAcc = make_idesc_bf16(kSbT, kSbD, 0, 1);   // dV, dK: tensor memory x MN-major
      constexpr uint32_t kIdescDq = make_idesc_bf16(kSbT, kSbD, 1, 1);    // dQ: MN-major x MN-major
      const uint64_t k_major0 = make_smem_desc_sw128(smem_base, 16, 1024);
      const uint64_t mn_major0 = make_smem_desc_sw128(smem_base, kSbTileBytes, 1024);
      const uint64_t ds_mn = make_smem_desc_sw128(smem_base + kSbDs, kSbTileBytes, 1024);
      auto q_tile = [](int i) { return i ? kQ1 : kQ0; };
      auto do_tile = [](int i) { return i ? kDo1 : kDo0; };
      auto k_tile = [](int j) { return j ? kK1 : kK0; };
      auto v_tile = [](int j) { return j ? kV1 : kV0; };
      auto slot = [&](int tile, uint32_t h) { return short_slot(tile, h, one_tile); };
      auto wait_tile = [&](int tile, uint32_t h, int where) {   // (a tile already seen complete returns at once)
        return mbar_wait(smem_u32(&bars.full[slot(tile, h)]), short_use(tile, h, one_tile), cta_err, where);
      };
      // [128 keys x live queries] = X[128 x 64] Y[. x 64]^T, both K-major
      auto issue_kk = [&](uint32_t d_col, uint32_t x_slot, uint32_t y_slot, int i) {
        const uint32_t idesc = make_idesc_bf16(kSbT, 0, 0, 0) | (static_cast<uint32_t>(short_live(p, i) >> 3) << 17);
        const uint64_t x = desc_advance(k_major0, x_slot * kSbTileBytes), y = desc_advance(k_major0, y_slot * kSbTileBytes);
#pragma unroll
        for (int ks = 0; ks < kSbD / 16; ++ks)
          umma_ss(tmem + d_col, desc_advance(x, ks * 32), desc_advance(y, ks * 32), idesc, ks > 0);
      };
      auto issue_s = [&](const ShortStep& s) -> bool {
        if (!wait_tile(q_tile(s.i), s.h, 20) || !wait_tile(k_tile(s.j), s.h, 21)) return false;
        tc_fence_after_sync();
        issue_kk(kSbA, slot(k_tile(s.j), s.h), slot(q_tile(s.i), s.h), s.i);
        umma_commit(smem_u32(&bars.s_full));
        return true;
      };
      auto issue_dp = [&](const ShortStep& s) -> bool {
        if (!wait_tile(do_tile(s.i), s.h, 22) || !wait_tile(v_tile(s.j), s.h, 23)) return false;
        tc_fence_after_sync();
        issue_kk(kSbB, slot(v_tile(s.j), s.h), slot(do_tile(s.i), s.h), s.i);
        umma_commit(smem_u32(&bars.dp_full));
        return true;
      };
      ShortStep s = {0, static_cast<int>(blockIdx.x), 0, 0};
      uint32_t step = 0, n_acc = 0;
      bool ok = issue_s(s) && issue_dp(s);
      while (ok && s.head < p.n_heads) {
        const ShortStep next = short_next<CAUSAL>(s, n_tiles);
        const bool more = next.head < p.n_heads;
        const bool first_of_j = s.i == (CAUSAL ? s.j : 0), last_of_j = s.i == n_tiles - 1;
        const int q16 = short_live(p, s.i) >> 4, k16 = short_live(p, s.j) >> 4;
        // dV_j += P^T dO_i
        ok = mbar_wait(smem_u32(&bars.p_ready), step & 1, cta_err, 24);
        if (ok && first_of_j) ok = mbar_wait(smem_u32(&bars.acc_empty), (n_acc & 1) ^ 1, cta_err, 25);
        if (!ok) break;
        tc_fence_after_sync();
        const uint64_t do_mn = desc_advance(mn_major0, slot(do_tile(s.i), s.h) * kSbTileBytes);
#pragma unroll 2
        for (int ks = 0; ks < q16; ++ks)
          umma_ts(tmem + kSbDv, tmem + kSbA + (ks >> 1) * 32 + (ks & 1) * 8, desc_advance(do_mn, ks * 2048), kIdescAcc,
                  (!first_of_j || ks > 0));
        // S^T of the next step, over P^T
        if (more) ok = issue_s(next);
        // dK_j += dS^T Q_i, dQ_i += dS K_j
        if (ok) ok = mbar_wait(smem_u32(&bars.ds_ready), step & 1, cta_err, 26);
        if (!ok) break;
        tc_fence_after_sync();
        const uint64_t q_mn = desc_advance(mn_major0, slot(q_tile(s.i), s.h) * kSbTileBytes);
#pragma unroll 2
        for (int ks = 0; ks < q16; ++ks)
          umma_ts(tmem + kSbDk, tmem + kSbB + (ks >> 1) * 32 + (ks & 1) * 8, desc_advance(q_mn, ks * 2048), kIdescAcc,
                  (!first_of_j || ks > 0));
        const uint64_t k_mn = desc_advance(mn_major0, slot(k_tile(s.j), s.h) * kSbTileBytes);
#pragma unroll 2
        for (int ks = 0; ks < k16; ++ks)
          umma_ss(tmem + kSbDq + s.i * kSbD, desc_advance(ds_mn, ks * 2048), desc_advance(k_mn, ks * 2048), kIdescDq,
                  (s.j > 0 || ks > 0));
        if (last_of_j) {
          umma_commit(smem_u32(&bars.empty[slot(k_tile(s.j), s.h)]));
          umma_commit(smem_u32(&bars.empty[slot(v_tile(s.j), s.h)]));
        }
        // query tiles are last used by the last key tile; with two tiles the slots of Q_0 and dO_0 stage dQ
        // before the activation threads release them
        if (s.j == n_tiles - 1 && (one_tile || s.i == 1)) {
          umma_commit(smem_u32(&bars.empty[slot(q_tile(s.i), s.h)]));
          umma_commit(smem_u32(&bars.empty[slot(do_tile(s.i), s.h)]));
        }
        if (last_of_j) {   // after the others: nothing waits for the slots of a block's last head
          umma_commit(smem_u32(&bars.acc_full));
          ++n_acc;
        }
        if (more) ok = issue_dp(next);
        s = next;
        ++step;
      }
    }
    __syncwarp();
  } else {
    const int g = warp >> 2;                     // 32-query column group
    const int tid = threadIdx.x & 127;           // key row of the tile; in the epilogues row of the output tile
    const int quarter = (warp & 3) * 32;
    const uint32_t lane_off = static_cast<uint32_t>(quarter) << 16;
    uint32_t step = 0, n_acc = 0;

    // This thread's 32 columns of an accumulator tile -> bf16 (times mul) -> staging tile
    auto stage_cols = [&](uint32_t t_col, int stage_off, float mul) {
      uint32_t o[32];
      tmem_ld32(tmem + lane_off + t_col + (g & 1) * 32, o);
      tmem_wait_ld();
      uint8_t* row = smem + stage_off + tid * 128;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint4 val;
        val.x = pack_bf16x2(mul * __uint_as_float(o[8 * c + 0]), mul * __uint_as_float(o[8 * c + 1]));
        val.y = pack_bf16x2(mul * __uint_as_float(o[8 * c + 2]), mul * __uint_as_float(o[8 * c + 3]));
        val.z = pack_bf16x2(mul * __uint_as_float(o[8 * c + 4]), mul * __uint_as_float(o[8 * c + 5]));
        val.w = pack_bf16x2(mul * __uint_as_float(o[8 * c + 6]), mul * __uint_as_float(o[8 * c + 7]));
        *reinterpret_cast<uint4*>(row + ((((g & 1) * 4 + c) ^ (tid & 7)) * 16)) = val;
      }
    };
    // Results of the key tile that step `e` finished (and of the head, if it finished that): groups 0 and 1 take
    // dV_j, 2 and 3 dK_j; then 0 and 1 dQ_0, 2 and 3 dQ_1.  The stores are not waited for here but before the
    // staging tiles are written again: dQ is staged where the next loads come last (with two tiles the slots of
    // the head's own Q_0 and dO_0, which wait for the head after the next; with one tile a slot that holds no
    // operand).
    uint32_t release = 0;   // thread 0: slots (1 + number, a byte each) to hand to the producer once read
    auto stores_read = [&]() {
      tma_wait_group_read<0>();
      for (; release != 0; release >>= 8) mbar_arrive(smem_u32(&bars.empty[(release & 255u) - 1]));
    };
    auto epilogue = [&](const ShortStep& e) -> bool {
      if (threadIdx.x == 0) stores_read();
      named_barrier_sync<1, kSbActThreads>();   // the staging tiles may be written
      if (!mbar_wait(smem_u32(&bars.acc_full), n_acc & 1, cta_err, 33)) return false;
      ++n_acc;
      tc_fence_after_sync();
      const bool head_done = e.j == n_tiles - 1;
      const uint32_t q_stage = one_tile ? 6 : short_slot(kQ0, e.h, false), do_stage = short_slot(kDo0, e.h, false);
      if (e.j * kSbT + quarter < p.N)
        stage_cols(g < 2 ? kSbDv : kSbDk, kSbStage + (g >> 1) * kSbTileBytes, g < 2 ? 1.0f : p.scale);
      if (head_done && (g >> 1) * kSbT + quarter < p.N)
        stage_cols(kSbDq + (g >> 1) * kSbD, (g < 2 ? q_stage : do_stage) * kSbTileBytes, p.scale);
      tc_fence_before_sync();
      mbar_arrive(smem_u32(&bars.acc_empty));
      fence_proxy_async_smem();
      named_barrier_sync<1, kSbActThreads>();
      if (threadIdx.x == 0) {   // (rows >= N are clipped)
        tma_store_3d(&tmDv, smem_base + kSbStage, 0, e.j * kSbT, e.head);
        tma_store_3d(&tmDk, smem_base + kSbStage + kSbTileBytes, 0, e.j * kSbT, e.head);
        if (head_done) {
          tma_store_3d(&tmDq, smem_base + q_stage * kSbTileBytes, 0, 0, e.head);
          if (!one_tile) {
            tma_store_3d(&tmDq, smem_base + do_stage * kSbTileBytes, 0, kSbT, e.head);
            release = (q_stage + 1) | ((do_stage + 1) << 8);
          }
        }
        tma_commit_group();
      }
      return true;
    };

    ShortStep s = {0, static_cast<int>(blockIdx.x), 0, 0}, pending = s;
    bool have_pending = false, ok = true;
    while (ok && s.head < p.n_heads) {
      const bool live = s.j * kSbT + quarter < p.N && g * 32 < short_live(p, s.i);
      const float slope = ALIBI ? __ldg(p.slopes + s.head % p.H) * kSbLog2e : 0.0f;
      const float bias = p.bias_vec ? __ldg(p.bias_vec + s.head) * kSbLog2e : p.bias_log2e;
      float pp[32];
      ok = mbar_wait(smem_u32(&bars.s_full), step & 1, cta_err, 30);
      if (!ok) break;
      tc_fence_after_sync();
      if (live) {
        uint32_t v[32], pk[16];
        tmem_ld32(tmem + kSbA + lane_off + g * 32, v);
        tmem_wait_ld();
        const float col_rel = static_cast<float>((s.j - s.i) * kSbT + tid);   // this key minus the tile's first query
        if (CAUSAL && s.i == s.j)
          bwd_sigmoid_chunk<1, ALIBI, CAUSAL>(v, pk, pp, p.scale_log2e, bias, slope, col_rel, g * 32, col_rel, 0.0f);
        else
          bwd_sigmoid_chunk<0, ALIBI, CAUSAL>(v, pk, pp, p.scale_log2e, bias, slope, col_rel, g * 32, 0.0f, 0.0f);
        tmem_st16(tmem + kSbA + lane_off + g * 32, pk);
        tmem_wait_st();
      }
      tc_fence_before_sync();
      mbar_arrive(smem_u32(&bars.p_ready));

      if (have_pending) {
        ok = epilogue(pending);
        have_pending = false;
        if (!ok) break;
      }

      ok = mbar_wait(smem_u32(&bars.dp_full), step & 1, cta_err, 31);
      if (!ok) break;
      tc_fence_after_sync();
      if (live) {
        uint8_t* ds_row = smem + kSbDs + (g >> 1) * kSbTileBytes + tid * 128;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t dp[16], ds[8];
          tmem_ld16(tmem + kSbB + lane_off + g * 32 + c * 16, dp);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 8; ++e)
            ds[e] = pack_bf16x2(pp[c * 16 + 2 * e] * __uint_as_float(dp[2 * e]),
                                pp[c * 16 + 2 * e + 1] * __uint_as_float(dp[2 * e + 1]));
#pragma unroll
          for (int q = 0; q < 2; ++q)
            *reinterpret_cast<uint4*>(ds_row + ((((g & 1) * 4 + c * 2 + q) ^ (tid & 7)) * 16)) =
                make_uint4(ds[4 * q + 0], ds[4 * q + 1], ds[4 * q + 2], ds[4 * q + 3]);
          tmem_st8(tmem + kSbB + lane_off + g * 32 + c * 8, ds);
        }
        tmem_wait_st();
      }
      tc_fence_before_sync();
      fence_proxy_async_smem();
      mbar_arrive(smem_u32(&bars.ds_ready));
      if (threadIdx.x == 0 && release != 0) stores_read();
      if (s.i == n_tiles - 1) {
        pending = s;
        have_pending = true;
      }
      s = short_next<CAUSAL>(s, n_tiles);
      ++step;
    }
    if (ok && have_pending) epilogue(pending);
    if (threadIdx.x == 0) tma_wait_group<0>();
  }

  tc_fence_before_sync();
  __syncthreads();
  if (cta_err_slot != 0) {
    if (threadIdx.x == 0) atomicExch(p.status, 500 + cta_err_slot);
    __nanosleep(100000);  // let copies in flight towards this thread block's shared memory land
  }
  if (warp == kSbMmaWarp) tmem_dealloc(tmem, 512);
}

template <bool CAUSAL, bool ALIBI>
int launch_short_bwd_variant(const CUtensorMap (&m)[7], const ShortBwdParams& sp, int num_sms, cudaStream_t stream,
                             cudaError_t* cuda_err) {
  auto kernel = sigattn_short_bwd_bf16_kernel<CAUSAL, ALIBI>;
  // a per-device attribute of the kernel: one bit per device ordinal, ordinals past 63 set it on every launch
  static std::atomic<unsigned long long> configured{0};
  int dev = 0;
  *cuda_err = cudaGetDevice(&dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  const unsigned long long bit = (dev >= 0 && dev < 64) ? (1ull << dev) : 0ull;
  if ((configured.load(std::memory_order_relaxed) & bit) == 0) {
    *cuda_err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSbDynBytes);
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
    configured.fetch_or(bit, std::memory_order_relaxed);
  }
  const int grid = sp.n_heads < num_sms ? sp.n_heads : num_sms;
  *cuda_err = launch_after(kernel, dim3(grid), kSbThreads, kSbDynBytes, stream, 0, m[0], m[1], m[2], m[3], m[4], m[5],
                           m[6], sp);
  return *cuda_err == cudaSuccess ? SIGATTN_OK : SIGATTN_ERR_CUDA;
}

}  // namespace

// Plain self-attention calls.  A single (batch, head) stays with the general kernels although this one is faster there up
// to 128 rows (N = 64 10.3 / 5.5 us, 128 12.3 / 6.7, 197 13.3 / 13.0, 256 14.4 / 14.3): forward, main kernel and conversion
// of one head are the three launches that callers who read sigattn_launch_count expect.
bool short_bwd_serves(const Problem& p) {
  return p.D == kSbD && p.N <= kSbMaxN && p.B * p.H > 1 && p.key_rows() == p.N && p.query_pos0() == 0 &&
         p.kv_heads() == p.H && p.seqlens == nullptr && p.row_scale == nullptr && p.cu_seqlens == nullptr &&
         p.dbias == nullptr && p.dtemp == nullptr && p.acc_only == 0;
}

int launch_short_bwd_bf16(const void* q, const void* k, const void* v, const void* d_o, void* dq, void* dk, void* dv,
                          const Problem& p, int* status, cudaStream_t stream, unsigned long long* launches,
                          cudaError_t* cuda_err) {
  int dev = 0, num_sms = 0;
  *cuda_err = cudaGetDevice(&dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  *cuda_err = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  ShortBwdParams sp = {};
  sp.H = p.H;
  sp.N = p.N;
  sp.n_tiles = (p.N + kSbT - 1) / kSbT;
  sp.n_heads = p.B * p.H;
  sp.scale = p.scale;
  sp.scale_log2e = p.scale * kSbLog2e;
  sp.bias_log2e = p.bias * kSbLog2e;
  sp.bias_vec = p.bias_vec;
  sp.slopes = p.slopes;
  sp.status = status;
  CUtensorMap maps[7];
  const void* ptrs[7] = {q, k, v, d_o, dq, dk, dv};
  for (int i = 0; i < 7; ++i) {
    if (make_map_3d(&maps[i], ptrs[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, sp.n_heads, p.N, kSbD, kSbT, 64) != 0) {
      *cuda_err = cudaErrorInvalidValue;
      return SIGATTN_ERR_CUDA;
    }
  }
  const bool alibi = p.slopes != nullptr;
  const int rc = p.causal ? (alibi ? launch_short_bwd_variant<true, true>(maps, sp, num_sms, stream, cuda_err)
                                   : launch_short_bwd_variant<true, false>(maps, sp, num_sms, stream, cuda_err))
                          : (alibi ? launch_short_bwd_variant<false, true>(maps, sp, num_sms, stream, cuda_err)
                                   : launch_short_bwd_variant<false, false>(maps, sp, num_sms, stream, cuda_err));
  if (rc == SIGATTN_OK) *launches += 1;
  return rc;
}

}  // namespace sigattn
