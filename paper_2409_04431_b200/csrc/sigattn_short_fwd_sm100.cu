// bf16 forward for short sequences, D = 64 and N <= 256 (one key pass): O = sigmoid(scale Q K^T + b ...) V.
//
// With at most 256 keys the logits of a 128-row query tile fit tensor memory whole (W = N rounded up to 32
// columns), so a work unit (head, query tile) is one product, one activation, one product:
//
//     S = Q_t K^T (N = W, one chain of four instructions)  ->  P over S  ->  O = P V  ->  store
//
// without a key loop, a ring or running accumulators.  A unit is a serial chain; what hides it is a second thread
// block on the same SM (256 columns of tensor memory and 97 KB of shared memory each) and the loads of the next
// unit: Q and K are free as soon as S is complete, V as soon as O is, so single buffers are enough.  Only what
// counts is evaluated: W columns instead of 256, no 32-row quarter that lies past row N, and with a causal mask
// no column past the tile's last row.
//
// What bounds it: the activation (W / 128 * 1024 MUFU cycles a unit and SM, more where unnormalised logits send
// warps through both evaluations) and the chain around it.  It serves every plain call of its size: measured
// against the general kernel when it was new, us: B32 H12 (no mask) N = 64 14.4 -> 10.3, 128 16.2 -> 14.3, 129 24.7 -> 18.6,
// 197 28.7 -> 25.8, 256 29.5 -> 28.8; causal B64 H16 N200 59.7 -> 47.7; B1 H12 N50 8.3 -> 6.2, N197 10.3 -> 9.8.  Now, one call
// after the other: 6.1, 9.3, 13.1, 17.9, 20.2; 42.7; 5.1, 5.9.
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

constexpr int kSfD = 64;
constexpr int kSfRows = 128;                 // query rows of a unit = tensor-memory lanes
constexpr int kSfMaxN = 256;
constexpr int kSfActWarps = 8;               // two groups of four: the columns of a row are divided between them
constexpr int kSfActThreads = 32 * kSfActWarps;
constexpr int kSfThreads = kSfActThreads + 64;
constexpr int kSfLoadWarp = kSfActWarps;
constexpr int kSfMmaWarp = kSfActWarps + 1;
constexpr int kSfTileBytes = kSfRows * 128;  // 128 rows of 64 bf16
// shared memory: Q, K (256 rows), V (256 rows), O
constexpr int kSfQ = 0, kSfK = kSfTileBytes, kSfV = 3 * kSfTileBytes, kSfO = 5 * kSfTileBytes;
constexpr int kSfDynBytes = 6 * kSfTileBytes + 1024;
constexpr float kSfLog2e = 1.4426950408889634f;

struct ShortFwdBarriers {
  uint64_t q_full, k_full, v_full, qk_empty, v_empty, s_full, p_full, o_full, o_empty;
};

struct ShortFwdParams {
  int H, N, n_tiles, n_units;
  float scale_log2e, bias_log2e;
  const float* bias_vec;   // one bias per (batch, head), or nullptr
  const float* slopes;
  int* status;
};

// Unit u: head u / n_tiles, the tile with more keys first.
struct ShortUnit {
  int head, row0;
  int width;    // logits columns, a multiple of 32
  int half;     // columns of the first activation group, a multiple of 32
  int o_col;    // where O is accumulated: beside the logits, or over logits that have been consumed
};

template <bool CAUSAL>
__device__ __forceinline__ ShortUnit short_unit(const ShortFwdParams& p, int u) {
  ShortUnit w;
  w.head = u / p.n_tiles;
  w.row0 = (p.n_tiles - 1 - (u - w.head * p.n_tiles)) * kSfRows;
  const int keys = CAUSAL ? min(p.N, w.row0 + kSfRows) : p.N;
  w.width = (keys + 31) & ~31;
  // The group's packed weights (16 columns per 32 logits) go over the start of its own columns.  Up to 192
  // columns leave [192, 256) for O; beyond that the first group's weights end at column 64 and O takes [64, 128).
  w.half = w.width > 192 ? 128 : ((w.width / 2 + 31) & ~31);
  w.o_col = w.width > 192 ? 64 : 192;
  return w;
}

template <bool CAUSAL, bool ALIBI>
__global__ void __launch_bounds__(kSfThreads, 2)
sigattn_short_fwd_bf16_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                              const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO,
                              const ShortFwdParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ ShortFwdBarriers bars;
  __shared__ uint32_t tmem_base_slot;
  __shared__ int cta_err_slot;
  volatile int* cta_err = &cta_err_slot;

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem_base = smem_u32(smem);
  // How many polls of a wait are unrolled (see mbar_wait_limit); forward, us, all / a loop / 8: causal B64 H16 N200
  // 42.66 / 42.93 / 42.92, B32 H12 N140 15.30 / 15.48 / 15.56; without a mask B64 H16 N200 39.6 / 39.4 / 39.1, B32 H12 N64
  // 6.24 / 6.15 / 6.06; causal ALiBi B64 H16 N200 40.7 / 40.4 / 40.2.
  constexpr int kPolls = (CAUSAL && !ALIBI) ? 64 : 8;
  const int warp = threadIdx.x >> 5;
  // contiguous runs of units per thread block: the units of a head share K and V
  const int u0 = static_cast<int>(static_cast<long long>(blockIdx.x) * p.n_units / gridDim.x);
  const int u1 = static_cast<int>(static_cast<long long>(blockIdx.x + 1) * p.n_units / gridDim.x);

  if (threadIdx.x == 0) {
    cta_err_slot = 0;
    mbar_init(smem_u32(&bars.q_full), 1);
    mbar_init(smem_u32(&bars.k_full), 1);
    mbar_init(smem_u32(&bars.v_full), 1);
    mbar_init(smem_u32(&bars.qk_empty), 1);
    mbar_init(smem_u32(&bars.v_empty), 1);
    mbar_init(smem_u32(&bars.s_full), 1);
    mbar_init(smem_u32(&bars.p_full), kSfActThreads);
    mbar_init(smem_u32(&bars.o_full), 1);
    mbar_init(smem_u32(&bars.o_empty), kSfActThreads);
    fence_mbar_init();
  }
  if (warp == kSfLoadWarp && elect_one()) {
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
    tma_prefetch_desc(&tmO);
  }
  if (warp == kSfMmaWarp) {
    tmem_alloc(smem_u32(&tmem_base_slot), 256);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_base_slot;
  grid_dependency_wait();
  grid_dependency_trigger();

  if (warp == kSfLoadWarp) {
    if ((threadIdx.x & 31) == 0) {
      const int kv_tiles = (p.N + kSfRows - 1) / kSfRows;
      auto load_kv = [&](const CUtensorMap* tm, uint32_t dst, uint64_t* full, int head) {
        const uint32_t bar = smem_u32(full);
        mbar_arrive_expect_tx(bar, kv_tiles * kSfTileBytes);
        for (int t = 0; t < kv_tiles; ++t) tma_load_3d(smem_base + dst + t * kSfTileBytes, tm, bar, 0, t * kSfRows, head);
      };
      int last_head = -1;
      for (int u = u0; u < u1; ++u) {
        const ShortUnit w = short_unit<CAUSAL>(p, u);
        const uint32_t i = u - u0;
        // unit i - 1 has computed its logits: Q and K may be overwritten; its O: V may be
        if (i > 0 && !mbar_wait<kPolls>(smem_u32(&bars.qk_empty), (i - 1) & 1, cta_err, 10)) break;
        if (w.head != last_head) load_kv(&tmK, kSfK, &bars.k_full, w.head);
        mbar_arrive_expect_tx(smem_u32(&bars.q_full), kSfTileBytes);
        tma_load_3d(smem_base + kSfQ, &tmQ, smem_u32(&bars.q_full), 0, w.row0, w.head);
        if (i > 0 && !mbar_wait<kPolls>(smem_u32(&bars.v_empty), (i - 1) & 1, cta_err, 11)) break;
        if (w.head != last_head) load_kv(&tmV, kSfV, &bars.v_full, w.head);
        last_head = w.head;
      }
    }
    __syncwarp();
  } else if (warp == kSfMmaWarp) {
    if (elect_one()) {
      constexpr uint32_t kIdescPV = make_idesc_bf16(kSfRows, kSfD, 0, 1);
      const uint64_t q_desc = make_smem_desc_sw128(smem_base + kSfQ, 16, 1024);
      const uint64_t k_desc = make_smem_desc_sw128(smem_base + kSfK, 16, 1024);
      const uint64_t v_desc = make_smem_desc_sw128(smem_base + kSfV, kSfTileBytes, 1024);
      int last_head = -1;
      uint32_t heads = 0;
      for (int u = u0; u < u1; ++u) {
        const ShortUnit w = short_unit<CAUSAL>(p, u);
        const uint32_t i = u - u0, par = i & 1;
        const bool new_head = w.head != last_head;
        last_head = w.head;
        if (new_head) ++heads;
        if (new_head && !mbar_wait<kPolls>(smem_u32(&bars.k_full), (heads - 1) & 1, cta_err, 20)) break;
        if (!mbar_wait<kPolls>(smem_u32(&bars.q_full), par, cta_err, 21)) break;
        if (i > 0 && !mbar_wait<kPolls>(smem_u32(&bars.o_empty), par ^ 1, cta_err, 22)) break;   // tensor memory free again
        tc_fence_after_sync();
        const uint32_t idesc_s = make_idesc_bf16(kSfRows, 0, 0, 0) | (static_cast<uint32_t>(w.width >> 3) << 17);
#pragma unroll
        for (int ks = 0; ks < kSfD / 16; ++ks)
          umma_ss(tmem, desc_advance(q_desc, ks * 32), desc_advance(k_desc, ks * 32), idesc_s, ks > 0);
        umma_commit(smem_u32(&bars.s_full));
        umma_commit(smem_u32(&bars.qk_empty));
        if (new_head && !mbar_wait<kPolls>(smem_u32(&bars.v_full), (heads - 1) & 1, cta_err, 23)) break;
        if (!mbar_wait<kPolls>(smem_u32(&bars.p_full), par, cta_err, 24)) break;
        tc_fence_after_sync();
        const int h16 = w.half >> 4, n16 = w.width >> 4;
#pragma unroll 4
        for (int ks = 0; ks < n16; ++ks) {
          const uint32_t p_col = ks < h16 ? ks * 8 : w.half + (ks - h16) * 8;
          umma_ts(tmem + w.o_col, tmem + p_col, desc_advance(v_desc, ks * 2048), kIdescPV, ks > 0);
        }
        umma_commit(smem_u32(&bars.v_empty));
        umma_commit(smem_u32(&bars.o_full));   // last: nothing waits for the v_empty of a block's last unit
      }
    }
    __syncwarp();
  } else {
    const int g = warp >> 2;                        // column group
    const int tid = threadIdx.x & 127;              // row of the tile
    const int quarter = (warp & 3) * 32;            // first row of this warp
    const uint32_t lane_off = static_cast<uint32_t>(quarter) << 16;
    for (int u = u0; u < u1; ++u) {
      const ShortUnit w = short_unit<CAUSAL>(p, u);
      const uint32_t par = (u - u0) & 1;
      const bool live = w.row0 + quarter < p.N;     // some row of this warp exists
      const int row = w.row0 + tid;
      const float slope = ALIBI ? __ldg(p.slopes + w.head % p.H) * kSfLog2e : 0.0f;
      const float bias = p.bias_vec ? __ldg(p.bias_vec + w.head) * kSfLog2e : p.bias_log2e;
      const int col0 = g ? w.half : 0;
      const int runs = ((g ? w.width : w.half) - col0) >> 5;
      if (!mbar_wait<kPolls>(smem_u32(&bars.s_full), par, cta_err, 30)) break;
      tc_fence_after_sync();
      if (live) {
        const uint32_t t0 = tmem + lane_off + col0;
        for (int r = 0; r < runs; ++r) {
          uint32_t s[32], pk[16];
          tmem_ld32(t0 + r * 32, s);
          tmem_wait_ld();
          const int c = col0 + r * 32;
          // causal: the mask cuts this run if its last column lies past the warp's first row
          sigmoid_cols<32, ALIBI, CAUSAL, fwd_emulate_every(kSfD, CAUSAL)>(
              s, pk, p.scale_log2e, bias, slope, static_cast<float>(row), c, CAUSAL && c + 31 > w.row0 + quarter,
              static_cast<float>(row));
          tmem_st16(t0 + r * 16, pk);
        }
        tmem_wait_st();
      }
      tc_fence_before_sync();
      mbar_arrive(smem_u32(&bars.p_full));

      // O: 32 of the 64 columns per group
      if (!mbar_wait<kPolls>(smem_u32(&bars.o_full), par, cta_err, 31)) break;
      tc_fence_after_sync();
      if (live) {
        uint32_t o[32];
        tmem_ld32(tmem + lane_off + w.o_col + g * 32, o);
        tmem_wait_ld();
        uint8_t* row_ptr = smem + kSfO + tid * 128;
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
          uint4 val;
          val.x = pack_bf16x2(__uint_as_float(o[8 * q4 + 0]), __uint_as_float(o[8 * q4 + 1]));
          val.y = pack_bf16x2(__uint_as_float(o[8 * q4 + 2]), __uint_as_float(o[8 * q4 + 3]));
          val.z = pack_bf16x2(__uint_as_float(o[8 * q4 + 4]), __uint_as_float(o[8 * q4 + 5]));
          val.w = pack_bf16x2(__uint_as_float(o[8 * q4 + 6]), __uint_as_float(o[8 * q4 + 7]));
          *reinterpret_cast<uint4*>(row_ptr + (((g * 4 + q4) ^ (tid & 7)) * 16)) = val;
        }
      }
      tc_fence_before_sync();
      mbar_arrive(smem_u32(&bars.o_empty));
      fence_proxy_async_smem();
      named_barrier_sync<1, kSfActThreads>();
      if (threadIdx.x == 0) {
        tma_store_3d(&tmO, smem_base + kSfO, 0, w.row0, w.head);   // (rows >= N are clipped)
        tma_commit_group();
        tma_wait_group_read<0>();   // before the next unit's rows are written there
      }
    }
    if (threadIdx.x == 0) tma_wait_group<0>();
  }

  tc_fence_before_sync();
  __syncthreads();
  if (cta_err_slot != 0) {
    if (threadIdx.x == 0) atomicExch(p.status, 400 + cta_err_slot);
    __nanosleep(100000);  // let copies in flight towards this thread block's shared memory land
  }
  if (warp == kSfMmaWarp) tmem_dealloc(tmem, 256);
}

template <bool CAUSAL, bool ALIBI>
int launch_short_fwd_variant(const CUtensorMap (&maps)[4], const ShortFwdParams& sp, int num_sms, cudaStream_t stream,
                             cudaError_t* cuda_err) {
  auto kernel = sigattn_short_fwd_bf16_kernel<CAUSAL, ALIBI>;
  // a per-device attribute of the kernel: one bit per device ordinal, ordinals past 63 set it on every launch
  static std::atomic<unsigned long long> configured{0};
  int dev = 0;
  *cuda_err = cudaGetDevice(&dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  const unsigned long long bit = (dev >= 0 && dev < 64) ? (1ull << dev) : 0ull;
  if ((configured.load(std::memory_order_relaxed) & bit) == 0) {
    *cuda_err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSfDynBytes);
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
    configured.fetch_or(bit, std::memory_order_relaxed);
  }
  const int slots = 2 * num_sms;
  *cuda_err = launch_after(kernel, dim3(sp.n_units < slots ? sp.n_units : slots), kSfThreads, kSfDynBytes, stream, 0,
                           maps[0], maps[1], maps[2], maps[3], sp);
  return *cuda_err == cudaSuccess ? SIGATTN_OK : SIGATTN_ERR_CUDA;
}

}  // namespace

bool short_fwd_serves(const Problem& p) {
  return p.D == kSfD && p.N <= kSfMaxN && p.key_rows() == p.N && p.query_pos0() == 0 && p.kv_heads() == p.H &&
         p.seqlens == nullptr && p.row_scale == nullptr && p.cu_seqlens == nullptr && p.split_ws == nullptr && p.acc_only == 0;
}

int launch_short_fwd_bf16(const void* q, const void* k, const void* v, void* o, const Problem& p, int* status,
                          cudaStream_t stream, unsigned long long* launches, cudaError_t* cuda_err) {
  int dev = 0, num_sms = 0;
  *cuda_err = cudaGetDevice(&dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  *cuda_err = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  const int heads = p.B * p.H;
  CUtensorMap maps[4];
  const void* ptrs[4] = {q, k, v, o};
  for (int i = 0; i < 4; ++i) {
    if (make_map_3d(&maps[i], ptrs[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, heads, p.N, kSfD, kSfRows, 64) != 0) {
      *cuda_err = cudaErrorInvalidValue;
      return SIGATTN_ERR_CUDA;
    }
  }
  ShortFwdParams sp = {};
  sp.H = p.H;
  sp.N = p.N;
  sp.n_tiles = (p.N + kSfRows - 1) / kSfRows;
  sp.n_units = heads * sp.n_tiles;
  sp.scale_log2e = p.scale * kSfLog2e;
  sp.bias_log2e = p.bias * kSfLog2e;
  sp.bias_vec = p.bias_vec;
  sp.slopes = p.slopes;
  sp.status = status;
  const bool alibi = p.slopes != nullptr;
  const int rc = p.causal ? (alibi ? launch_short_fwd_variant<true, true>(maps, sp, num_sms, stream, cuda_err)
                                   : launch_short_fwd_variant<true, false>(maps, sp, num_sms, stream, cuda_err))
                          : (alibi ? launch_short_fwd_variant<false, true>(maps, sp, num_sms, stream, cuda_err)
                                   : launch_short_fwd_variant<false, false>(maps, sp, num_sms, stream, cuda_err));
  if (rc == SIGATTN_OK) *launches += 1;
  return rc;
}

}  // namespace sigattn
