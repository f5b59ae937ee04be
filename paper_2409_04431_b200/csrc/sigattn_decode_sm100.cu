// Generation with a cache, bf16: a few query rows per key/value head against a long run of keys.
//
// The rows of all query heads that read one key/value head are one block of R = (query heads per key/value
// head) * N_q consecutive rows of Q and O.  The general forward gives such a block a 128-row tile and spends
// its activation on 128 rows, however few count; here the logits are formed transposed,
//
//     S^T = K_j Q^T      M = 128 keys (tensor-memory lanes), N = R rounded up to 16
//     P                  a thread owns one key and evaluates its R weights -> bf16, shared memory [row][key]
//     O += P V_j         M = 128 rows of which R count (the others read whatever follows in shared memory and
//                        end in lanes nobody reads), N = D
//
// so that the exponentials cost 128 x R instead of 128 x 128 per key tile and the tensor work is small next to
// the time the tile takes to arrive.  What bounds the kernel is then HBM (long caches) or its own latency
// (short ones).
//
// The keys of a head are divided over the thread blocks of a cluster (up to 16, see decode_plan); each keeps its
// partial O in shared memory and the cluster adds the partial rows through distributed shared memory, in rank
// order, and stores bf16.  Sigmoid has no row normalisation, so partial rows are plain summands: no scratch in
// global memory, nothing to clear before and nothing to convert after, and the result does not depend on timing.
// Few heads with long caches are divided over several clusters, whose sums meet in the caller's scratch (fp32
// additions in order of arrival, then a conversion pass).
//
// Measured, one new token per sequence, H = 32, H_kv = 8, D = 128, device time (before: the general forward with
// split keys between a clearing and a conversion launch):
//   B = 8, N_k = 16384   117.5 -> 82 us, 4.6 -> 6.5 TB/s of K and V (the measured copy rate)
//   B = 32, N_k = 4096   115 -> 85 us;   B = 1, N_k = 2000   14.9 -> 8.3 us;   B = 1, N_k = 65536   63 -> 52 us
#include <atomic>

#include "launch.h"
#include "sigattn_internal.h"
#include "sm100_primitives.cuh"
#include "tensor_map.h"
#include "../../include/sigattn.h"

namespace sigattn {
namespace {

using namespace sm100;

constexpr int kDecTile = 128;               // keys per tile
constexpr int kDecMaxRows = 64;             // packed query rows per key/value head
constexpr int kDecActThreads = 128;         // thread = key
constexpr int kDecThreads = kDecActThreads + 64;
constexpr int kDecLoadWarp = 4;
constexpr int kDecMmaWarp = 5;
constexpr int kDecMaxStages = 12;
constexpr uint32_t kDecTmemCols = 256;      // S^T twice (64 columns each at most), O (D columns)
constexpr int kDecMaxSmem = 220 * 1024;     // dynamic shared memory of one thread block that has an SM to itself
constexpr float kDecLog2e = 1.4426950408889634f;

struct DecodeBarriers {
  uint64_t q_full, o_full;
  uint64_t s_full[2], p_full[2], p_empty[2];
  uint64_t kv_full[kDecMaxStages], kv_empty[kDecMaxStages];
};

struct DecodeParams {
  int rows, rows16;       // packed rows per key/value head, and rounded up to 16
  int n_q, group;         // rows per query head, query heads per key/value head
  int n_tiles, n_keys;    // key tiles and keys of a head
  int pos0;               // position of query 0 relative to key 0
  int causal;
  int stages;             // key/value ring
  int cluster;            // thread blocks per cluster
  float* acc;             // several clusters per head: their sums are added here (fp32, cleared), else nullptr
  float scale_log2e, bias_log2e;
  const float* bias_vec;  // one bias per (batch, query head), or nullptr
  const float* slopes;    // one slope per query head, or nullptr
  int H;                  // query heads
  void* o;
  int* status;
};

// One weight: P = 1 / (1 + 2^-a).  NaN stays NaN: a cache row that holds one is seen in the result.
__device__ __forceinline__ float decode_weight(float a) {
  return rcp_approx(1.0f + ex2_approx(fmin_nan(-a, 120.0f)));
}

// All polls of a wait unrolled: the kernel is one short chain of waits, each code fetched once, and a loop answers later
// (us, loop / unrolled: B1 H32 H_kv8 300 keys 5.83 / 5.80, 5000 keys 8.65 / 8.58, B8 H32 four queries 1500 keys D64
// 17.3 / 17.0; from 16384 keys on the same).
constexpr int kDecPolls = 64;

template <int D, bool ALIBI>
__global__ void __launch_bounds__(kDecThreads, 1)
sigattn_decode_bf16_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                           const __grid_constant__ CUtensorMap tmV, const DecodeParams p) {
  constexpr int kPanels = D / 64;
  constexpr int kPanelBytes = kDecTile * 128;
  constexpr int kTileBytes = kPanels * kPanelBytes;
  extern __shared__ uint8_t smem_raw[];
  __shared__ DecodeBarriers bars;
  __shared__ __align__(16) float row_bias[kDecMaxRows], row_slope[kDecMaxRows];   // both times log2 e
  __shared__ __align__(16) int row_pos[kDecMaxRows], row_last[kDecMaxRows];   // position, and of the last key it sees
  __shared__ uint32_t tmem_base_slot;
  __shared__ int cta_err_slot;
  volatile int* cta_err = &cta_err_slot;

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem_base = smem_u32(smem);
  const int warp = threadIdx.x >> 5;
  const int rows16 = p.rows16;
  // shared memory: P twice (rows16 x 128 keys), Q (rows16 x D), then the ring.  The products that read P take
  // 128 rows from its start, i.e. up to 16 KB past it: always inside the ring.
  const uint32_t p_panel = rows16 * 128, p_bytes = 2 * p_panel;
  const uint32_t q_panel = rows16 * 128;
  const uint32_t q_off = 2 * p_bytes, ring_off = q_off + kPanels * q_panel;

  const uint32_t n_split = p.cluster;                       // thread blocks of a cluster
  const uint32_t split = n_split > 1 ? cluster_ctarank() : 0u;
  const int head = blockIdx.y;                              // (batch, key/value head)
  const int share = blockIdx.x, shares = gridDim.x;         // the clusters of a head divide its key tiles
  const int tile0 = share * p.n_tiles / shares;
  const int n = (share + 1) * p.n_tiles / shares - tile0;   // key tiles of this thread block, >= 1

  if (threadIdx.x == 0) {
    cta_err_slot = 0;
    mbar_init(smem_u32(&bars.q_full), 1);
    mbar_init(smem_u32(&bars.o_full), 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&bars.s_full[s]), 1);
      mbar_init(smem_u32(&bars.p_full[s]), kDecActThreads);
      mbar_init(smem_u32(&bars.p_empty[s]), 1);
    }
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&bars.kv_full[s]), 1);
      mbar_init(smem_u32(&bars.kv_empty[s]), 1);
    }
    fence_mbar_init();
  }
  if (warp == kDecLoadWarp && elect_one()) {
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
  }
  if (warp == kDecMmaWarp) {
    tmem_alloc(smem_u32(&tmem_base_slot), kDecTmemCols);
    tmem_relinquish();
  }
  grid_dependency_wait();
  if (threadIdx.x < rows16) {
    // rows past the end only fill the tile; their weights are never used
    const int r = min(static_cast<int>(threadIdx.x), p.rows - 1);
    const int g = r / p.n_q;
    const int q_head = head * p.group + g;
    row_bias[threadIdx.x] = p.bias_vec ? __ldg(p.bias_vec + q_head) * kDecLog2e : p.bias_log2e;
    if (ALIBI) row_slope[threadIdx.x] = __ldg(p.slopes + q_head % p.H) * kDecLog2e;
    row_pos[threadIdx.x] = r - g * p.n_q + p.pos0;
    row_last[threadIdx.x] = p.causal ? r - g * p.n_q + p.pos0 : p.n_keys - 1;
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_base_slot;
  grid_dependency_trigger();   // (after the allocation of tensor memory: see launch.h)
  const uint32_t tmem_o = tmem + 128;

  if (warp == kDecLoadWarp) {
    if ((threadIdx.x & 31) == 0) {
      mbar_arrive_expect_tx(smem_u32(&bars.q_full), kPanels * q_panel);
      for (int pn = 0; pn < kPanels; ++pn)
        tma_load_3d(smem_base + q_off + pn * q_panel, &tmQ, smem_u32(&bars.q_full), pn * 64, 0, head);
      // ring order K_0, V_0, K_1, V_1, ...
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int i = 0; ok && i < 2 * n; ++i) {
        ok = mbar_wait<kDecPolls>(smem_u32(&bars.kv_empty[stage]), phase ^ 1, cta_err, 10);
        if (!ok) break;
        const uint32_t bar = smem_u32(&bars.kv_full[stage]);
        mbar_arrive_expect_tx(bar, kTileBytes);
        const CUtensorMap* tm = (i & 1) ? &tmV : &tmK;
#pragma unroll
        for (int pn = 0; pn < kPanels; ++pn)
          tma_load_3d(smem_base + ring_off + stage * kTileBytes + pn * kPanelBytes, tm, bar, pn * 64,
                      (tile0 + (i >> 1)) * kDecTile, head);
        if (++stage == p.stages) { stage = 0; phase ^= 1; }
      }
    }
    __syncwarp();
  } else if (warp == kDecMmaWarp) {
    if (elect_one()) {
      const uint32_t idesc_s = make_idesc_bf16(kDecTile, 0, 0, 0) | (static_cast<uint32_t>(rows16 >> 3) << 17);
      constexpr uint32_t kIdescPV = make_idesc_bf16(kDecTile, D, 0, 1);
      const uint64_t q_desc = make_smem_desc_sw128(smem_base + q_off, 16, 1024);
      // ring cursors: K tiles and V tiles are consumed two and one steps apart
      int k_stage = 0, v_stage = 1;
      uint32_t k_phase = 0, v_phase = 0;
      auto advance = [&](int& stage, uint32_t& phase) {
        stage += 2;
        if (stage >= p.stages) { stage -= p.stages; phase ^= 1; }
      };
      auto issue_s = [&](int j) -> bool {
        if (!mbar_wait<kDecPolls>(smem_u32(&bars.kv_full[k_stage]), k_phase, cta_err, 20)) return false;
        tc_fence_after_sync();
        const uint64_t k_desc = make_smem_desc_sw128(smem_base + ring_off + k_stage * kTileBytes, 16, 1024);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          const uint32_t in_panel = (ks & 3) * 32;
          umma_ss(tmem + (j & 1) * 64, desc_advance(k_desc, (ks >> 2) * kPanelBytes + in_panel),
                  desc_advance(q_desc, (ks >> 2) * q_panel + in_panel), idesc_s, ks > 0);
        }
        umma_commit(smem_u32(&bars.s_full[j & 1]));
        umma_commit(smem_u32(&bars.kv_empty[k_stage]));
        advance(k_stage, k_phase);
        return true;
      };
      bool ok = mbar_wait<kDecPolls>(smem_u32(&bars.q_full), 0, cta_err, 21) && issue_s(0) && (n < 2 || issue_s(1));
      for (int j = 0; ok && j < n; ++j) {
        ok = mbar_wait<kDecPolls>(smem_u32(&bars.kv_full[v_stage]), v_phase, cta_err, 22) &&
             mbar_wait<kDecPolls>(smem_u32(&bars.p_full[j & 1]), (j >> 1) & 1, cta_err, 23);
        if (!ok) break;
        tc_fence_after_sync();
        const uint64_t v_desc = make_smem_desc_sw128(smem_base + ring_off + v_stage * kTileBytes, kPanelBytes, 1024);
        const uint64_t p_desc = make_smem_desc_sw128(smem_base + (j & 1) * p_bytes, 16, 1024);
#pragma unroll
        for (int ks = 0; ks < kDecTile / 16; ++ks)
          umma_ss(tmem_o, desc_advance(p_desc, (ks >> 2) * p_panel + (ks & 3) * 32), desc_advance(v_desc, ks * 2048),
                  kIdescPV, (j > 0 || ks > 0));
        umma_commit(smem_u32(&bars.kv_empty[v_stage]));
        umma_commit(smem_u32(&bars.p_empty[j & 1]));
        advance(v_stage, v_phase);
        // (the activation has read S^T of this tile: its columns may be written again)
        if (j + 2 < n) ok = issue_s(j + 2);
      }
      if (ok) umma_commit(smem_u32(&bars.o_full));
    }
    __syncwarp();
  } else {
    const int key = threadIdx.x;   // row of the key tile = tensor-memory lane
    const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t p_lo = (key & 7) * 2, p_chunk = (key & 63) >> 3;
    bool ok = true;
    for (int j = 0; ok && j < n; ++j) {
      const int buf = j & 1;
      ok = mbar_wait<kDecPolls>(smem_u32(&bars.s_full[buf]), (j >> 1) & 1, cta_err, 30) &&
           (j < 2 || mbar_wait<kDecPolls>(smem_u32(&bars.p_empty[buf]), ((j >> 1) & 1) ^ 1, cta_err, 31));
      if (!ok) break;
      tc_fence_after_sync();
      const int key_pos = (tile0 + j) * kDecTile + key;
      // the mask cuts only tiles that reach beyond the first query's position, or beyond the last key (such rows read as
      // zeros, and a query that holds Inf makes NaN of them)
      const int seen = p.causal ? p.pos0 + 1 : p.n_keys;   // (causal: pos0 + 1 <= n_keys)
      const bool cut = (tile0 + j + 1) * kDecTile > seen;
      uint8_t* p_col = smem + buf * p_bytes + (key >> 6) * p_panel + p_lo;
      // sixteen rows at a time, the rows past the end with them: straight-line code, so that the exponentials
      // and reciprocals of different rows overlap (with a test per row a tile of 32 rows took 5300 cycles)
      for (int r0 = 0; r0 < rows16; r0 += 16) {
        uint32_t s[16];
        tmem_ld16(tmem + buf * 64 + lane_off + r0, s);
        tmem_wait_ld();
        float w[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) w[e] = fmaf(__uint_as_float(s[e]), p.scale_log2e, row_bias[r0 + e]);
        if (ALIBI) {
#pragma unroll
          for (int e = 0; e < 16; ++e)
            w[e] = fmaf(-row_slope[r0 + e], fabsf(static_cast<float>(row_pos[r0 + e] - key_pos)), w[e]);
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) w[e] = decode_weight(w[e]);
        if (cut) {
#pragma unroll
          for (int e = 0; e < 16; ++e)
            if (key_pos > row_last[r0 + e]) w[e] = 0.0f;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e)
          *reinterpret_cast<__nv_bfloat16*>(p_col + (r0 + e) * 128 + ((p_chunk ^ (e & 7)) * 16)) = __float2bfloat16_rn(w[e]);
      }
      fence_proxy_async_smem();
      tc_fence_before_sync();
      mbar_arrive(smem_u32(&bars.p_full[buf]));
    }
    // partial O: lanes 0 ... rows - 1 -> shared memory [row][D], fp32, over the ring (every load has landed and
    // every product that read it is done)
    if (ok && warp * 32 < p.rows) {
      ok = mbar_wait<kDecPolls>(smem_u32(&bars.o_full), 0, cta_err, 32);
      if (ok) {
        tc_fence_after_sync();
        float* dst = reinterpret_cast<float*>(smem + ring_off) + key * D;
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t o[32];
          tmem_ld32(tmem_o + lane_off + c * 32, o);
          tmem_wait_ld();
          if (key < p.rows) {
#pragma unroll
            for (int e = 0; e < 8; ++e)   // 16-byte pieces in a row-dependent order: the lanes spread over the banks
              *reinterpret_cast<uint4*>(dst + ((c * 8 + e) ^ (key & 7)) * 4) =
                  make_uint4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]);
          }
        }
      }
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (n_split > 1) cluster_sync();
  {
    // rank c adds every n_split-th run of the rows over all ranks, in rank order, and stores it
    const uint32_t part = smem_base + ring_off;
    const int n_vec4 = p.rows * (D / 4);
    uint2* o = static_cast<uint2*>(p.o) + static_cast<size_t>(head) * n_vec4;
    for (int i = static_cast<int>(split) * kDecThreads + threadIdx.x; i < n_vec4; i += static_cast<int>(n_split) * kDecThreads) {
      float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      const uint32_t piece = part + (i ^ ((i / (D / 4)) & 7)) * 16;
      for (uint32_t c = 0; c < n_split; ++c) {
        const float4 v = ld_cluster_v4(map_to_cta(piece, c));
        acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
      }
      if (p.acc != nullptr)
        red_add_v4_f32(p.acc + (static_cast<size_t>(head) * n_vec4 + i) * 4, acc.x, acc.y, acc.z, acc.w);
      else
        o[i] = make_uint2(pack_bf16x2(acc.x, acc.y), pack_bf16x2(acc.z, acc.w));
    }
  }
  if (n_split > 1) cluster_sync();   // nobody leaves while its partial rows may still be read
  if (cta_err_slot != 0) {
    if (threadIdx.x == 0) atomicExch(p.status, 300 + cta_err_slot);
    __nanosleep(100000);  // let copies in flight towards this thread block's shared memory land
  }
  if (warp == kDecMmaWarp) tmem_dealloc(tmem, kDecTmemCols);
}

struct DecodePlan {
  int cluster;   // thread blocks per cluster
  int parts;     // clusters per head
};

template <int D, bool ALIBI>
int launch_decode_variant(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                          const DecodeParams& dp, int shares, int heads, size_t smem_bytes, cudaStream_t stream,
                          cudaError_t* cuda_err) {
  auto kernel = sigattn_decode_bf16_kernel<D, ALIBI>;
  // per-device attributes of the kernel: one bit per device ordinal, ordinals past 63 set them on every launch
  static std::atomic<unsigned long long> configured{0};
  int dev = 0;
  *cuda_err = cudaGetDevice(&dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  const unsigned long long bit = (dev >= 0 && dev < 64) ? (1ull << dev) : 0ull;
  if ((configured.load(std::memory_order_relaxed) & bit) == 0) {
    *cuda_err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDecMaxSmem);
    if (*cuda_err == cudaSuccess)
      *cuda_err = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
    configured.fetch_or(bit, std::memory_order_relaxed);
  }
  *cuda_err = launch_after(kernel, dim3(static_cast<unsigned>(shares), static_cast<unsigned>(heads)), kDecThreads, smem_bytes,
                           stream, static_cast<unsigned>(dp.cluster), tmQ, tmK, tmV, dp);
  return *cuda_err == cudaSuccess ? SIGATTN_OK : SIGATTN_ERR_CUDA;
}

// How the keys of a head are divided.  The aim is 120 to 256 thread blocks; within that a single cluster per head
// is best, because it needs neither scratch nor further launches, up to the point where its thread blocks get so
// many tiles that the idle SMs cost more (us, one token, D = 128; single cluster of 8 or 16 / clusters of 4
// with sums in scratch):
//   8 heads, 16 tiles 8.3 / 12.3;  128 tiles 23.0 (16 blocks: 28.8, not all clusters resident at once) / 24.6;
//   512 tiles 69.1 / 52.4;  4 heads, 64 tiles 12.3 (16) / 12.4;  512 tiles 41.8 (16) / 35.4;
//   2 heads, 128 tiles 16.5 (16) / 14.4;  1 head, 512 tiles 39.2 (16) / 21.5;
//   24 heads, 64 tiles: clusters of 4 24.7, of 8 25.1;  32 heads of 16 tiles: 8 12.5, 4 13.6;  64 heads of 128: 2
DecodePlan decode_plan(long long heads, int n_tiles) {
  const int most = heads <= 4 ? 16 : 8;
  DecodePlan d = {1, 1};
  while (d.cluster < most && 2 * d.cluster <= n_tiles && heads * d.cluster < 96) d.cluster *= 2;
  const int tiles = (n_tiles + d.cluster - 1) / d.cluster;
  if (heads * d.cluster < 96 && tiles > (d.cluster == 16 ? 8 : 16)) {
    d.cluster = 4;
    // (128 thread blocks: with 144 not every cluster of four is resident at once, and the 4-head case takes 51.4)
    d.parts = static_cast<int>(128 / (4 * heads));
    if (4 * d.parts > n_tiles) d.parts = n_tiles / 4;   // (every thread block has a tile)
  }
  return d;
}

}  // namespace

bool decode_kernel_serves(const Problem& p) {
  const int group = p.H / p.kv_heads();
  return static_cast<long long>(p.N) * group <= kDecMaxRows && p.seqlens == nullptr && p.row_scale == nullptr &&
         p.cu_seqlens == nullptr && p.acc_only == 0;
}

int launch_decode_bf16(const void* q, const void* k, const void* v, void* o, const Problem& p, int* status,
                       cudaStream_t stream, unsigned long long* launches, cudaError_t* cuda_err) {
  const int group = p.H / p.kv_heads();
  const int heads = p.B * p.kv_heads();
  DecodeParams dp = {};
  dp.rows = p.N * group;
  dp.rows16 = (dp.rows + 15) & ~15;
  dp.n_q = p.N;
  dp.group = group;
  dp.n_keys = p.key_rows();
  dp.n_tiles = (dp.n_keys + kDecTile - 1) / kDecTile;
  dp.pos0 = p.query_pos0();
  dp.causal = p.causal;
  dp.scale_log2e = p.scale * kDecLog2e;
  dp.bias_log2e = p.bias * kDecLog2e;
  dp.bias_vec = p.bias_vec;
  dp.slopes = p.slopes;
  dp.H = p.H;
  dp.o = o;
  dp.status = status;
  const DecodePlan plan = decode_plan(heads, dp.n_tiles);
  const int shares = plan.cluster * plan.parts;
  dp.cluster = plan.cluster;
  // The ring: everything that fits when each SM has one thread block, half of that when two share an SM.
  const int tile_bytes = kDecTile * p.D * 2;
  const int fixed = 4 * dp.rows16 * 128 + dp.rows16 * p.D * 2 + 1024;
  const int most = 2 * ((dp.n_tiles + shares - 1) / shares);   // nothing to gain beyond a thread block's own tiles
  const bool two_per_sm = static_cast<long long>(heads) * shares > 148 && (kDecMaxSmem / 2 - fixed) / tile_bytes >= 3;
  int stages = ((two_per_sm ? kDecMaxSmem / 2 : kDecMaxSmem) - fixed) / tile_bytes;   // (three at least: K_0, V_0, K_1)
  if (stages > most) stages = most;
  if (stages > kDecMaxStages) stages = kDecMaxStages;
  dp.stages = stages;
  const size_t smem_bytes = static_cast<size_t>(fixed) + static_cast<size_t>(stages) * tile_bytes;

  CUtensorMap tmQ, tmK, tmV;
  if (make_map_3d(&tmQ, q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, heads, dp.rows, p.D, dp.rows16, 64) != 0 ||
      make_map_3d(&tmK, k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, heads, p.key_rows(), p.D, kDecTile, 64) != 0 ||
      make_map_3d(&tmV, v, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, heads, p.key_rows(), p.D, kDecTile, 64) != 0) {
    *cuda_err = cudaErrorInvalidValue;
    return SIGATTN_ERR_CUDA;
  }
  const size_t n_elems = static_cast<size_t>(heads) * dp.rows * p.D;
  if (plan.parts > 1) {
    dp.acc = p.split_ws;
    *cuda_err = cudaMemsetAsync(dp.acc, 0, n_elems * sizeof(float), stream);
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  }
#define SIGATTN_DECODE_CASE(DD, AA) launch_decode_variant<DD, AA>(tmQ, tmK, tmV, dp, shares, heads, smem_bytes, stream, cuda_err)
  const bool alibi = p.slopes != nullptr;
  const int rc = p.D == 128 ? (alibi ? SIGATTN_DECODE_CASE(128, true) : SIGATTN_DECODE_CASE(128, false))
                            : (alibi ? SIGATTN_DECODE_CASE(64, true) : SIGATTN_DECODE_CASE(64, false));
#undef SIGATTN_DECODE_CASE
  if (rc != SIGATTN_OK) return rc;
  *launches += 1;
  if (plan.parts > 1) return launch_acc_to_bf16(p.split_ws, o, n_elems, 1.0f, stream, launches, cuda_err);
  return SIGATTN_OK;
}

}  // namespace sigattn
