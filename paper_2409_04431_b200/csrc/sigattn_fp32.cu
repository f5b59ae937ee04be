// float32 debug path on CUDA cores: the definition evaluated with exact expf and a
// true division, fp32 FMA accumulation, no tensor cores (TF32 would cost 1e-3 of
// accuracy).  A thread block owns four rows (queries for the forward and dQ, keys for dK and
// dV) and walks the other side in tiles of 64 rows that are copied to shared memory ahead of
// use; nothing is shared between blocks, so every tensor output is deterministic (the optional
// bias gradient is a sum over all blocks of a head and is added with fp32 atomics).
//
// The sizes this path is used at (one to a few heads, N up to about 500) are bound by latency:
// launches, one trip to memory, and the dependent sums.  Hence 256 threads for four rows (a
// weight per thread and tile, four partial sums per dot product, the keys of the second
// product divided over thread groups), both tiles of the next step in flight, and one launch
// for the whole backward.  Measured, B = H = 1, N = 128, D = 64, against one block per row
// with every thread reading its own row from global memory: forward 14.4 -> 6.2 us, backward (two
// launches before) 30.8 -> 8.3 us.
//
// N counts query rows, N_k key/value rows; query i has position i + off relative to key 0
// (off = N_k - N when the queries are the last N positions, 0 for self-attention; any value,
// also negative, for a shard of keys and values).
//
// Forward: Eq. 3 / Algorithm 1.  Backward: the sigmoid column of the forward/backward
// table in Appendix F.1 / Algorithm 2, with the factor scale = 1/sqrt(d) in dQ and dK.
#include <atomic>

#include "launch.h"
#include "sigattn_internal.h"
#include "../../include/sigattn.h"

namespace sigattn {
namespace {

constexpr int kThreads = 256;
constexpr int kOwn = 4;      // rows a block owns
constexpr int kTile = 64;    // rows of the other side per step
constexpr int kSlices = kThreads / kTile;   // = kOwn: one weight per thread and step
static_assert(kSlices == kOwn, "a thread evaluates one weight of each tile");

__device__ __forceinline__ float sigmoid_exact(float x) { return 1.0f / (1.0f + expf(-x)); }

// P (1 - P) evaluated as sigmoid(x) * sigmoid(-x): the same quantity (1 - sigmoid(x) =
// sigmoid(-x)), but without the cancellation of 1 - P when P rounds to 1.
__device__ __forceinline__ float sigmoid_slope(float x) { return sigmoid_exact(x) * sigmoid_exact(-x); }

// Batch stored without padding: the sequence that owns `row` (largest s with cu[s] <= row).
__device__ __forceinline__ int seq_of_row_fp32(const int* __restrict__ cu, int n_seqs, int row) {
  int lo = 0, hi = n_seqs;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (cu[mid] <= row) lo = mid; else hi = mid;
  }
  return lo;
}

struct Fp32Args {
  const float *q, *k, *v, *d_o;
  float *o, *dq, *dk, *dv;
  int B, H, H_kv, N, N_k, off, causal;
  float scale, bias;
  const float *slopes, *bias_vec, *row_scale;
  float* dbias;
  const int *seqlens, *cu;
  int n_seqs;
  int dq_blocks;   // backward: blocks below this number own query rows, the others key rows
};

enum Fp32Pass { kForward, kGradQ, kGradKV };

// Shared memory of a pass: the tile pairs (double-buffered) and the block's own rows.  Rows are padded by four
// floats, so that the 16-byte reads of different rows fall into different banks.
template <int D>
struct Fp32Smem {
  static constexpr int kStride = D + 4;
  float x[2][kTile * kStride], y[2][kTile * kStride];
  float own_a[kOwn][D], own_b[kOwn][D];
  float w1[kOwn][kTile], w2[kOwn][kTile];
  float4 part[2][kThreads];
};

__device__ __forceinline__ void copy_async16(float* dst, const float* src, bool valid) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  const int n = valid ? 16 : 0;   // rows that do not exist are filled with zeros
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

template <int D>
__device__ __forceinline__ float dot_rows(const float* a, const float* b) {
  float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 8
  for (int d = 0; d < D; d += 4) {
    const float4 u = *reinterpret_cast<const float4*>(a + d), w = *reinterpret_cast<const float4*>(b + d);
    s.x = fmaf(u.x, w.x, s.x);
    s.y = fmaf(u.y, w.y, s.y);
    s.z = fmaf(u.z, w.z, s.z);
    s.w = fmaf(u.w, w.w, s.w);
  }
  return (s.x + s.y) + (s.z + s.w);
}

// One pass of one block.  Own rows: queries (forward, dQ) or keys (dK, dV); tiles: the rows on the other side.
//   s = <own_a, x>, dp = <own_b, y>;  forward: sum P y;  dQ: sum dS x;  dK: sum dS x and dV: sum P y.
// `head`: (batch, query head) for the first two, (batch, key/value head) for the last.
template <int D, Fp32Pass PASS>
__device__ void fp32_pass(const Fp32Args& p, Fp32Smem<D>& sm, int row0, int head) {
  const int t = threadIdx.x, slice = t / kTile, lane = t % kTile;
  const int group = p.H / p.H_kv;
  const int n_own = PASS == kGradKV ? p.N_k : p.N, n_other = PASS == kGradKV ? p.N : p.N_k;
  const int batch = PASS == kGradKV ? head / p.H_kv : head / p.H;
  const int kv_head = PASS == kGradKV ? head : batch * p.H_kv + (head % p.H) / group;
  const float* own_a = (PASS == kGradKV ? p.k : p.q) + static_cast<size_t>(head) * n_own * D;
  const float* own_b = (PASS == kGradKV ? p.v : p.d_o) + static_cast<size_t>(head) * n_own * D;

  for (int e = t; e < kOwn * D; e += kThreads) {
    const int r = e / D, d = e % D, row = row0 + r;
    const bool there = row < n_own;
    const size_t at = static_cast<size_t>(row) * D + d;
    sm.own_a[r][d] = there ? own_a[at] : 0.0f;
    if (PASS != kForward) {
      float b = there ? own_b[at] : 0.0f;
      if (PASS == kGradQ && p.row_scale && there) b *= p.row_scale[row];   // O = r (P V): the row's factor passes to dO
      sm.own_b[r][d] = b;
    }
  }

  // The rows [lo, hi) of the other side that a given own row meets.
  const int n_valid = p.seqlens ? max(0, min(p.N, p.seqlens[batch])) : n_other;
  auto range = [&](int row, int& lo, int& hi, int& seq) {
    lo = 0;
    hi = 0;
    seq = 0;
    if (row >= n_own || (p.seqlens && row >= n_valid)) return;
    hi = n_valid;
    if (p.causal) {
      if (PASS == kGradKV) lo = max(0, row - p.off);
      else hi = min(hi, max(0, row + p.off + 1));
    }
    if (p.cu) {   // batch without padding: only rows of the own row's sequence
      seq = seq_of_row_fp32(p.cu, p.n_seqs, row);
      lo = max(lo, p.cu[seq]);
      hi = min(hi, p.cu[seq + 1]);
    }
  };
  int lo, hi, seq;                      // of the own row whose weights this thread evaluates
  range(row0 + slice, lo, hi, seq);
  int first = n_other, last = 0;        // union over the block's own rows
  int all_lo = 0, all_hi = n_other;     // and what all of them meet
  for (int r = 0; r < kOwn; ++r) {
    int l, h, s;
    range(row0 + r, l, h, s);
    if (row0 + r < n_own) {
      all_lo = max(all_lo, l);
      all_hi = min(all_hi, h);
    }
    if (l < h) {
      first = min(first, l);
      last = max(last, h);
    }
  }
  const int tiles = last > first ? (last - first + kTile - 1) / kTile : 0;
  const int heads = PASS == kGradKV ? group : 1;
  const int steps = tiles * heads;

  auto load = [&](int step) {
    const int g = step / tiles, base_row = first + (step - g * tiles) * kTile, buf = step & 1;
    const int other = PASS == kGradKV ? batch * p.H + (head % p.H_kv) * group + g : kv_head;
    const size_t base = static_cast<size_t>(other) * n_other * D;
    const float* x = (PASS == kGradKV ? p.q : p.k) + base;
    const float* y = (PASS == kGradKV ? p.d_o : p.v) + base;
    for (int e = t; e < kTile * (D / 4); e += kThreads) {
      const int r = e / (D / 4), d = (e % (D / 4)) * 4, row = base_row + r;
      const bool there = row < last;
      const size_t at = static_cast<size_t>(there ? row : 0) * D + d;
      copy_async16(&sm.x[buf][r * Fp32Smem<D>::kStride + d], x + at, there);
      copy_async16(&sm.y[buf][r * Fp32Smem<D>::kStride + d], y + at, there);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  // second product: thread = four columns of one own row, over a share of the tile's rows
  constexpr int kColGroups = D / 4, kShares = kThreads / kColGroups / kOwn;   // 4 shares at D = 64, 2 at D = 128
  const int c4 = (t % kColGroups) * 4, own = (t / kColGroups) % kOwn, share = t / kColGroups / kOwn;
  int own_lo, own_hi, own_seq;   // what that row meets
  range(row0 + own, own_lo, own_hi, own_seq);
  float4 acc1 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), acc2 = acc1;
  float ds_sum = 0.0f;
  int bias_head = -1;
  float bias = p.bias, slope = 0.0f;

  if (steps > 0) load(0);
  for (int step = 0; step < steps; ++step) {
    if (step + 1 < steps) {
      load(step + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const int g = step / tiles, base_row = first + (step - g * tiles) * kTile, buf = step & 1;
    const int q_head = PASS == kGradKV ? batch * p.H + (head % p.H_kv) * group + g : head;
    if (q_head != bias_head) {
      bias_head = q_head;
      slope = p.slopes ? p.slopes[q_head % p.H] : 0.0f;
      bias = p.bias_vec ? p.bias_vec[p.cu ? seq * p.H + q_head : q_head] : p.bias;
    }
    {
      const int other = base_row + lane;
      const int i = PASS == kGradKV ? other : row0 + slice, j = PASS == kGradKV ? row0 + slice : other;
      const float s = dot_rows<D>(sm.own_a[slice], &sm.x[buf][lane * Fp32Smem<D>::kStride]);
      float w1 = 0.0f, w2 = 0.0f;
      const bool live = other >= lo && other < hi;
      const float x = fmaf(p.scale, s, bias) - slope * fabsf(static_cast<float>(i + p.off - j));
      if (PASS == kForward) {
        if (live) w1 = sigmoid_exact(x);
      } else {
        const float dp = dot_rows<D>(sm.own_b[slice], &sm.y[buf][lane * Fp32Smem<D>::kStride]);
        if (live) {
          w1 = sigmoid_slope(x) * dp;
          if (PASS == kGradKV) {
            const float r = p.row_scale ? p.row_scale[i] : 1.0f;   // both products see r dO
            w1 *= r;
            w2 = r * sigmoid_exact(x);
          }
        }
        if (PASS == kGradQ) ds_sum += w1;
      }
      sm.w1[slice][lane] = w1;
      if (PASS == kGradKV) sm.w2[slice][lane] = w2;
    }
    __syncthreads();
    const float* first_src = PASS == kForward ? sm.y[buf] : sm.x[buf];
    auto add = [&](int r) {
      const float w = sm.w1[own][r];
      const float4 u = *reinterpret_cast<const float4*>(&first_src[r * Fp32Smem<D>::kStride + c4]);
      acc1.x = fmaf(w, u.x, acc1.x);
      acc1.y = fmaf(w, u.y, acc1.y);
      acc1.z = fmaf(w, u.z, acc1.z);
      acc1.w = fmaf(w, u.w, acc1.w);
      if (PASS == kGradKV) {
        const float z = sm.w2[own][r];
        const float4 y = *reinterpret_cast<const float4*>(&sm.y[buf][r * Fp32Smem<D>::kStride + c4]);
        acc2.x = fmaf(z, y.x, acc2.x);
        acc2.y = fmaf(z, y.y, acc2.y);
        acc2.z = fmaf(z, y.z, acc2.z);
        acc2.w = fmaf(z, y.w, acc2.w);
      }
    };
    // What lies outside the own row's range is not touched: it may hold Inf or NaN, whose product with a weight of 0
    // counts.  (Rows past `last` hold zeros.  Bounds in every tile cost 7 to 11 %.)
    const int r0 = share * (kTile / kShares), r1 = r0 + kTile / kShares;
    if (base_row >= all_lo && min(base_row + kTile, last) <= all_hi) {
#pragma unroll 8
      for (int e = 0; e < kTile / kShares; ++e) add(r0 + e);
    } else {
#pragma unroll 4
      for (int r = max(r0, own_lo - base_row), end = min(r1, own_hi - base_row); r < end; ++r) add(r);
    }
    __syncthreads();   // the tile's buffer and the weights may be overwritten
  }

  // the shares of a row, added in order
  sm.part[0][t] = acc1;
  if (PASS == kGradKV) sm.part[1][t] = acc2;
  __syncthreads();
  const int row = row0 + own;
  if (share == 0 && row < n_own) {
    auto total = [&](const float4* part) {
      float4 s = part[t];
#pragma unroll
      for (int c = 1; c < kShares; ++c) {
        const float4 u = part[t + c * kColGroups * kOwn];
        s.x += u.x;
        s.y += u.y;
        s.z += u.z;
        s.w += u.w;
      }
      return s;
    };
    const size_t at = (static_cast<size_t>(head) * n_own + row) * D + c4;
    float4 s = total(sm.part[0]);
    const float mul = PASS == kForward ? (p.row_scale ? p.row_scale[row] : 1.0f) : p.scale;
    s = make_float4(mul * s.x, mul * s.y, mul * s.z, mul * s.w);
    *reinterpret_cast<float4*>((PASS == kForward ? p.o : PASS == kGradQ ? p.dq : p.dk) + at) = s;
    if (PASS == kGradKV) *reinterpret_cast<float4*>(p.dv + at) = total(sm.part[1]);
  }
  if (PASS == kGradQ && p.dbias) {   // d(bias): sum of dS over the row, then over the rows (atomics)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ds_sum += __shfl_xor_sync(0xffffffffu, ds_sum, o);
    if ((t & 31) == 0 && row0 + slice < n_own) atomicAdd(p.dbias + (p.cu ? seq * p.H + head : head), ds_sum);
  }
}

template <int D>
__global__ void __launch_bounds__(kThreads) fwd_fp32_kernel(const Fp32Args p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int blocks = (p.N + kOwn - 1) / kOwn, head = blockIdx.x / blocks;
  grid_dependency_wait();
  grid_dependency_trigger();
  fp32_pass<D, kForward>(p, *reinterpret_cast<Fp32Smem<D>*>(smem_raw), (blockIdx.x - head * blocks) * kOwn, head);
}

template <int D>
__global__ void __launch_bounds__(kThreads) bwd_fp32_kernel(const Fp32Args p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  Fp32Smem<D>& sm = *reinterpret_cast<Fp32Smem<D>*>(smem_raw);
  grid_dependency_wait();
  grid_dependency_trigger();
  if (static_cast<int>(blockIdx.x) < p.dq_blocks) {
    const int blocks = (p.N + kOwn - 1) / kOwn, head = blockIdx.x / blocks;
    fp32_pass<D, kGradQ>(p, sm, (blockIdx.x - head * blocks) * kOwn, head);
  } else {
    const int b = blockIdx.x - p.dq_blocks, blocks = (p.N_k + kOwn - 1) / kOwn, head = b / blocks;
    fp32_pass<D, kGradKV>(p, sm, (b - head * blocks) * kOwn, head);
  }
}

// Row factors of the sequence-length normalisation: n_k^-alpha without a mask, else
// (pos + 1)^-alpha with pos = i + pos0 the query's position (0 for a row that keeps no key).
__global__ void seqlen_norm_kernel(float* __restrict__ out, int N, int N_k, int pos0, int causal, float alpha) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float count = causal ? static_cast<float>(i + pos0 + 1) : static_cast<float>(N_k);
  out[i] = count >= 1.0f ? powf(count, -alpha) : 0.0f;
}

}  // namespace

int launch_seqlen_norm(float* out, int N, int N_k, int pos0, int causal, float alpha, cudaStream_t stream,
                       unsigned long long* launches, cudaError_t* cuda_err) {
  seqlen_norm_kernel<<<(N + 255) / 256, 256, 0, stream>>>(out, N, N_k, pos0, causal, alpha);
  *launches += 1;
  *cuda_err = cudaGetLastError();
  return *cuda_err == cudaSuccess ? SIGATTN_OK : SIGATTN_ERR_CUDA;
}

namespace {

Fp32Args fp32_args(const Problem& p) {
  Fp32Args a = {};
  a.B = p.B;
  a.H = p.H;
  a.H_kv = p.kv_heads();
  a.N = p.N;
  a.N_k = p.key_rows();
  a.off = p.query_pos0();
  a.causal = p.causal;
  a.scale = p.scale;
  a.bias = p.bias;
  a.slopes = p.slopes;
  a.bias_vec = p.bias_vec;
  a.row_scale = p.row_scale;
  a.dbias = p.dbias;
  a.seqlens = p.seqlens;
  a.cu = p.cu_seqlens;
  a.n_seqs = p.n_seqs;
  return a;
}

template <int D, bool BACKWARD>
int launch_fp32(const Fp32Args& a, long long blocks, cudaStream_t stream, cudaError_t* cuda_err) {
  auto kernel = BACKWARD ? bwd_fp32_kernel<D> : fwd_fp32_kernel<D>;
  // a per-device attribute of the kernel: one bit per device ordinal, ordinals past 63 set it on every launch
  static std::atomic<unsigned long long> configured{0};
  int dev = 0;
  *cuda_err = cudaGetDevice(&dev);
  if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  const unsigned long long bit = (dev >= 0 && dev < 64) ? (1ull << dev) : 0ull;
  if ((configured.load(std::memory_order_relaxed) & bit) == 0) {
    *cuda_err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(Fp32Smem<D>));
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
    configured.fetch_or(bit, std::memory_order_relaxed);
  }
  *cuda_err = launch_after(kernel, dim3(static_cast<unsigned>(blocks)), kThreads, sizeof(Fp32Smem<D>), stream, 0, a);
  return *cuda_err == cudaSuccess ? SIGATTN_OK : SIGATTN_ERR_CUDA;
}

}  // namespace

int launch_fwd_fp32(const float* q, const float* k, const float* v, float* o, const Problem& p,
                    cudaStream_t stream, unsigned long long* launches, cudaError_t* cuda_err) {
  Fp32Args a = fp32_args(p);
  a.q = q;
  a.k = k;
  a.v = v;
  a.o = o;
  const long long blocks = static_cast<long long>((p.N + kOwn - 1) / kOwn) * p.B * p.H;
  const int rc = p.D == 128 ? launch_fp32<128, false>(a, blocks, stream, cuda_err)
                            : launch_fp32<64, false>(a, blocks, stream, cuda_err);
  if (rc == SIGATTN_OK) *launches += 1;
  return rc;
}

// dtemp[b*H + h] = sum_i <q_i, dq_i> (see the bf16 conversion kernel): one block per (batch, head).
__global__ void __launch_bounds__(256)
dtemp_fp32_kernel(const float* __restrict__ q, const float* __restrict__ dq, size_t per_head, float* __restrict__ dtemp) {
  const size_t base = static_cast<size_t>(blockIdx.x) * per_head;
  double sum = 0.0;
  for (size_t i = threadIdx.x; i < per_head; i += blockDim.x) sum += static_cast<double>(q[base + i]) * dq[base + i];
  __shared__ double part[256];
  part[threadIdx.x] = sum;
  __syncthreads();
  for (int off = 128; off > 0; off >>= 1) {
    if (static_cast<int>(threadIdx.x) < off) part[threadIdx.x] += part[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) dtemp[blockIdx.x] = static_cast<float>(part[0]);
}

int launch_bwd_fp32(const float* q, const float* k, const float* v, const float* d_o, float* dq, float* dk,
                    float* dv, const Problem& p, cudaStream_t stream, unsigned long long* launches,
                    cudaError_t* cuda_err) {
  if (p.dbias) {
    const size_t n_bias = p.cu_seqlens ? static_cast<size_t>(p.n_seqs) * p.H : static_cast<size_t>(p.B) * p.H;
    *cuda_err = cudaMemsetAsync(p.dbias, 0, n_bias * sizeof(float), stream);
    if (*cuda_err != cudaSuccess) return SIGATTN_ERR_CUDA;
  }
  Fp32Args a = fp32_args(p);
  a.q = q;
  a.k = k;
  a.v = v;
  a.d_o = d_o;
  a.dq = dq;
  a.dk = dk;
  a.dv = dv;
  a.dq_blocks = (p.N + kOwn - 1) / kOwn * p.B * p.H;
  const long long blocks = a.dq_blocks + static_cast<long long>((p.key_rows() + kOwn - 1) / kOwn) * p.B * p.kv_heads();
  const int rc = p.D == 128 ? launch_fp32<128, true>(a, blocks, stream, cuda_err)
                            : launch_fp32<64, true>(a, blocks, stream, cuda_err);
  if (rc != SIGATTN_OK) return rc;
  *launches += 1;
  if (p.dtemp != nullptr) {
    dtemp_fp32_kernel<<<p.B * p.H, 256, 0, stream>>>(q, dq, static_cast<size_t>(p.N) * p.D, p.dtemp);
    *launches += 1;
  }
  *cuda_err = cudaGetLastError();
  return *cuda_err == cudaSuccess ? SIGATTN_OK : SIGATTN_ERR_CUDA;
}

}  // namespace sigattn
