// Sigmoid evaluation shared by the bf16 forward and backward kernels.
//
// With a = log2(e) * x and u = 2^a the weight is P = u / (1 + u) and 1 - P = 1 / (1 + u).
// Both kernels work on a block of 32 or 64 logits of one thread at a time and evaluate
//
//   common path  P = u - u^2 + u^3, the alternating series of u / (1 + u) (relative error
//                u^3 <= 2^-12 for a <= -4, below bf16 resolution), and P (1 - P) = P - P^2;
//                one exponential per element; where the MUFU pipe is the bound (forward at
//                D = 64) a fixed share of them is evaluated on the FMA pipe (ex2_emulated).
//   exact path   e = 2^-a,  r = 1 / (1 + e),  P = r,  P (1 - P) = r e r, taken if any logit of
//                the block has a > -4.  In the forward the reciprocal is formed on the FMA and ALU
//                pipes (an integer first guess and two Newton steps, see rcp_newton), so this path
//                also costs one MUFU op per element there (measured: +13 % on the ViT shape, +9 % at
//                b = 0); the backward, whose activation is not MUFU-bound, keeps the MUFU reciprocal
//                (the Newton form measured 3-8 % slower there).  At b = -log n with normalised q, k almost no
//                block needs it; with unnormalised inputs of unit variance at n = 197 (the ViT
//                shape) about one thread in five does, and since the threads of a warp decide
//                one by one, most warps then need both paths (see sigmoid_block).
//
// The paper evaluates sigmoid as 0.5 (1 + tanh(x / 2)) with the hardware tanh (Section 4).
// On B200 tanh.approx.f32 followed by 0.5 + 0.5 t loses P's relative accuracy for x << 0
// (measured: 1 % at x = -9, 100 % below x = -16), which at b = -log n is where all the
// mass is, so the exponential form is used instead; it costs the same single MUFU op.
#pragma once

#include "sm100_primitives.cuh"

namespace sigattn {

constexpr float kFastPathMaxA = -4.0f;

// max of N values (N = 32 or 64) as a tree of 3-input max ops
template <int N>
__device__ __forceinline__ float max_tree(const float (&a)[N]) {
  static_assert(N == 32 || N == 64, "unsupported width");
  float m[N / 2];
  // level 1: N values -> ceil(N / 3) partial maxima
  constexpr int L1 = (N + 2) / 3;
#pragma unroll
  for (int i = 0; i < N / 3; ++i) m[i] = sm100::fmax3(a[3 * i], a[3 * i + 1], a[3 * i + 2]);
  if (N % 3 == 2) m[L1 - 1] = fmaxf(a[N - 2], a[N - 1]);
  if (N % 3 == 1) m[L1 - 1] = a[N - 1];
  int n = L1;  // 11 or 22
#pragma unroll
  for (int level = 0; level < 4; ++level) {
    if (n > 1) {
      const int groups = n / 3, rest = n % 3;
#pragma unroll
      for (int i = 0; i < groups; ++i) m[i] = sm100::fmax3(m[3 * i], m[3 * i + 1], m[3 * i + 2]);
      if (rest == 2) m[groups] = fmaxf(m[n - 2], m[n - 1]);
      if (rest == 1) m[groups] = m[n - 1];
      n = groups + (rest ? 1 : 0);
    }
  }
  return m[0];
}

// 2^a on the FMA and ALU pipes instead of the MUFU pipe: a = n + f with n = round(a),
// 2^f from a cubic on [-0.5, 0.5] (relative error 7.5e-5 = 2^-13.7, fitted for this
// interval), 2^n by adding n to the exponent field.  Valid for -120 <= a (clamped) and
// a < 100.  Used for a fixed share of the elements to take load off the MUFU pipe, which
// otherwise bounds the activation at 16 elements per clock per SM.
__device__ __forceinline__ float ex2_emulated(float a) {
  a = fmaxf(a, -120.0f);
  const float t = a + 12582912.0f;  // 1.5 * 2^23: the rounded integer lands in the low mantissa bits
  const float f = a - (t - 12582912.0f);
  float p = fmaf(0.05517145885f, f, 0.2426108620f);
  p = fmaf(p, f, 0.6932609924f);
  p = fmaf(p, f, 0.9999280895f);
  return __int_as_float(__float_as_int(p) + (__float_as_int(t) << 23));
}

// Common path: u / (1 + u) = u - u^2 + u^3 - ..., cut after u^3 and evaluated as
// u - u (u - u^2): two FMAs; relative error u^3 <= 2^-12 for a <= -4.
// EMULATE_EVERY = m > 0 evaluates every m-th exponential on the FMA pipe, 0 none.
template <int N, bool WITH_SLOPE, int EMULATE_EVERY>
__device__ __forceinline__ void sigmoid_common(const float (&a)[N], float (&pr)[N], float* pp) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const bool emulate = EMULATE_EVERY > 0 && i % (EMULATE_EVERY > 0 ? EMULATE_EVERY : 1) == EMULATE_EVERY - 1;
    const float u = emulate ? ex2_emulated(a[i]) : sm100::ex2_approx(a[i]);
    const float w = fmaf(-u, u, u);
    pr[i] = fmaf(-u, w, u);
    if (WITH_SLOPE) pp[i] = fmaf(-pr[i], pr[i], pr[i]);  // P <= 1/17 here: no cancellation in P - P^2
  }
}

// 1 / y for 1 <= y < 2^126 without the MUFU pipe: the bit pattern of y subtracted from a constant
// gives a first guess within 5 %, and two Newton steps r <- r (2 - y r) bring the relative error to
// 7e-6 (checked over [1, 2) times every power of two used; the error pattern repeats per binade).
__device__ __forceinline__ float rcp_newton(float y) {
  float r = __int_as_float(0x7EF311C7 - __float_as_int(y));
  r = r * fmaf(-y, r, 2.0f);
  r = r * fmaf(-y, r, 2.0f);
  return r;
}

// Exact path: r = 1 / (1 + 2^-a) = P, and 1 - P = 2^-a r (no subtraction from a rounded P).
template <int N, bool WITH_SLOPE>
__device__ __forceinline__ void sigmoid_exact(const float (&a)[N], float (&pr)[N], float* pp) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float e = sm100::ex2_approx(fminf(-a[i], 120.0f));
    const float r = WITH_SLOPE ? sm100::rcp_approx(1.0f + e) : rcp_newton(1.0f + e);
    pr[i] = r;
    if (WITH_SLOPE) pp[i] = r * (e * r);
  }
}

// Both paths from one exponential, for a warp in which some threads need the exact path (`exact`, per thread) and
// others do not: u = 2^a, P = u / (1 + u), 1 - P = 1 / (1 + u).  Run one after the other, as divergent branches, the
// two paths cost a warp two exponentials per element.
// Backward: the thread's choice holds for its block.  Forward: element by element, a > -4 takes 1 - r (relative error
// of P at most 1.5e-5, checked over u in [1/16, 8]), the others the series; the corrections are predicated and few
// elements need them (4 % faster on the whole forward than a selection between two results).
template <int N, bool WITH_SLOPE, int EMULATE_EVERY>
__device__ __forceinline__ void sigmoid_mixed(const float (&a)[N], bool exact, float (&pr)[N], float* pp) {
  static_assert(EMULATE_EVERY == 0, "one exponential for both paths");
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float u = sm100::ex2_approx(fminf(a[i], 120.0f));
    const float w = fmaf(-u, u, u);
    float p = fmaf(-u, w, u);
    if constexpr (WITH_SLOPE) {
      const float r = sm100::rcp_approx(1.0f + u);
      const float p_exact = u * r;
      pr[i] = exact ? p_exact : p;
      pp[i] = exact ? p_exact * r : fmaf(-p, p, p);
    } else {
      if (a[i] > kFastPathMaxA) p = 1.0f - rcp_newton(1.0f + u);
      pr[i] = p;
    }
  }
}

// The same for warps of causal kernels, with the results of the divergent branches to the last bit: a thread needs
// only 2^a (common path) or 2^-a (exact path), so one exponential of the argument with the thread's sign serves both.
template <int N, bool WITH_SLOPE, int EMULATE_EVERY>
__device__ __forceinline__ void sigmoid_signed(const float (&a)[N], bool exact, float (&pr)[N], float* pp) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const bool emulate = EMULATE_EVERY > 0 && i % (EMULATE_EVERY > 0 ? EMULATE_EVERY : 1) == EMULATE_EVERY - 1;
    float v = sm100::ex2_approx(fminf(exact ? -a[i] : a[i], 120.0f));
    if (emulate && !exact) v = ex2_emulated(a[i]);
    const float w = fmaf(-v, v, v);
    const float p_common = fmaf(-v, w, v);
    const float r = WITH_SLOPE ? sm100::rcp_approx(1.0f + v) : rcp_newton(1.0f + v);
    pr[i] = exact ? r : p_common;
    if (WITH_SLOPE) pp[i] = exact ? r * (v * r) : fmaf(-p_common, p_common, p_common);
  }
}

// How a warp evaluates a block whose threads need different paths.
enum Mixing {
  kBranches,   // one path after the other
  kShared,     // sigmoid_mixed
  kSigned      // sigmoid_signed
};

// Which form a kernel uses.  Short sequences, where b = -log n leaves most warps mixed, gain from one exponential:
// without a mask B32 H12 N197 D64 forward 24.6 -> 20.6 us, backward 65.0 -> 61.8; N577 50.9 -> 45.1, 108 -> 103.
// Causal instantiations keep the branches: B8 H16 N2048 D64 ALiBi (hardly any mixed warp) went from 131 to 137 us
// with the shared form, and b = 0 at D = 128 (nearly all warps exact) from 47.4 to 54.1.  Documents packed without
// padding (RAGGED) are mostly short whatever the mask.
__host__ __device__ constexpr Mixing mixing(bool causal, bool ragged) {
  return !causal ? kShared : ragged ? kSigned : kBranches;
}

// a[N] (already scaled by log2 e) -> P[N]; if WITH_SLOPE also P (1 - P) in pp[N].
// The block's largest a decides between the two paths before anything else is evaluated.
template <int N, bool WITH_SLOPE, int EMULATE_EVERY, Mixing MIXING>
__device__ __forceinline__ void sigmoid_block(const float (&a)[N], float (&pr)[N], float* pp) {
  const bool exact = max_tree<N>(a) > kFastPathMaxA;
  if constexpr (MIXING == kBranches) {
    if (!exact) sigmoid_common<N, WITH_SLOPE, EMULATE_EVERY>(a, pr, pp);
    else sigmoid_exact<N, WITH_SLOPE>(a, pr, pp);
  } else {   // (the warp is converged here)
    if (!__any_sync(0xffffffffu, exact)) sigmoid_common<N, WITH_SLOPE, EMULATE_EVERY>(a, pr, pp);
    else if constexpr (MIXING == kShared) sigmoid_mixed<N, WITH_SLOPE, EMULATE_EVERY>(a, exact, pr, pp);
    else sigmoid_signed<N, WITH_SLOPE, EMULATE_EVERY>(a, exact, pr, pp);
  }
}

// Share of the forward's exponentials evaluated on the FMA pipe (every m-th, 0 = none).
// At D = 128 the shorter instruction stream wins (emulating every 4th measured -6 %); at
// D = 64, where a tile step has half the tensor work per exponential, unloading the MUFU
// pipe gains 1-3 % with a causal mask (N = 2048 and 8192) and loses 3-5 % without one
// (N = 2048 and 8100), so only the causal instantiations do it.
__host__ __device__ constexpr int fwd_emulate_every(int D, bool causal) { return (D == 64 && causal) ? 8 : 0; }

// NC logits of one row -> NC / 2 packed bf16x2 sigmoid values.
//   a = s * scale_log2e + c0   (c0 carries the bias and, with ALiBi, the position term)
// CAUSAL: every key that keeps its weight sits at or before the query, so |i - j| = i - j there and the
// position term is linear in the column: one FMA per logit from a per-call constant instead of a
// difference and an FMA with |.| (what a masked key gets instead is blanked afterwards).
template <int NC, bool ALIBI, bool CAUSAL, int EMULATE_EVERY, bool TWO_SIDED = false>
__device__ __forceinline__ void sigmoid_cols(const uint32_t (&s)[NC], uint32_t (&out)[NC / 2],
                                             float scale_log2e, float bias_log2e, float slope_log2e, float row_rel,
                                             int col_base, bool masked, float mask_limit, float mask_first = 0.0f) {
  float a[NC];
  const float c_first = fmaf(-slope_log2e, row_rel - static_cast<float>(col_base), bias_log2e);   // column col_base
#pragma unroll
  for (int i = 0; i < NC; ++i) {
    float c0 = bias_log2e;
    if (ALIBI && CAUSAL) {
      c0 = fmaf(slope_log2e, static_cast<float>(i), c_first);
    } else if (ALIBI) {
      const float dist = row_rel - static_cast<float>(col_base + i);
      c0 = fmaf(-slope_log2e, fabsf(dist), bias_log2e);
    }
    a[i] = fmaf(__uint_as_float(s[i]), scale_log2e, c0);
  }
  float pr[NC];
  sigmoid_block<NC, false, EMULATE_EVERY, mixing(CAUSAL, TWO_SIDED)>(a, pr, nullptr);
  if (masked) {  // keys after the query (and, in a padded batch, past the sequence's end) get weight 0
#pragma unroll
    for (int i = 0; i < NC; ++i)
      if (static_cast<float>(col_base + i) > mask_limit ||
          (TWO_SIDED && static_cast<float>(col_base + i) < mask_first))   // keys before the row's own sequence
        pr[i] = 0.0f;
  }
#pragma unroll
  for (int i = 0; i < NC / 2; ++i) out[i] = sm100::pack_bf16x2(pr[2 * i], pr[2 * i + 1]);
}

// ------------------------------------------------------------------ backward

// 32 logits (transposed tile: this thread's key against 32 queries) -> P as bf16x2 for
// the dV product and P (1 - P) in fp32 for dS.
//   a = log2(e) * (scale * s + b - slope * |i - j|);  u = 2^a;  P = u / (1 + u);  1 - P = 1 / (1 + u)
// MASK: 0 no element masked, 1 causal only (queries before mask_lo), 2 both ends (padded batch)
// CAUSAL: a query that keeps its weight sits at or after the key, so the position term is linear in the
// query index: one FMA per logit from a per-call constant (a masked query is blanked afterwards).
template <int MASK, bool ALIBI, bool CAUSAL, bool RAGGED = false>
__device__ __forceinline__ void bwd_sigmoid_chunk(const uint32_t (&s)[32], uint32_t (&p_out)[16], float (&pp)[32],
                                                  float scale_log2e, float bias_log2e, float slope_log2e,
                                                  float col_rel, int q_base, float mask_lo, float mask_hi) {
  float a[32];
  const float c_first = fmaf(-slope_log2e, static_cast<float>(q_base) - col_rel, bias_log2e);   // query q_base
#pragma unroll
  for (int e = 0; e < 32; ++e) {
    float c0 = bias_log2e;
    if (ALIBI && CAUSAL) c0 = fmaf(-slope_log2e, static_cast<float>(e), c_first);
    else if (ALIBI) c0 = fmaf(-slope_log2e, fabsf(static_cast<float>(q_base + e) - col_rel), bias_log2e);
    a[e] = fmaf(__uint_as_float(s[e]), scale_log2e, c0);
  }
  float pr[32];
  sigmoid_block<32, true, 0, mixing(CAUSAL, RAGGED)>(a, pr, pp);
  if (MASK == 1) {
#pragma unroll
    for (int e = 0; e < 32; ++e)
      if (static_cast<float>(q_base + e) < mask_lo) { pr[e] = 0.0f; pp[e] = 0.0f; }  // query before key
  }
  if (MASK == 2) {
#pragma unroll
    for (int e = 0; e < 32; ++e)
      // query before key (causal), or, in a padded batch, past the end of the sequence
      if (static_cast<float>(q_base + e) < mask_lo || static_cast<float>(q_base + e) >= mask_hi) {
        pr[e] = 0.0f;
        pp[e] = 0.0f;
      }
  }
#pragma unroll
  for (int e = 0; e < 16; ++e) p_out[e] = sm100::pack_bf16x2(pr[2 * e], pr[2 * e + 1]);
}

}  // namespace sigattn
