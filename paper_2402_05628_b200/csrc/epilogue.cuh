// Shared GEMM epilogue: zero-point correction, de-quantization, bias, GELU, residual, and the optional
// re-quantization of Eq. 4.  Used by both the tensor-memory GEMM and the warp-MMA GEMM so that the two
// produce identical results.
#pragma once
#include <cuda_bf16.h>
#include <cstdint>

#include "../../include/repq.h"
#include "f32x2.cuh"

namespace repq {

struct EpilogueParams {
  const float* s_w;        // per output channel or nullptr
  const int32_t* z_w;      // per output channel or nullptr
  float s_w_scalar;
  int32_t z_w_scalar;
  const float* bias;       // or nullptr
  float scale_a;           // alpha * s_a
  int32_t z_a;
  int32_t K;
  int32_t N;
  int32_t gelu;
  const void* residual;    // or nullptr
  int32_t residual_bf16;
  int64_t ld_residual;
  int32_t out_kind;
  int32_t qmax;            // 2^out_bits - 1
  int32_t pack4;           // out_bits == 4
  int32_t group_width;     // N / out_groups
  float inv_out_scale[REPQ_MAX_OUT_GROUPS];
  int32_t out_zero[REPQ_MAX_OUT_GROUPS];
  void* out;
  int64_t ldo;
  int32_t* out_row_sum;    // or nullptr
  int32_t* acc_debug;      // or nullptr, dense M x N
  // steps on pairs of neighbouring columns (LLaMA block form), applied to v before the output conversion
  const float2* rope;      // (cos, sin) table [rope_period][rope_dim / 2], or nullptr
  int32_t rope_period;
  int32_t rope_dim;
  int32_t rope_cols;       // columns below this bound are rotated
  int32_t glu;             // columns (2i, 2i+1) = (gate, up): output column i = silu(gate) * up
};

// Per-column constants of the epilogue, gathered once per output column.
struct ColumnTerms {
  float scale;    // alpha * s_a * s_w[j]
  float bias;
  int32_t z_w;
  int32_t kzz;    // K * z_a * z_w[j] - z_a * wsum[j]
  float inv_so;
  float zo_lo, zo_hi;
  int32_t zo;
};

__device__ __forceinline__ ColumnTerms column_terms(const EpilogueParams& p, int j, int32_t wsum_j) {
  ColumnTerms c;
  const float sw = p.s_w ? __ldg(p.s_w + j) : p.s_w_scalar;
  c.z_w = p.z_w ? __ldg(p.z_w + j) : p.z_w_scalar;
  c.scale = p.scale_a * sw;
  c.bias = p.bias ? __ldg(p.bias + j) : 0.f;
  // wrap-around integer arithmetic: only the final correction has to fit 32 bits
  c.kzz = int32_t(uint32_t(p.K) * uint32_t(p.z_a) * uint32_t(c.z_w) - uint32_t(p.z_a) * uint32_t(wsum_j));
  const int g = p.out_kind == REPQ_OUT_CODES ? j / p.group_width : 0;
  c.inv_so = p.inv_out_scale[g];
  c.zo = p.out_zero[g];
  c.zo_lo = float(-c.zo);
  c.zo_hi = float(p.qmax - c.zo);
  return c;
}

// erf-form GELU, v * Phi(v), without branches.  With |v| clamped to 4 sqrt2 (erfc(4) < 2e-8; beyond, v Phi(v) is 0 or v to within
// 5e-8: -4.4e-8 for -inf, inf for inf, NaN for NaN) and t = |v| / sqrt2,
//     erfc(t) = 2^(-t q(t)),   Phi(v) = h for v < 0,   1 - h otherwise,   h = erfc(t) / 2 = 2^(-t q(t) - 1),
// so v Phi(v) = max(v, 0) - |v| h, one multiply-add (a select between h and 1 - h, then a product: 12608 x 3072 x 768 42.7 us, 41.5 so),
// and q, which is smooth (q(0) = 2 / (sqrt(pi) ln 2), q(t) ~ t / ln 2), is a degree-6 polynomial fitted so that
// the error of erf stays below 1e-7.  It is evaluated in n = -|v| directly: -t q(t) = n p(n) with p(n) = q(-n / sqrt2) / sqrt2, whose
// coefficients are q's times powers of 1 / sqrt2 (one product less per value: 12608 x 3072 x 768 43.2 -> 41.8 us, 18464 x 4096 x 1024 76.8 ->
// 74.2).  Against the float64 erf form the float32 result is within 1.2e-7 |v| (4 million values: 1.09e-7, 1.12e-7 by way of t), and
// within 2e-7 of itself for v > 0; of the small values of the negative tail it is off by 1e-6 at -2, 3e-5 at -3, 1.2e-3 at -4 and 10 % at the
// clamp (1.6e-7 in absolute terms at most).
constexpr float kGeluLow = -5.65685424949238f;                               // -4 sqrt2
__device__ __forceinline__ float max_nan(float a, float b) {                 // (fmaxf drops a NaN)
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float gelu_erf(float v) {
  const float n = fmaxf(fminf(v, -v), kGeluLow);                             // -|v|, clamped; -t q(t) = n p(n)
  float p = -8.858894034e-06f;
  p = fmaf(p, n, -5.770146163e-05f);
  p = fmaf(p, n, 4.069651186e-04f);
  p = fmaf(p, n, 7.363100536e-03f);
  p = fmaf(p, n, 5.266658589e-02f);
  p = fmaf(p, n, -4.591643214e-01f);
  p = fmaf(p, n, 1.151108861e+00f);
  float h;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(h) : "f"(fmaf(n, p, -1.f)));
  return fmaf(n, h, max_nan(v, 0.f));
}

// The same on two values at once (packed float pairs where the operation exists in that form): every lane goes through
// the operations of gelu_erf in the same order, so the results are the same bits.
__device__ __forceinline__ void gelu_erf_pair(float& v0, float& v1) {
  const f32x2 n = pack2(fmaxf(fminf(v0, -v0), kGeluLow), fmaxf(fminf(v1, -v1), kGeluLow));
  f32x2 p = splat2(-8.858894034e-06f);
  p = fma2(p, n, splat2(-5.770146163e-05f));
  p = fma2(p, n, splat2(4.069651186e-04f));
  p = fma2(p, n, splat2(7.363100536e-03f));
  p = fma2(p, n, splat2(5.266658589e-02f));
  p = fma2(p, n, splat2(-4.591643214e-01f));
  p = fma2(p, n, splat2(1.151108861e+00f));
  float e0, e1, h0, h1;
  unpack2(fma2(n, p, splat2(-1.f)), e0, e1);
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(h0) : "f"(e0));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(h1) : "f"(e1));
  unpack2(fma2(n, pack2(h0, h1), pack2(max_nan(v0, 0.f), max_nan(v1, 0.f))), v0, v1);
}

// acc -> corrected integer -> float value before the output conversion.
__device__ __forceinline__ float epilogue_value(const EpilogueParams& p, const ColumnTerms& c, int32_t acc,
                                                int32_t asum_m, int64_t m, int j) {
  const int32_t corr = int32_t(uint32_t(acc) - uint32_t(c.z_w) * uint32_t(asum_m) + uint32_t(c.kzz));
  float v = fmaf(c.scale, float(corr), c.bias);
  if (p.gelu) v = gelu_erf(v);
  if (p.residual) {
    const int64_t off = m * p.ld_residual + j;
    v += p.residual_bf16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(p.residual)[off])
                         : static_cast<const float*>(p.residual)[off];
  }
  return v;
}

// Rotary position embedding of one pair: (a, b) at column pair index `pair` of its head, row position `pos`.
__device__ __forceinline__ void rope_rotate(const float2 cs, float& a, float& b) {
  const float ra = fmaf(a, cs.x, -(b * cs.y));
  const float rb = fmaf(a, cs.y, b * cs.x);
  a = ra;
  b = rb;
}

// silu(g) * u, silu(x) = x / (1 + exp(-x)); exp(-x) = +inf for very negative x gives -0 * u.
__device__ __forceinline__ float silu_mul(float g, float u) { return __fdividef(g, 1.f + __expf(-g)) * u; }

// Eq. 4 with the output quantizer: clip(round(v / s_o) + z_o, 0, qmax).
__device__ __forceinline__ int32_t requantize(const ColumnTerms& c, float v) {
  float t = v * c.inv_so;
  t = fminf(fmaxf(t, c.zo_lo), c.zo_hi);
  return __float2int_rn(t) + c.zo;
}

}  // namespace repq
