// Internal launchers shared between translation units of the repq library.
#pragma once
#include "common.h"
#include "epilogue.cuh"

namespace repq {

// Whether a kernel may read its parameters (weight codes, normalisation factors) ahead of the dependency wait.  `streamed`:
// no, like every other operand they may be the work of the kernel just ahead in the stream (the entry points of the library
// promise stream order).  `settled`: a kernel of the same chain that waited for everything before the chain has started
// already, so whatever wrote the parameters has completed (the kernels of a block behind its first one).
// `beside` (the first LayerNorm of a block): the kernel just ahead in the stream has waited for everything before it and does work that
// this kernel does not need; the two run side by side, and this kernel ends only when the one ahead has.
enum class Params { streamed, settled, beside };

// LayerNorm + quantization (repq_ln_quant), which can also set a run of words to zero: row-sum accumulators that later
// kernels of a chain add into, without a launch of their own.
struct ClearWords { int32_t* at = nullptr; int64_t n = 0; };
repq_status launch_ln_quant(const void* x, int x_dtype, int64_t rows, int D, int64_t ldx, const float* gamma_t,
                            const float* beta_t, float eps, int norm_kind, float s_t, int z_t, int bits, uint8_t* codes,
                            int64_t ld_codes_bytes, int32_t* row_sum, ClearWords clear, Params params, cudaStream_t st);

// repq_qgemm, with the caller's word on the weights.
repq_status run_qgemm(const repq_gemm_desc& d, void* workspace, size_t workspace_bytes, Params params, cudaStream_t st);

// Row sums of a code matrix: out[r] = sum_c codes[r, c] (zero-point correction terms).
repq_status launch_row_sum(const uint8_t* codes, int bits, int64_t rows, int64_t n, int64_t ld_bytes,
                           int32_t* out, cudaStream_t st);

// 4-bit packed codes -> one code per byte (dst rows of ld_dst bytes, zero-padded up to n_pad codes).
repq_status launch_expand4(const uint8_t* src, int64_t rows, int64_t n, int64_t ld_src, uint8_t* dst,
                           int64_t ld_dst, int64_t n_pad, cudaStream_t st);

// Warp-MMA integer GEMM (any shape, batched).
repq_status qgemm_mma(const repq_gemm_desc& d, const EpilogueParams& ep, cudaStream_t st);

// Attention-score kernel: batched code-by-code products with scalar quantizers, K <= 128, float32 output.
bool scores_supported(const repq_gemm_desc& d);
repq_status launch_scores(const repq_gemm_desc& d, cudaStream_t st);
// The same on tcgen05 (byte codes, 16-byte aligned operand rows and output rows); call only if scores_supported.
bool scores_tc_supported(const repq_gemm_desc& d);
repq_status launch_scores_tc(const repq_gemm_desc& d, cudaStream_t st);

// The two integer GEMMs on tcgen05 and how each would cut a problem up, with its estimated time in microseconds (measured in
// CUDA graphs over 1..16384 tokens, N and K 384..22016; half of the estimates are within 3 %, 99 of 100 within 15 %).  One
// estimate serves the choice between the two and the choice of form within each.
//
// 128-row or 256-row tiles (plain products with TMA-compatible operands).  bn: tile width, 0 where the kernel does not take the
// problem; pair: 256 x 256 tiles by pairs of CTAs.
struct TcPlan { int bn = 0; bool pair = false; float us = 0.f; };
bool qgemm_tc_supported(const repq_gemm_desc& d);
TcPlan qgemm_tc_plan(const repq_gemm_desc& d);
size_t qgemm_tc_workspace(const repq_gemm_desc& d);
repq_status qgemm_tc(const repq_gemm_desc& d, const EpilogueParams& ep, const TcPlan& plan, void* ws, size_t ws_bytes,
                     cudaStream_t st);
// Few tokens (weights on the M side of the tensor-core instruction): plain products, byte codes, both row sums given.  mt:
// tokens per tile, 0 where the kernel does not take the problem; split: CTAs that share a tile's K range; two: SMs take two CTAs.
struct SkinnyPlan { int mt = 0, split = 0; bool two = false; float us = 0.f; };
SkinnyPlan qgemm_skinny_plan(const repq_gemm_desc& d);
repq_status qgemm_skinny(const repq_gemm_desc& d, const EpilogueParams& ep, const SkinnyPlan& plan, Params params, cudaStream_t st);

// Packed weights of a plain product in the form the GEMM kernels take, one code per byte: the same problem on byte codes (its w_codes still
// to be set), the scratch it needs then and the bytes of its weights.  False: the problem has no such form.
bool qgemm_byte_form(const repq_gemm_desc& d, repq_gemm_desc* as_bytes, size_t* scratch, size_t* bytes);
// The packed weights of several products written in that form by one kernel, which reads them behind its dependency wait.
constexpr int kMostExpansions = 4;
struct Expansion { const uint8_t* src; int rows, k; int64_t ld_src; uint8_t* dst; int64_t ld_dst; };
repq_status launch_expand_all(const Expansion* e, int n, int bits, cudaStream_t st);

// Workspace of a GEMM: with room for a byte copy of packed weights, and the least it can run in.
size_t qgemm_workspace(const repq_gemm_desc& d);
size_t qgemm_workspace_least(const repq_gemm_desc& d);

// P.V (Eqs. 16-17): kernel parameters shared by the two implementations, storage widths already resolved
// (bits_v is 4 for packed codes, 8 for byte codes).
struct PvParams {
  const uint8_t* p; int bits_p; int64_t ldp, p_pair;
  const uint8_t* v; int bits_v; int64_t ldv, v_so, v_si;
  int Lq, Lk, d_h, batch_inner, causal;
  int z_v;
  float scale;               // s_p * s_v
  int out_kind, qmax, pack4;
  float inv_so; int zo;
  void* out; int64_t ldo, o_so, o_si;
  int32_t* out_row_sum;
};
// Tensor-memory (tcgen05) P.V kernel: needs V rows that allow vector loads; the warp-MMA kernel covers the rest.
bool pv_tc_supported(const repq_pv_desc& d);
repq_status launch_pv_tc(const repq_pv_desc& d, const PvParams& P, cudaStream_t st);

// One-thread kernel whose mbarrier wait can only run out (see repq_bounded_wait_selftest).
repq_status launch_wait_selftest(long long limit_cycles, cudaStream_t st);

// Device-side health word (bounded waits report here instead of trapping); nullptr on failure.
int32_t* device_status_word();

}  // namespace repq
