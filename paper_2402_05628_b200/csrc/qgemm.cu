// repq_qgemm: argument validation, path selection and the small helper kernels (row sums, 4-bit
// expansion) around the two integer-GEMM kernels.
#include "kernels.h"

namespace repq {
namespace {

__global__ void row_sum_kernel(const uint8_t* __restrict__ codes, int bits, int64_t rows, int64_t n,
                               int64_t ld, int32_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  const int64_t nbytes = bits == 4 ? (n >> 1) : n;
  for (int64_t r = warp; r < rows; r += nwarps) {
    const uint8_t* p = codes + r * ld;
    int s = 0;
    if (bits == 6) {
      // four codes in three bytes (padding bits of the last group are zero): byte-wise, 24 bits at a time
      const int64_t nb6 = (n * 3 + 3) / 4;
      for (int64_t g = lane; g * 3 < nb6; g += 32) {
        uint32_t f = p[3 * g];
        if (3 * g + 1 < nb6) f |= uint32_t(p[3 * g + 1]) << 8;
        if (3 * g + 2 < nb6) f |= uint32_t(p[3 * g + 2]) << 16;
        s += int((f & 0x3Fu) + ((f >> 6) & 0x3Fu) + ((f >> 12) & 0x3Fu) + (f >> 18));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) out[r] = s;
      continue;
    }
    const bool vec = (reinterpret_cast<uintptr_t>(p) & 15) == 0;
    int64_t b = 0;
    if (vec) {
      for (b = int64_t(lane) * 16; b + 16 <= nbytes; b += 32 * 16) {
        const uint4 v = *reinterpret_cast<const uint4*>(p + b);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (bits == 4) {
            s = __dp4a(w[i] & 0x0F0F0F0Fu, 0x01010101u, uint32_t(s));
            s = __dp4a((w[i] >> 4) & 0x0F0F0F0Fu, 0x01010101u, uint32_t(s));
          } else {
            s = __dp4a(w[i], 0x01010101u, uint32_t(s));
          }
        }
      }
      b = nbytes / 16 * 16;
    }
    for (int64_t i = b + lane; i < nbytes; i += 32) s += bits == 4 ? (p[i] & 15) + (p[i] >> 4) : p[i];
    if (bits == 4 && (n & 1) && lane == 0) s += p[nbytes] & 15;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) out[r] = s;
  }
}

// Each thread expands 8 source bytes (16 codes) into 16 destination bytes.
__global__ void expand4_kernel(const uint8_t* __restrict__ src, int64_t rows, int64_t n, int64_t ld_src,
                               uint8_t* __restrict__ dst, int64_t ld_dst, int64_t n_pad) {
  grid_dependency_wait();            // (no early trigger: a GEMM's persistent blocks would take this grid's later ones' places)
  const int64_t groups_per_row = n_pad / 16;
  const int64_t total = rows * groups_per_row;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total;
       i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = i / groups_per_row, gq = i % groups_per_row;
    const int64_t c0 = gq * 16;
    const uint8_t* s = src + r * ld_src + c0 / 2;
    uint32_t w[2] = {0u, 0u};
    if (c0 + 16 <= n && ((reinterpret_cast<uintptr_t>(s) & 7) == 0)) {
      const uint2 v = *reinterpret_cast<const uint2*>(s);
      w[0] = v.x; w[1] = v.y;
    } else {
      for (int e = 0; e < 8; ++e) {
        const int64_t c = c0 + 2 * e;
        uint32_t byte = 0;
        if (c < n) byte = s[e];
        if (c + 1 >= n) byte &= 0x0F;
        w[e >> 2] |= byte << (8 * (e & 3));
      }
    }
    uint4 o;
    uint32_t lo = w[0] & 0x0F0F0F0Fu, hi = (w[0] >> 4) & 0x0F0F0F0Fu;
    o.x = __byte_perm(lo, hi, 0x5140);
    o.y = __byte_perm(lo, hi, 0x7362);
    lo = w[1] & 0x0F0F0F0Fu; hi = (w[1] >> 4) & 0x0F0F0F0Fu;
    o.z = __byte_perm(lo, hi, 0x5140);
    o.w = __byte_perm(lo, hi, 0x7362);
    *reinterpret_cast<uint4*>(dst + r * ld_dst + c0) = o;
  }
}

// Packed weight codes -> one byte per code, 64 codes (32 or 48 bytes) per thread and step.  Settled weights are requested
// before the kernel ahead in the stream has finished; the scratch is written after it in any case.
template <int kBits>
__device__ __forceinline__ void expand_words(const uint32_t (&w)[2 * kBits], uint32_t (&o)[16]) {
  if constexpr (kBits == 4) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t lo = w[i] & 0x0F0F0F0Fu, hi = (w[i] >> 4) & 0x0F0F0F0Fu;
      o[2 * i] = __byte_perm(lo, hi, 0x5140);
      o[2 * i + 1] = __byte_perm(lo, hi, 0x7362);
    }
  } else {
    auto spread = [](uint32_t f) {      // four 6-bit fields of f[23:0] -> four bytes
      return (f & 0x3Fu) | ((f & 0xFC0u) << 2) | ((f & 0x3F000u) << 4) | ((f & 0xFC0000u) << 6);
    };
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t w0 = w[3 * i], w1 = w[3 * i + 1], w2 = w[3 * i + 2];
      o[4 * i] = spread(w0);
      o[4 * i + 1] = spread(__funnelshift_r(w0, w1, 24));
      o[4 * i + 2] = spread(__funnelshift_r(w1, w2, 16));
      o[4 * i + 3] = spread(w2 >> 8);
    }
  }
}
template <int kBits>
__global__ void __launch_bounds__(256) expand_weights_kernel(const uint8_t* __restrict__ src, int rows, int groups, int64_t ld_src,
                                                             uint8_t* __restrict__ dst, int64_t ld_dst, bool settled) {
  constexpr int kIn = 8 * kBits;                           // packed bytes of 64 codes
  const int64_t total = int64_t(rows) * groups, stride = int64_t(gridDim.x) * blockDim.x;
  grid_dependency_trigger();
  if (!settled) {
    // what the kernel ahead may still write comes into L2 at least (where its writes end up as well)
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < total) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + (i / groups) * ld_src + (i % groups) * kIn));
    grid_dependency_wait();
  }
  bool waited = !settled;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += stride) {
    const int64_t r = i / groups;
    const int g = int(i - r * groups);
    uint32_t w[2 * kBits], o[16];
#pragma unroll
    for (int q = 0; q < kIn / 16; ++q) {                   // (a row ends on a 16-byte boundary)
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (int64_t(g) * kIn + 16 * q < ld_src) v = __ldcg(reinterpret_cast<const uint4*>(src + r * ld_src + int64_t(g) * kIn) + q);
      w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
    }
    expand_words<kBits>(w, o);
    if (!waited) { grid_dependency_wait(); waited = true; }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (int64_t(g) * 64 + 16 * q < ld_dst)
        *(reinterpret_cast<uint4*>(dst + r * ld_dst + int64_t(g) * 64) + q) = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
  }
  if (!waited) grid_dependency_wait();
}

// The same for several matrices, as one run of 64-code units.  Everything is read and written behind the dependency wait, and the next
// kernel may start as soon as that is over.
struct ExpandSet {
  const uint8_t* src[kMostExpansions]; uint8_t* dst[kMostExpansions];
  int64_t ld_src[kMostExpansions], ld_dst[kMostExpansions];
  int groups[kMostExpansions], end[kMostExpansions];       // units of a row; units up to the end of this matrix
};
template <int kBits>
__global__ void __launch_bounds__(256) expand_all_kernel(const __grid_constant__ ExpandSet E) {
  constexpr int kIn = 8 * kBits;
  grid_dependency_wait();
  grid_dependency_trigger();
  for (int u = int(blockIdx.x) * 256 + int(threadIdx.x); u < E.end[kMostExpansions - 1]; u += int(gridDim.x) * 256) {
    const uint8_t* src = E.src[0];
    uint8_t* dst = E.dst[0];
    int64_t ld_src = E.ld_src[0], ld_dst = E.ld_dst[0];
    int groups = E.groups[0], first = 0;
#pragma unroll
    for (int m = 1; m < kMostExpansions; ++m)
      if (u >= E.end[m - 1]) { src = E.src[m]; dst = E.dst[m]; ld_src = E.ld_src[m]; ld_dst = E.ld_dst[m]; groups = E.groups[m]; first = E.end[m - 1]; }
    const int r = (u - first) / groups, g = u - first - r * groups;
    uint32_t w[2 * kBits], o[16];
#pragma unroll
    for (int q = 0; q < kIn / 16; ++q) {                   // (a row ends on a 16-byte boundary)
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (int64_t(g) * kIn + 16 * q < ld_src) v = __ldcg(reinterpret_cast<const uint4*>(src + r * ld_src + int64_t(g) * kIn) + q);
      w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
    }
    expand_words<kBits>(w, o);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (int64_t(g) * 64 + 16 * q < ld_dst)
        *(reinterpret_cast<uint4*>(dst + r * ld_dst + int64_t(g) * 64) + q) = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
  }
}

// The byte form of packed weights in the caller's workspace, where it has the room (repq_qgemm_workspace_bytes asks for it): one
// pass over the weights, after which every GEMM kernel takes them.  The GEMM that expands the tiles it copies (bound by its
// converters' shared-memory traffic, once per row tile) remains for smaller workspaces.  Measured (packed against that form):
// 3152 tokens through a DeiT-B block with 6-bit weights 125 -> 96 us (bytes: 84), a 7B-shaped decoder block of 48 tokens with
// 4-bit weights 1860 -> 139 us (bytes: 75).
struct ByteWeights { size_t offset = 0, total = 0; int64_t ld = 0; };
bool byte_weights(const repq_gemm_desc& d, repq_gemm_desc* as_bytes, ByteWeights* B) {
  if (!(packed4(d.bits_w) || packed6(d.bits_w)) || d.batch_outer != 1 || d.batch_inner != 1) return false;
  if (!aligned(d.w_codes, 16) || d.ldw_bytes % 16 != 0) return false;
  *as_bytes = d;
  as_bytes->bits_w = quant_bits(d.bits_w) | REPQ_BYTE_CODES;
  B->ld = round_up(d.K, 16);
  as_bytes->ldw_bytes = B->ld;
  if (!qgemm_tc_supported(*as_bytes) && qgemm_skinny_plan(*as_bytes).mt == 0) return false;
  B->offset = (qgemm_tc_supported(*as_bytes) ? qgemm_tc_workspace(*as_bytes) : 0);
  B->offset = (B->offset + 255) / 256 * 256;
  B->total = B->offset + size_t(d.N) * size_t(B->ld);
  return true;
}

repq_status launch_expand_weights(const repq_gemm_desc& d, uint8_t* dst, int64_t ld, Params params, cudaStream_t st) {
  const int groups = int((int64_t(d.K) + 63) / 64);
  const int64_t blocks = (int64_t(d.N) * groups + 255) / 256, most = int64_t(sm_count()) * 8;
  auto kern = packed4(d.bits_w) ? expand_weights_kernel<4> : expand_weights_kernel<6>;
  REPQ_CUDA(launch_chained(kern, dim3(unsigned(blocks < most ? blocks : most)), dim3(256), 0, st, d.w_codes, d.N, groups, d.ldw_bytes, dst, ld, params == Params::settled));
  note_launch();
  return REPQ_OK;
}

repq_status validate(const repq_gemm_desc& d) {
  REPQ_REQUIRE(d.M >= 0 && d.N > 0 && d.K > 0, REPQ_INVALID_ARG, "qgemm: M >= 0, N > 0, K > 0 required");
  REPQ_REQUIRE(d.batch_outer > 0 && d.batch_inner > 0, REPQ_INVALID_ARG, "qgemm: batch counts must be positive");
  REPQ_REQUIRE(bits_ok(d.bits_a) && bits_w_ok(d.bits_w), REPQ_INVALID_ARG, "qgemm: bits must be 4, 6 or 8");
  if (d.M == 0) return REPQ_OK;
  REPQ_REQUIRE(d.a_codes && d.w_codes && d.out, REPQ_INVALID_ARG, "qgemm: NULL operand or output");
  REPQ_REQUIRE(d.lda_bytes >= code_row_bytes(d.K, d.bits_a) && d.ldw_bytes >= code_row_bytes(d.K, d.bits_w),
               REPQ_INVALID_ARG, "qgemm: operand row stride shorter than K codes");
  REPQ_REQUIRE(int64_t(d.K) * 255 * 255 < (int64_t(1) << 31), REPQ_UNSUPPORTED, "qgemm: K too large for int32 accumulators");
  REPQ_REQUIRE(d.s_a > 0.f, REPQ_INVALID_ARG, "qgemm: s_a must be positive");
  REPQ_REQUIRE(d.out_kind == REPQ_OUT_F32 || d.out_kind == REPQ_OUT_BF16 || d.out_kind == REPQ_OUT_CODES,
               REPQ_INVALID_ARG, "qgemm: unknown out_kind");
  const bool batched = d.batch_outer * int64_t(d.batch_inner) > 1;
  if (batched)
    REPQ_REQUIRE(!d.residual && !d.acc_debug && !d.out_row_sum && !d.a_row_sum && !d.w_row_sum, REPQ_UNSUPPORTED,
                 "qgemm: residual / row sums / acc_debug are for plain (unbatched) products");
  if (packed6(d.bits_w))
    REPQ_REQUIRE(!batched, REPQ_UNSUPPORTED, "qgemm: REPQ_PACKED6 is for the weights of a plain (unbatched) product");
  const int n_out = d.glu ? d.N / 2 : d.N;        // output columns
  if (d.glu) {
    REPQ_REQUIRE(d.out_groups <= 1, REPQ_UNSUPPORTED, "qgemm: glu takes one output group");
    REPQ_REQUIRE(!(d.out_kind == REPQ_OUT_CODES && packed4(d.out_bits)), REPQ_UNSUPPORTED,
                 "qgemm: glu writes float outputs or codes stored one per byte");
  }
  if (d.out_kind == REPQ_OUT_CODES) {
    REPQ_REQUIRE(bits_ok(d.out_bits), REPQ_INVALID_ARG, "qgemm: out_bits must be 4, 6 or 8");
    REPQ_REQUIRE(d.out_groups >= 1 && d.out_groups <= REPQ_MAX_OUT_GROUPS && d.N % d.out_groups == 0,
                 REPQ_INVALID_ARG, "qgemm: out_groups must be 1..4 and divide N");
    for (int g = 0; g < d.out_groups; ++g) {
      REPQ_REQUIRE(d.out_scale[g] > 0.f, REPQ_INVALID_ARG, "qgemm: out_scale[%d] must be positive", g);
      REPQ_REQUIRE(d.out_zero[g] > -(1 << 20) && d.out_zero[g] < (1 << 20), REPQ_INVALID_ARG, "qgemm: |out_zero| must be below 2^20");
    }
    REPQ_REQUIRE(d.ldo >= code_row_bytes(n_out, d.out_bits), REPQ_INVALID_ARG, "qgemm: ldo shorter than a row of codes");
    if (packed4(d.out_bits)) REPQ_REQUIRE((n_out / d.out_groups) % 2 == 0, REPQ_UNSUPPORTED, "qgemm: 4-bit output groups must have even width");
  } else {
    REPQ_REQUIRE(d.ldo >= n_out, REPQ_INVALID_ARG, "qgemm: ldo < output columns");
    const size_t esz = d.out_kind == REPQ_OUT_F32 ? 4 : 2;
    REPQ_REQUIRE(aligned(d.out, esz), REPQ_ALIGNMENT, "qgemm: out is not element-aligned");
  }
  if (d.residual) {
    REPQ_REQUIRE(d.residual_dtype == REPQ_F32 || d.residual_dtype == REPQ_BF16, REPQ_INVALID_ARG, "qgemm: residual_dtype");
    REPQ_REQUIRE(d.ld_residual >= d.N, REPQ_INVALID_ARG, "qgemm: ld_residual < N");
  }
  if (d.rope_cos_sin || d.glu) {
    REPQ_REQUIRE(!batched && !d.gelu && !d.residual, REPQ_UNSUPPORTED,
                 "qgemm: rope / glu are for plain products without gelu or residual");
    REPQ_REQUIRE(!(d.rope_cos_sin && d.glu), REPQ_UNSUPPORTED, "qgemm: rope and glu exclude each other");
    REPQ_REQUIRE(d.N % 2 == 0, REPQ_INVALID_ARG, "qgemm: rope / glu need an even N");
  }
  if (d.rope_cos_sin) {
    const int groups = d.out_groups >= 1 ? d.out_groups : 1;
    REPQ_REQUIRE(groups <= REPQ_MAX_OUT_GROUPS && d.N % groups == 0, REPQ_INVALID_ARG, "qgemm: out_groups must be 1..4 and divide N");
    REPQ_REQUIRE(d.rope_period > 0 && d.rope_dim > 0 && d.rope_dim % 16 == 0 && (d.N / groups) % d.rope_dim == 0,
                 REPQ_INVALID_ARG, "qgemm: rope_dim must be a multiple of 16 that divides N / out_groups, rope_period positive");
    REPQ_REQUIRE(d.rope_groups >= 1 && d.rope_groups <= groups, REPQ_INVALID_ARG, "qgemm: rope_groups must be 1..out_groups");
    REPQ_REQUIRE(aligned(d.rope_cos_sin, 16), REPQ_ALIGNMENT, "qgemm: rope_cos_sin must be 16-byte aligned");
  }
  return REPQ_OK;
}

EpilogueParams make_epilogue(const repq_gemm_desc& d) {
  EpilogueParams ep{};
  ep.s_w = d.s_w; ep.z_w = d.z_w; ep.s_w_scalar = d.s_w_scalar; ep.z_w_scalar = d.z_w_scalar;
  ep.bias = d.bias;
  ep.scale_a = d.alpha * d.s_a;
  ep.z_a = d.z_a; ep.K = d.K; ep.N = d.N;
  ep.gelu = d.gelu;
  ep.residual = d.residual; ep.residual_bf16 = d.residual_dtype == REPQ_BF16; ep.ld_residual = d.ld_residual;
  ep.out_kind = d.out_kind;
  const bool codes = d.out_kind == REPQ_OUT_CODES;
  ep.qmax = codes ? code_max(d.out_bits) : 0;
  ep.pack4 = codes && packed4(d.out_bits);
  ep.group_width = codes ? d.N / d.out_groups : d.N;
  for (int g = 0; g < REPQ_MAX_OUT_GROUPS; ++g) {
    const bool on = codes && g < d.out_groups;
    ep.inv_out_scale[g] = on ? 1.f / d.out_scale[g] : 1.f;
    ep.out_zero[g] = on ? d.out_zero[g] : 0;
  }
  ep.out = d.out; ep.ldo = d.ldo;
  ep.out_row_sum = codes ? d.out_row_sum : nullptr;
  ep.acc_debug = d.acc_debug;
  ep.rope = reinterpret_cast<const float2*>(d.rope_cos_sin);
  ep.rope_period = d.rope_period;
  ep.rope_dim = d.rope_dim;
  ep.rope_cols = d.rope_cos_sin ? d.rope_groups * (d.N / (d.out_groups >= 1 ? d.out_groups : 1)) : 0;
  ep.glu = d.glu;
  return ep;
}

}  // namespace

bool qgemm_byte_form(const repq_gemm_desc& d, repq_gemm_desc* as_bytes, size_t* scratch, size_t* bytes) {
  ByteWeights B;
  if (!byte_weights(d, as_bytes, &B)) return false;
  *scratch = B.offset;
  *bytes = B.total - B.offset;
  return true;
}

repq_status launch_expand_all(const Expansion* e, int n, int bits, cudaStream_t st) {
  ExpandSet E{};
  int64_t units = 0;
  for (int m = 0; m < kMostExpansions; ++m) {
    if (m < n) {
      E.src[m] = e[m].src; E.dst[m] = e[m].dst; E.ld_src[m] = e[m].ld_src; E.ld_dst[m] = e[m].ld_dst;
      E.groups[m] = (e[m].k + 63) / 64;
      units += int64_t(e[m].rows) * E.groups[m];
    }
    E.end[m] = int(units);
  }
  REPQ_REQUIRE(units < (int64_t(1) << 30), REPQ_UNSUPPORTED, "qgemm: too many weights to expand at once");
  // (four blocks per SM: they leave room for the kernel that runs beside this one)
  const int64_t blocks = (units + 255) / 256, most = int64_t(sm_count()) * 4;
  auto kern = packed4(bits) ? expand_all_kernel<4> : expand_all_kernel<6>;
  REPQ_CUDA(launch_chained(kern, dim3(unsigned(blocks < most ? blocks : most)), dim3(256), 0, st, E));
  note_launch();
  return REPQ_OK;
}

size_t qgemm_workspace_least(const repq_gemm_desc& d) {
  return !scores_supported(d) && qgemm_tc_supported(d) ? qgemm_tc_workspace(d) : 0;
}
size_t qgemm_workspace(const repq_gemm_desc& d) {
  repq_gemm_desc as_bytes;
  ByteWeights B;
  return byte_weights(d, &as_bytes, &B) ? B.total : qgemm_workspace_least(d);
}

repq_status launch_row_sum(const uint8_t* codes, int bits, int64_t rows, int64_t n, int64_t ld_bytes,
                           int32_t* out, cudaStream_t st) {
  if (rows == 0) return REPQ_OK;
  const int64_t blocks = (rows + 7) / 8;
  const int grid = int(blocks < 4096 ? blocks : 4096);
  row_sum_kernel<<<grid, 256, 0, st>>>(codes, packed4(bits) ? 4 : packed6(bits) ? 6 : 8, rows, n, ld_bytes, out);
  REPQ_CUDA(cudaGetLastError());
  note_launch();
  return REPQ_OK;
}

repq_status launch_expand4(const uint8_t* src, int64_t rows, int64_t n, int64_t ld_src, uint8_t* dst,
                           int64_t ld_dst, int64_t n_pad, cudaStream_t st) {
  if (rows == 0) return REPQ_OK;
  const int64_t total = rows * (n_pad / 16);
  const int64_t blocks = (total + 255) / 256;
  const int grid = int(blocks < 8192 ? blocks : 8192);
  REPQ_CUDA(launch_chained(expand4_kernel, dim3(grid), dim3(256), 0, st, src, rows, n, ld_src, dst, ld_dst, n_pad));
  note_launch();
  return REPQ_OK;
}

}  // namespace repq

using namespace repq;

extern "C" repq_status repq_qgemm_workspace_bytes(const repq_gemm_desc* d, size_t* bytes) {
  REPQ_REQUIRE(d && bytes, REPQ_INVALID_ARG, "qgemm_workspace_bytes: NULL argument");
  REPQ_TRY(validate(*d));
  *bytes = d->M > 0 ? qgemm_workspace(*d) : 0;
  return REPQ_OK;
}

repq_status repq::run_qgemm(const repq_gemm_desc& given, void* workspace, size_t workspace_bytes, Params params, cudaStream_t st) {
  const repq_gemm_desc* d = &given;
  REPQ_TRY(validate(*d));
  if (d->M == 0) return REPQ_OK;
  if (scores_supported(*d)) return scores_tc_supported(*d) ? launch_scores_tc(*d, st) : launch_scores(*d, st);
  repq_gemm_desc as_bytes;
  ByteWeights B;
  if (byte_weights(*d, &as_bytes, &B) && workspace && workspace_bytes >= B.total && aligned(workspace, 256)) {
    uint8_t* w = static_cast<uint8_t*>(workspace) + B.offset;
    REPQ_TRY(launch_expand_weights(*d, w, B.ld, params, st));
    as_bytes.w_codes = w;
    d = &as_bytes;
    params = Params::streamed;                             // (the expansion is the kernel just ahead now)
  }
  const EpilogueParams ep = make_epilogue(*d);
  const SkinnyPlan few = qgemm_skinny_plan(*d);
  const TcPlan tiles = qgemm_tc_plan(*d);
  if (few.mt != 0 && (tiles.bn == 0 || few.us < tiles.us)) return qgemm_skinny(*d, ep, few, params, st);
  if (tiles.bn != 0) {
    const size_t need = qgemm_tc_workspace(*d);
    REPQ_REQUIRE(workspace_bytes >= need && (need == 0 || workspace), REPQ_WORKSPACE_TOO_SMALL,
                 "qgemm: workspace of %zu bytes given, %zu needed", workspace_bytes, need);
    return qgemm_tc(*d, ep, tiles, workspace, workspace_bytes, st);
  }
  return qgemm_mma(*d, ep, st);
}

extern "C" repq_status repq_qgemm(const repq_gemm_desc* d, void* workspace, size_t workspace_bytes, void* stream) {
  REPQ_REQUIRE(d, REPQ_INVALID_ARG, "qgemm: NULL descriptor");
  return run_qgemm(*d, workspace, workspace_bytes, Params::streamed, static_cast<cudaStream_t>(stream));
}
