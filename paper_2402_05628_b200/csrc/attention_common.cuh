// What the two fused attention kernels share: parameters, byte helpers, the K tensor map, the output conversion.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>

#include "f32x2.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace repq {
namespace attn {

using namespace tc;

__device__ __forceinline__ bool wait_for(uint32_t bar, uint32_t parity, volatile int* abort, int code, int32_t* status) {
  return tc::mbar_wait<false>(bar, parity, abort, code, status);
}

constexpr int kRows = 128;                        // query rows per tile (MMA M)
constexpr uint32_t kQBytes = kRows * 128;         // Q tile: rows of 128 bytes (the head's codes, zero-padded)
constexpr uint32_t kMagicBits = 0x4B400000u;      // float 1.5 * 2^23

// Division by a number that is fixed per launch: q = (t + ((n - t) >> sh1)) >> sh2 with t = umulhi(n, mul), exact for every 32-bit n
// (Granlund and Montgomery, Division by invariant integers using multiplication, 1994).  A division by a run-time number is some 20
// instructions, and every role of a CTA takes two per tile.
struct FixedDiv { uint32_t mul; int sh1, sh2; };
inline FixedDiv fixed_div(uint32_t d) {
  int l = 0;
  while ((uint64_t(1) << l) < d) ++l;                     // ceil(log2 d)
  return {uint32_t((((uint64_t(1) << l) - d) << 32) / d + 1), l < 1 ? l : 1, l > 1 ? l - 1 : 0};
}
__device__ __forceinline__ int div_by(int n, const FixedDiv& f) {
  const uint32_t t = __umulhi(uint32_t(n), f.mul);
  return int((t + ((uint32_t(n) - t) >> f.sh1)) >> f.sh2);
}

struct AttnParams {
  const uint8_t* q; const uint8_t* k; const uint8_t* v;
  int64_t ldq, ldk, ldv, q_so, q_si, k_so, k_si, v_so, v_si;
  int Lq, Lk, dh, batch_inner, causal;
  float scale;            // alpha s_q s_k
  int zq, zk;
  float log2_s;           // log2 of the log-sqrt2 scale
  int qmax_p;             // 2^bits_p - 1
  int z_v, v_small;
  float out_scale;        // s_p s_v
  int out_kind, qmax, pack4;
  float inv_so; int zo;
  void* out; int64_t ldo, o_so, o_si;
  int32_t* out_row_sum;
  int n_pad, tmem_cols, vec_store;
  int no_f8;                                         // keep integer scores where the 8-bit float form would apply
  FixedDiv by_pairs, by_inner;
  int pairs, tiles;                                  // (batch, head) pairs and query tiles of 128 rows: the grid is their product
  int32_t* status;
};

__device__ __forceinline__ uint32_t tile_offset(int row, int piece) {
  return uint32_t(row >> 3) * 1024u + uint32_t(row & 7) * 128u + (uint32_t(piece ^ (row & 7)) << 4);
}
__device__ __forceinline__ int sum_bytes(const uint4& v) {
  return __dp4a(v.x, 0x01010101u, __dp4a(v.y, 0x01010101u, __dp4a(v.z, 0x01010101u, __dp4a(v.w, 0x01010101u, 0u))));
}
// Bytewise c - z (two's complement) for codes and zero points below 128: with the top bit of every byte of c set
// no borrow crosses a byte, and flipping that bit back leaves c - z mod 256.
__device__ __forceinline__ uint32_t sub_bytes(uint32_t c, uint32_t z4) { return ((c | 0x80808080u) - z4) ^ 0x80808080u; }
__device__ __forceinline__ uint4 sub_bytes(const uint4& c, uint32_t z4) {
  return make_uint4(sub_bytes(c.x, z4), sub_bytes(c.y, z4), sub_bytes(c.z, z4), sub_bytes(c.w, z4));
}
// Bytes in two's complement (within [-127, 127]) -> sign bit and magnitude.
__device__ __forceinline__ uint32_t sign_magnitude(uint32_t x) { return __vabs4(x) | (x & 0x80808080u); }
__device__ __forceinline__ uint4 sign_magnitude(const uint4& c) {
  return make_uint4(sign_magnitude(c.x), sign_magnitude(c.y), sign_magnitude(c.z), sign_magnitude(c.w));
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}


// Output conversion of 16 values of one row, channels c0 .. c0 + 15: byte codes (Eq. 4) by 16-byte stores ...
__device__ __forceinline__ void store_codes(const AttnParams& P, const float (&v)[16], int64_t roff, int c0, int& code_sum) {
  // t = v / s_o clamped, rounded half to even by the float adder (1.5 * 2^23), z_o added as an integer
  const float zo_lo = float(-P.zo), zo_hi = float(P.qmax - P.zo);
  const f32x2 inv2 = splat2(P.inv_so), magic2 = splat2(__uint_as_float(kMagicBits));
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t u[4];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      float t0, t1, u0, u1;
      unpack2(mul2(pack2(v[4 * i + 2 * k], v[4 * i + 2 * k + 1]), inv2), t0, t1);
      unpack2(add2(pack2(fminf(fmaxf(t0, zo_lo), zo_hi), fminf(fmaxf(t1, zo_lo), zo_hi)), magic2), u0, u1);
      u[2 * k] = __float_as_uint(u0) + uint32_t(P.zo);
      u[2 * k + 1] = __float_as_uint(u1) + uint32_t(P.zo);
    }
    w[i] = __byte_perm(__byte_perm(u[0], u[1], 0x0040), __byte_perm(u[2], u[3], 0x0040), 0x5410);
    code_sum = int(__dp4a(w[i], 0x01010101u, uint32_t(code_sum)));
  }
  *reinterpret_cast<uint4*>(static_cast<uint8_t*>(P.out) + roff + c0) = make_uint4(w[0], w[1], w[2], w[3]);
}
// ... and every form (float, packed codes, rows off the 16-byte grid).
__device__ __forceinline__ void store_values(const AttnParams& P, const float (&v)[16], int64_t roff, int c0, int& code_sum) {
  if (P.out_kind == REPQ_OUT_F32) {
    float* o = static_cast<float*>(P.out) + roff + c0;
    if (P.vec_store) {
#pragma unroll
      for (int e = 0; e < 4; ++e) reinterpret_cast<float4*>(o)[e] = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) o[e] = v[e];
    }
  } else if (P.out_kind == REPQ_OUT_BF16) {
    __nv_bfloat16* o = static_cast<__nv_bfloat16*>(P.out) + roff + c0;
    if (P.vec_store) {
      uint32_t w[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
        w[e] = *reinterpret_cast<const uint32_t*>(&h);
      }
      reinterpret_cast<uint4*>(o)[0] = make_uint4(w[0], w[1], w[2], w[3]);
      reinterpret_cast<uint4*>(o)[1] = make_uint4(w[4], w[5], w[6], w[7]);
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) o[e] = __float2bfloat16_rn(v[e]);
    }
  } else if (!P.pack4 && P.vec_store) {
    store_codes(P, v, roff, c0, code_sum);
  } else {
    const float zo_lo = float(-P.zo), zo_hi = float(P.qmax - P.zo);
    uint32_t q[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const float tq = fminf(fmaxf(v[e] * P.inv_so, zo_lo), zo_hi);
      q[e] = uint32_t(__float2int_rn(tq) + P.zo);
      code_sum += int(q[e]);
    }
    uint8_t* orow = static_cast<uint8_t*>(P.out) + roff;
    if (P.pack4) {
      uint32_t w0 = 0u, w1 = 0u;
#pragma unroll
      for (int e = 0; e < 8; ++e) { w0 |= q[e] << (4 * e); w1 |= q[8 + e] << (4 * e); }
      if (P.vec_store) *reinterpret_cast<uint2*>(orow + (c0 >> 1)) = make_uint2(w0, w1);
      else {
#pragma unroll
        for (int e = 0; e < 4; ++e) { orow[(c0 >> 1) + e] = uint8_t(w0 >> (8 * e)); orow[(c0 >> 1) + 4 + e] = uint8_t(w1 >> (8 * e)); }
      }
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) orow[c0 + e] = uint8_t(q[e]);
    }
  }
}

// Tensor map of the K codes for the bulk-copy variant: (bytes of a row, keys, batch items); a box is 128 bytes x the keys of a visit.
inline repq_status make_k_map(CUtensorMap* map, const AttnParams& P, int batch_outer, int keys) {
  EncodeTiledFn fn = encode_fn();
  REPQ_REQUIRE(fn != nullptr, REPQ_CUDA_ERROR, "attention: cuTensorMapEncodeTiled is not available");
  const cuuint64_t span = cuuint64_t(P.batch_inner - 1) * cuuint64_t(P.k_si) + cuuint64_t(P.dh);    // bytes the heads cover
  const cuuint64_t dims[3] = {span, cuuint64_t(P.Lk), cuuint64_t(batch_outer)};
  const cuuint64_t strides[2] = {cuuint64_t(P.ldk), cuuint64_t(P.k_so)};
  const cuuint32_t box[3] = {128, cuuint32_t(keys), 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t*>(P.k), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  REPQ_REQUIRE(r == CUDA_SUCCESS, REPQ_CUDA_ERROR, "attention: K tensor map failed with code %d", int(r));
  return REPQ_OK;
}


// The persistent kernel (attention_pipe.cu); call only if it is supported.
bool pipe_supported(const AttnParams& P, int qmax_qk);
repq_status launch_pipe(const AttnParams& P, int64_t pairs, int qmax_qk, cudaStream_t st);

}  // namespace attn
}  // namespace repq
