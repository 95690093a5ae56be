// Fused attention on integer codes, persistent form (quantizers of at most 7 bits): scores (Eq. 3 with quantized Q and K),
// Softmax, log-sqrt2 codes (Eq. 15) and P.V with the reparameterized log2 de-quantization (Eqs. 16-17) in one kernel.
// Scores and codes never leave the SM.  The code of a score depends on the row's final Softmax sum, so the keys are walked
// twice, a visit being 64 keys (heads of up to 64 channels and more tiles than SMs) or 128 keys (wider heads, few tiles):
//   pass 1   S = Q K^T per visit (tcgen05.mma on 8-bit operands into one of two slots of tensor memory), running row
//            maximum m and sum Z = sum 2^(c (S - m))
//   pass 2   S again, t = 2 (log2 Z + log2 s) - 2 c (S - m), code p = clip(round(t), 0, 2^b - 1), operand values
//            2^(-ceil(p/2)) split by the parity of p into E and O, written back over the columns of tensor memory the
//            scores came from, from where the P.V MMAs take their A operand; O = s s_v (acc_E + sqrt2 acc_O)
//
// A byte below 128 is q - z_q as a signed byte in the Q tile and the raw code in the K tile: S' = sum (q - z_q) k differs from
// the zero-point-corrected sum by a number that is the same for every key of a row and drops out of the Softmax, so K comes
// by bulk tensor copies untouched.
//
// What bounds it: the workers' instructions (ncu, 577 keys, 64 channels: issue slots 58 % busy, a third of the issues spent on
// waits; ex2 alone takes 8 cycles of a scheduler per 32 scores) and the latency of their chains, not the tensor pipe (13 %).
// Hence:
//  - CTAs are persistent (two per SM for heads of up to 64 channels, one for wider heads) and walk their share of the
//    tiles; K tiles stream in by bulk tensor copies across tile boundaries and the Q tile of the next tile is staged during
//    pass 2 of the present one, so that its S MMAs follow without a gap (a tile of 197 keys is only eight visits: launched one
//    CTA per tile, half of its time was start and end);
//  - a worker thread has one row (its tensor-memory lane) and 32 columns of every visit, which it loads at once: one
//    barrier wait and one tensor-memory load per 32 scores, all of the warp's arithmetic independent behind it (16 columns at a
//    time with the next 16 in flight: 20 % slower, more waits and spilled registers);
//  - warps none of whose rows sees a column of theirs skip it;
//  - 4-bit codes of 4-bit values (scale s >= 1): the operands 2^(8 - ceil(p/2)) and z_v - v are 8-bit floats (e4m3), exact,
//    so P.V runs at K = 32 per instruction, and the operand bytes of eight keys are selected together from q = 15 - p in nibbles
//    (odd q: E = 0x3C + 4 q, even q: O = 0x38 + 4 q) instead of a table look-up per key (32 x 16 heads, 577 keys, block pass 398.7 ->
//    394.4 us against clipping, rounding and masking bytes key by key);
//  - wider codes take their bf16 operand pair from a per-lane table in shared memory (one bank per lane).
// Measured against one CTA per tile with two groups of warps on alternate visits: 64 x 12 heads of 64 channels with 197 keys,
// 4-bit codes, 83 -> 64 us; 32 x 16 heads, 577 keys 240 -> 192; 4 x 32 heads of 128 channels, 2048 causal keys, 8-bit codes,
// 400 -> 305.  A warp of its own for the V tiles was slower (one warp's chain of loads and conversions per visit).
// Roles: worker warps, then a warp each (one lane issues) for the S MMAs, the P.V MMAs and the K copies.  Every mbarrier wait is
// bounded; when one runs out the kernel records a status code, all roles leave their loops, MMAs and copies in flight are
// drained, tensor memory is freed and the kernel returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math_constants.h>

#include <type_traits>

#include "attention_common.cuh"

namespace repq {
namespace attn {
namespace {

constexpr int kCols = 32;                       // S columns of a thread and visit

template <int NB> struct Shape {
  static constexpr int kKeys = NB == 1 ? 64 : 128;                  // keys per visit
  static constexpr int kParts = kKeys / kCols;                      // threads that share a row
  static constexpr int kWork = 4 * kParts;                          // worker warps
  static constexpr int kWorkThreads = 32 * kWork;
  static constexpr int kThreads = kWorkThreads + 96;
  static constexpr int kCtas = NB == 1 ? 2 : 1;                     // resident per SM
  static constexpr int kK = NB == 1 ? 3 : 4;                        // K tiles in flight
  static constexpr int kTmem = 256 * NB;                            // 2 S slots + 2 accumulators
};

template <int NB, int kLutBits, bool kChains>
struct PipeShared {
  using Sh = Shape<NB>;
  static constexpr uint32_t kKBytes = Sh::kKeys * 128;
  static constexpr uint32_t kVBlockBytes = Sh::kKeys * 128;         // the visit's keys x 128 bytes (64 channels of bf16, or one row of bytes)
  alignas(1024) uint8_t q[2][kQBytes];            // of this tile and the next
  alignas(1024) uint8_t k[Sh::kK][kKBytes];
  static constexpr int kV = NB == 1 && kLutBits != 8 ? 3 : 2;       // V tiles (two where the table takes 33 KB of half an SM)
  alignas(1024) uint8_t v[kV][NB * kVBlockBytes];
  float stat_m[Sh::kParts][kRows], stat_z[Sh::kParts][kRows];
  float visit_m[kChains ? 2 : 1][kChains ? 4 : 1][kRows], visit_z[kChains ? 2 : 1][kChains ? 2 : 1][kRows];  // kChains: what two parts tell each other
  static constexpr int kLutEntries = kLutBits ? (1 << kLutBits) + 1 : 1;
  uint32_t lut[kLutEntries][32];                  // [code][lane] = E value | O value << 16; the last entry repeats the top code
                                                  // (a clamp at 2^bits that rounds up lands there)
  alignas(8) uint64_t k_full[Sh::kK];
  uint64_t k_empty[Sh::kK], v_empty[kV];
  uint64_t s_full[2], s_empty[2], s_spent[2], p_full[2];            // s_empty: read in pass 1; s_spent: P.V MMAs have read the operands
  uint64_t q_full, acc_full, acc_empty, done_s, done_pv, merged[4];   // merged: statistics of a lane quarter's rows are there
  uint64_t visit[kChains ? 8 : 1];                // kChains: both parts of a chain and lane quarter have told
  uint32_t tmem_base;
  volatile int abort;
};

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
// (the registers count as written by the wait: the compiler can neither read nor move them while the load is in flight)
__device__ __forceinline__ void tmem_ld_wait32(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                 "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                 "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29])
               :: "memory");
  asm volatile("" : "+r"(r[30]), "+r"(r[31]));
}
// D[tmem] (+)= A[tmem] * B[smem], 8-bit floats, K = 32 (a 32-bit column of A holds four consecutive K elements)
__device__ __forceinline__ void umma_f8_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// Four bytes out of the eight of (b, a), chosen by the low three bits of a nibble of `sel`; a nibble's fourth bit replicates the sign.
__device__ __forceinline__ uint32_t select_bytes(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}
__device__ __forceinline__ float fma_sat(float a, float b, float c) {       // fma clamped to [0, 1]
  float d;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Tile number `it` of CTA `cta` of `ctas`: slot by slot over all pairs.  Under a causal mask a pair's last tile comes first, and
// the tiles are dealt forwards and backwards in turn, so that every CTA gets about the same work; without a mask the short
// last tiles come last (dealt pair by pair, half of the CTAs got only the short tiles of rows of 129 to 256 queries: 64 x 12
// heads, 197 queries 64 -> 60 us, 32 x 16 heads, 577 queries 193 -> 186).
struct Tile { int bo, bi, q0, k_end, nb; };
template <int kKeys>
__device__ __forceinline__ bool tile_at(const AttnParams& P, int it, int cta, int ctas, Tile& t) {
  const int pos = it * ctas + (P.causal && (it & 1) ? ctas - 1 - cta : cta);
  if (pos >= P.pairs * P.tiles) return false;
  const int slot = div_by(pos, P.by_pairs), pair = pos - slot * P.pairs, tile = P.causal ? P.tiles - 1 - slot : slot;
  t.bo = div_by(pair, P.by_inner);
  t.bi = pair - t.bo * P.batch_inner;
  t.q0 = tile * kRows;
  t.k_end = P.causal ? max(1, min(P.Lk, min(t.q0 + kRows, P.Lq) + P.Lk - P.Lq)) : P.Lk;
  t.nb = (t.k_end + kKeys - 1) / kKeys;
  return true;
}

// v - z_v of eight codes as bf16.
struct VShift {
  __nv_bfloat162 z2;
  float z;
  __device__ __forceinline__ explicit VShift(const AttnParams& P)
      : z2(__float2bfloat162_rn(128.f + float(P.z_v))), z(12582912.f + float(P.z_v)) {}      // 1.5 * 2^23 + z_v
  __device__ __forceinline__ uint4 bf16(const uint2& c, int small) const {
    uint32_t o4[4];
    if (small) {
      // for codes below 128, 128 + v is the bit pattern 0x4300 | v and the bf16 subtraction exact
      const uint32_t w[4] = {__byte_perm(c.x, 0x43434343u, 0x4140), __byte_perm(c.x, 0x43434343u, 0x4342),
                             __byte_perm(c.y, 0x43434343u, 0x4140), __byte_perm(c.y, 0x43434343u, 0x4342)};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 hh = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&w[e]), z2);
        o4[e] = *reinterpret_cast<const uint32_t*>(&hh);
      }
    } else {
      float f[8];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        f[e] = __uint_as_float(__byte_perm(c.x, kMagicBits, 0x7650 + e)) - z;
        f[4 + e] = __uint_as_float(__byte_perm(c.y, kMagicBits, 0x7650 + e)) - z;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 hh = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
        o4[e] = *reinterpret_cast<const uint32_t*>(&hh);
      }
    }
    return make_uint4(o4[0], o4[1], o4[2], o4[3]);
  }
};

// z - v of four 4-bit codes in sign and magnitude (z at most 15, shift4 = 128 - z in every byte): t = 128 + v - z is that
// byte already where v >= z, and 128 - t is the magnitude where it is not.
__device__ __forceinline__ uint32_t zero_minus(uint32_t v, uint32_t shift4) {
  const uint32_t t = v + shift4, low = (~t >> 7) & 0x01010101u;
  return (t ^ (low * 0x7Fu)) + low;
}

// kLutBits: width of the table of operand pairs (4, 6, 8; P.V in bf16), or 0: 4-bit codes of 4-bit values, P.V in 8-bit
// floats.  kF8: 4-bit Q / K codes read as 8-bit floats (a byte below 16 is the e4m3 number byte * 2^-9; the accumulator holds
// 2^-18 sum (q - z_q) k as a float, exactly); otherwise signed x unsigned bytes.
// kChains: heads of up to 64 channels in visits of 128 keys (few tiles).  An item's Softmax sums must not depend on how many items
// share the call, so they are formed as in visits of 64 keys: two chains, the even and the odd blocks of 32 keys, each a running
// maximum m and z <- z 2^(c (m' - m)) + sum of the block.  A chain's two blocks of a visit belong to two threads, which tell each other
// their block's maximum before they sum (in shared memory, an mbarrier per pair of warps and visit); the second's sum joins a visit later.
// kBytes: the output is byte codes by 16-byte stores, as in a block; the other output forms have kernels of their own, since their code
// (10 of 50 KB) stood between what every tile runs: the warps wait for instructions (ncu, 64 x 197: two of three issues).
template <int NB, int kLutBits, bool kF8, bool kChains, bool kBytes>
__global__ void __launch_bounds__(Shape<NB>::kThreads, Shape<NB>::kCtas)
attention_pipe_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ AttnParams P) {
  static_assert(!kChains || NB == 2, "chains are those of two 64-key visits in one of 128");
  using Sh = Shape<NB>;
  using Shared = PipeShared<NB, kLutBits, kChains>;
  constexpr int kKeys = Sh::kKeys, kWork = Sh::kWork, kParts = Sh::kParts, kT = Sh::kWorkThreads, kK = Sh::kK, kV = Shared::kV;
  constexpr bool kLut = kLutBits != 0;
  constexpr int kAccCol = 2 * kKeys;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  Shared& S = *reinterpret_cast<Shared*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ksteps = (P.dh + 31) >> 5;                    // S MMAs of K = 32 per visit
  const int pieces = P.dh >> 4;                           // 16-byte pieces of a Q / K row

  if (tid == 0) {
    for (int s = 0; s < kK; ++s) { mbar_init(smem_u32(&S.k_full[s]), 1); mbar_init(smem_u32(&S.k_empty[s]), 1); }
    for (int s = 0; s < kV; ++s) mbar_init(smem_u32(&S.v_empty[s]), 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&S.s_full[s]), 1);
      mbar_init(smem_u32(&S.s_empty[s]), kWork);
      mbar_init(smem_u32(&S.s_spent[s]), 1);
      mbar_init(smem_u32(&S.p_full[s]), kWork);
    }
    mbar_init(smem_u32(&S.q_full), kWork);
    mbar_init(smem_u32(&S.acc_full), 1);
    for (int s = 0; s < 4; ++s) mbar_init(smem_u32(&S.merged[s]), kParts);
    for (int s = 0; s < (kChains ? 8 : 0); ++s) mbar_init(smem_u32(&S.visit[s]), 2);
    mbar_init(smem_u32(&S.acc_empty), kWork);
    mbar_init(smem_u32(&S.done_s), 1);
    mbar_init(smem_u32(&S.done_pv), 1);
    S.abort = 0;
    if (smem_u32(smem_raw) & 1023u) {                     // the swizzled tiles need this alignment
      atomicCAS(P.status, 0, 49);
      S.abort = 1;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kWork) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)), "n"(Sh::kTmem) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (kLut && warp < kWork) {
    for (int i = tid; i < Shared::kLutEntries * 32; i += kT) {
      const uint32_t code = min(uint32_t(i >> 5), uint32_t(Shared::kLutEntries - 2)), kk = (code + 1u) >> 1;
      const uint32_t bits16 = kk > 126u ? 0u : (127u - kk) << 7;   // bf16 bits of 2^-ceil(code/2) (0 below the normal range)
      S.lut[0][i] = (code & 1u) ? bits16 << 16 : bits16;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = S.tmem_base;
  volatile int* abort = &S.abort;
  // everything above touched no global memory of the kernel chain
  grid_dependency_wait();
  grid_dependency_trigger();

  Tile t;
  if (warp == kWork) {
    // ---------------------------------------------------------------- S MMAs
    // (the whole warp walks the loop, one lane issues: what every lane holds alike stays in uniform registers, from which these
    // instructions take their operands; with the loop in one lane a visit of two MMAs and two commits took 350 cycles.  The loops are
    // kept short, since a visit costs as many issue latencies as they have instructions)
    const bool issues = elect_one();
    // D = s32 from signed x unsigned bytes, or D = f32 from e4m3 x e4m3; both K-major, M = 128, N = the visit's keys
    constexpr uint32_t idesc = (kF8 ? (1u << 4) : (2u << 4) | (1u << 7)) | (uint32_t(kKeys >> 3) << 17) | (uint32_t(kRows >> 4) << 24);
    const uint64_t dk0 = smem_desc_sw128(smem_u32(S.k[0]));
    int g = 0;                                            // visits, over both passes and all tiles
    // a bit per slot: parity of the hand-backs waited for, whether the slot has been used, and by which pass last
    uint32_t ph_empty = 0, ph_spent = 0, used = 0, pass2 = 0;
    uint32_t ks = 0, kp = 0;                              // K ring: slot and parity
    bool ok = true;
    for (int it = 0; ok && !given_up(abort) && tile_at<kKeys>(P, it, blockIdx.x, gridDim.x, t); ++it) {
      ok = wait_for(smem_u32(&S.q_full), it & 1, abort, 40, P.status);
      const uint64_t dq = smem_desc_sw128(smem_u32(S.q[it & 1]));
#pragma unroll 1
      for (int b = 0; b < 2 * t.nb; ++b, ++g) {
        const int slot = g & 1;
        const uint32_t bit = 1u << slot;
        ok = ok && wait_for(smem_u32(&S.k_full[ks]), kp, abort, 41, P.status);
        if (ok && (used & bit)) {
          const bool spent = (pass2 & bit) != 0;
          ok = wait_for(spent ? smem_u32(&S.s_spent[slot]) : smem_u32(&S.s_empty[slot]), ((spent ? ph_spent : ph_empty) >> slot) & 1u, abort, 42,
                        P.status);
          if (spent) ph_spent ^= bit; else ph_empty ^= bit;
        }
        if (!(ok = __all_sync(0xffffffffu, ok))) break;   // (all lanes leave together)
        used |= bit;
        pass2 = b >= t.nb ? pass2 | bit : pass2 & ~bit;
        tc_fence_after();
        if (issues) {
          const uint64_t dk = dk0 + uint64_t(ks * (Shared::kKBytes >> 4));
          const uint32_t d = tmem_base + uint32_t(slot * kKeys);
#pragma unroll
          for (int s = 0; s < 2 * NB; ++s) {
            if (s < ksteps) {
              if (kF8) umma_f8(d, dq + uint64_t(2 * s), dk + uint64_t(2 * s), idesc, s != 0 ? 1u : 0u);
              else umma_i8(d, dq + uint64_t(2 * s), dk + uint64_t(2 * s), idesc, s != 0 ? 1u : 0u);
            }
          }
          umma_commit(smem_u32(&S.s_full[slot]));
          umma_commit(smem_u32(&S.k_empty[ks]));
        }
        __syncwarp();
        if (++ks == kK) { ks = 0; kp ^= 1u; }
      }
    }
    if (issues) umma_commit(smem_u32(&S.done_s));
    __syncwarp();
    mbar_drain(smem_u32(&S.done_s), 0);
  } else if (warp == kWork + 1) {
    // ---------------------------------------------------------------- P.V MMAs
    const bool issues = elect_one();
    // D = f32, A (tensor memory) and B = bf16 or e4m3, B MN-major, N = n_pad, M = 128
    const uint32_t idesc = (kLut ? (1u << 4) | (1u << 7) | (1u << 10) : (1u << 4)) | (1u << 16) | (uint32_t(P.n_pad >> 3) << 17) |
                           (uint32_t(kRows >> 4) << 24);
    constexpr int kStep = kLut ? 16 : 32;                 // keys per MMA
    const uint64_t dv0 = smem_desc_sw128(smem_u32(S.v[0]), Shared::kVBlockBytes);
    const uint32_t d_e = tmem_base + uint32_t(kAccCol), d_o = d_e + uint32_t(P.n_pad);
    int g = 0;
    uint32_t ph_p = 0, vs = 0;
    bool ok = true;
    for (int it = 0; ok && !given_up(abort) && tile_at<kKeys>(P, it, blockIdx.x, gridDim.x, t); ++it) {
      g += t.nb;
      if (it > 0) ok = wait_for(smem_u32(&S.acc_empty), (it - 1) & 1, abort, 50, P.status);
#pragma unroll 1
      for (int j = 0; j < t.nb; ++j, ++g) {
        const int slot = g & 1;
        ok = ok && wait_for(smem_u32(&S.p_full[slot]), (ph_p >> slot) & 1u, abort, 43, P.status);
        if (!(ok = __all_sync(0xffffffffu, ok))) break;
        ph_p ^= 1u << slot;
        tc_fence_after();
        const int left = t.k_end - j * kKeys;             // keys from the visit's first on
        if (issues) {
          const uint64_t dv = dv0 + uint64_t(vs * (NB * Shared::kVBlockBytes >> 4));
          const uint32_t a_base = tmem_base + uint32_t(slot * kKeys);
#pragma unroll
          for (int s = 0; s < kKeys / kStep; ++s) {
            if (s * kStep < left) {
              const uint32_t accumulate = s != 0 ? 1u : j != 0 ? 1u : 0u;
              const uint64_t b = dv + uint64_t(kStep * 128 / 16 * s);
              const uint32_t a_e = a_base + uint32_t(kStep * s);       // E words first, then as many O words
              if (kLut) {
                umma_f16_ts(d_e, a_e, b, idesc, accumulate);
                umma_f16_ts(d_o, a_e + 8u, b, idesc, accumulate);
              } else {
                umma_f8_ts(d_e, a_e, b, idesc, accumulate);
                umma_f8_ts(d_o, a_e + 8u, b, idesc, accumulate);
              }
            }
          }
          umma_commit(smem_u32(&S.s_spent[slot]));
          umma_commit(smem_u32(&S.v_empty[vs]));
          if (j + 1 == t.nb) umma_commit(smem_u32(&S.acc_full));
        }
        __syncwarp();
        if (++vs == kV) vs = 0;
      }
    }
    if (issues) umma_commit(smem_u32(&S.done_pv));
    __syncwarp();
    mbar_drain(smem_u32(&S.done_pv), 0);
  } else if (warp == kWork + 2) {
    // ---------------------------------------------------------------- K tiles by bulk tensor copies
    const bool issues = elect_one();
    uint32_t ks = 0, kp = 0;
    int issued = 0;
    bool ok = true;
    for (int it = 0; ok && !given_up(abort) && tile_at<kKeys>(P, it, blockIdx.x, gridDim.x, t); ++it) {
#pragma unroll 1
      for (int b = 0; b < 2 * t.nb; ++b) {
        ok = wait_for(smem_u32(&S.k_empty[ks]), kp ^ 1u, abort, 48, P.status);
        if (!(ok = __all_sync(0xffffffffu, ok))) break;
        const uint32_t bar = smem_u32(&S.k_full[ks]);
        // box: 128 bytes of the head's row (bytes past d_h meet zero bytes of the Q tile), the visit's keys (rows past Lk
        // are zero-filled), one batch item
        if (issues) {
          mbar_expect_tx(bar, Shared::kKBytes);
          tma_load_3d(smem_u32(S.k[ks]), &map_k, bar, t.bi * int(P.k_si), (b < t.nb ? b : b - t.nb) * kKeys, t.bo);
        }
        __syncwarp();
        ++issued;
        if (++ks == kK) { ks = 0; kp ^= 1u; }
      }
    }
    // the copies issued last must have landed before this CTA may exit
    for (int i = issued < kK ? issued : kK; i > 0; --i) {
      if (ks == 0) { ks = kK - 1; kp ^= 1u; } else { --ks; }
      mbar_drain(smem_u32(&S.k_full[ks]), kp);
    }
  } else {
    // ---------------------------------------------------------------- Softmax arithmetic, V tiles, epilogue
    const int quarter = warp & 3, part = warp >> 2;
    const int r = quarter * 32 + lane;                    // the thread's row inside the tile = its tensor-memory lane
    const float c = 1.4426950408889634f;
    const float magic = __uint_as_float(kMagicBits);
    const uint32_t taddr_s = tmem_base + (uint32_t(quarter * 32) << 16) + uint32_t(part * kCols);
    const uint32_t lut_addr = smem_u32(&S.lut[0][lane]) - (kMagicBits << 7);

    // ---- Q tile: q - z_q as signed bytes (kF8: sign and magnitude), two 16-byte pieces per thread.  The next tile's is
    // requested and written during the first visit of pass 2, into the other of two buffers, so that the next tile's S MMAs
    // follow this tile's without a gap.
    constexpr int kQRow = 4 * NB, kQPer = 2;              // pieces of a row (64 or 128 channels) and of a thread
    static_assert(kRows * kQRow == kQPer * kT, "every piece of the Q tile has a thread");
    const int qrow = tid / (kQRow / kQPer), qp0 = (tid % (kQRow / kQPer)) * kQPer;
    const uint32_t zq4 = uint32_t(P.zq) * 0x01010101u;
    uint4 qreg[kQPer];
    auto fetch_q = [&](const Tile& n) {
      const uint8_t* row = P.q + n.bo * P.q_so + n.bi * P.q_si + int64_t(n.q0 + qrow) * P.ldq;
#pragma unroll
      for (int i = 0; i < kQPer; ++i) {
        qreg[i] = make_uint4(zq4, zq4, zq4, zq4);
        if (n.q0 + qrow < P.Lq && qp0 + i < pieces) qreg[i] = __ldg(reinterpret_cast<const uint4*>(row) + qp0 + i);
      }
    };
    auto stage_q = [&](uint8_t* tile) {
#pragma unroll
      for (int i = 0; i < kQPer; ++i) {
        uint4 w = sub_bytes(qreg[i], zq4);
        if (kF8) w = sign_magnitude(w);
        if (qp0 + i < 2 * ksteps) *reinterpret_cast<uint4*>(tile + tile_offset(qrow, qp0 + i)) = w;
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&S.q_full));
    };

    // ---- V tile of a visit.  8-bit floats: a thread has one key and 16 channels, z_v - v in sign and magnitude (byte * 2^-9).
    // bf16: a thread keeps its group of 8 channels and moves down the keys, 32 per step.
    using VRaw = typename std::conditional<kLut, uint2, uint4>::type;
    constexpr int kVItems = kLut ? kKeys / 32 : 1, kVChan = kLut ? 8 : 16, kVGroups = (kLut ? 64 * NB : 64) / kVChan;
    const int v_g = tid % kVGroups, v_key0 = tid / kVGroups;
    const bool v_live = v_g * kVChan < P.dh;
    const uint32_t v_off = kLut ? uint32_t(v_g >> 3) * Shared::kVBlockBytes + tile_offset(v_key0, v_g & 7) : tile_offset(v_key0, v_g);
    const VShift vshift(P);
    const uint32_t shift4 = (128u - uint32_t(P.z_v)) * 0x01010101u;
    const uint8_t* v_ptr = nullptr;
    VRaw vraw[kVItems];
    auto fetch_v = [&](int block) {
      const uint8_t* p = v_ptr + int64_t(block * kKeys) * P.ldv;
#pragma unroll
      for (int i = 0; i < kVItems; ++i)
        if (v_live && block * kKeys + v_key0 + i * 32 < t.k_end) vraw[i] = __ldg(reinterpret_cast<const VRaw*>(p + int64_t(i * 32) * P.ldv));
    };
    auto stage_v = [&](int block, uint8_t* tile) {
#pragma unroll
      for (int i = 0; i < kVItems; ++i) {
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (v_live && block * kKeys + v_key0 + i * 32 < t.k_end) {
          if constexpr (kLut) w = vshift.bf16(vraw[i], P.v_small);
          else w = make_uint4(zero_minus(vraw[i].x, shift4), zero_minus(vraw[i].y, shift4), zero_minus(vraw[i].z, shift4), zero_minus(vraw[i].w, shift4));
        }
        *reinterpret_cast<uint4*>(tile + v_off + uint32_t(i) * 4096u) = w;
      }
    };

    // The thread's 32 scores of the visit in `slot`, in units of the score scale, as floats: the accumulators themselves
    // (kF8) or converted.
    auto load_scores = [&](int slot, float (&sf)[kCols]) {
      uint32_t rn[kCols];
      __syncwarp();
      tmem_ld32(taddr_s + uint32_t(slot * kKeys), rn);
      tmem_ld_wait32(rn);
#pragma unroll
      for (int e = 0; e < kCols; ++e) sf[e] = kF8 ? __uint_as_float(rn[e]) : float(int32_t(rn[e]));
    };

    float m = -CUDART_INF_F, z = 0.f;       // running maximum (in units of the score scale) and sum of this thread's columns
    const float sc = P.scale * c;           // exponent of 2 per unit
    // Largest of `start` and the thread's scores, and sum of 2^(sc (sf - mn)) over them: of all columns, or of the columns e < seen.
    auto max_all = [&](const float (&sf)[kCols], float start) {
      float b0 = max3(sf[0], sf[1], sf[2]), b1 = max3(sf[3], sf[4], sf[5]);
#pragma unroll
      for (int e = 6; e + 3 < kCols; e += 4) { b0 = max3(b0, sf[e], sf[e + 1]); b1 = max3(b1, sf[e + 2], sf[e + 3]); }
      return fmaxf(max3(start, b0, b1), fmaxf(sf[kCols - 2], sf[kCols - 1]));
    };
    auto sum_all = [&](const float (&sf)[kCols], float mn) {
      const f32x2 sc2 = splat2(sc), nm2 = splat2(-(mn * sc));
      f32x2 acc[2] = {0ull, 0ull};
#pragma unroll
      for (int e = 0; e < kCols; e += 2) {
        float a0, a1;
        unpack2(fma2(pack2(sf[e], sf[e + 1]), sc2, nm2), a0, a1);
        acc[(e >> 1) & 1] = add2(acc[(e >> 1) & 1], pack2(ex2(a0), ex2(a1)));
      }
      float z0, z1;
      unpack2(add2(acc[0], acc[1]), z0, z1);
      return z0 + z1;
    };
    auto max_some = [&](const float (&sf)[kCols], int seen, float start) {
      float bm = sf[0];
#pragma unroll
      for (int e = 1; e < kCols; ++e)
        if (e < seen) bm = fmaxf(bm, sf[e]);
      return fmaxf(start, bm);
    };
    auto sum_some = [&](const float (&sf)[kCols], int seen, float mn) {
      const float nm = -(mn * sc);
      float acc = 0.f;
#pragma unroll
      for (int e = 0; e < kCols; ++e)
        if (e < seen) acc += ex2(fmaf(sf[e], sc, nm));
      return acc;
    };
    // `seen`: columns e < seen are keys the row sees
    auto stats = [&](const float (&sf)[kCols], int seen) {
      if (__builtin_expect(seen >= kCols, 1)) {
        const float mn = max_all(sf, m);
        z = fmaf(z, ex2((m - mn) * sc), sum_all(sf, mn));               // m = -inf at first: factor 0
        m = mn;
      } else if (seen > 0) {
        const float mn = max_some(sf, seen, m);
        z = fmaf(z, ex2((m - mn) * sc), sum_some(sf, seen, mn));
        m = mn;
      }
    };
    // kChains: m is the chain's maximum after the visit, `mid` between its two blocks; z and `mid` belong to the first part, the
    // second's `block_z` waits for the next visit.  A block without keys is one of maximum -inf and sum 0: it changes no bit.
    float mid = -CUDART_INF_F, block_z = 0.f;
    int told = 0;                           // visits of pass 1, over all tiles
    auto chain_stats = [&](const float (&sf)[kCols], int seen) -> bool {
      auto sum = [&](float mn) { return seen >= kCols ? sum_all(sf, mn) : seen > 0 ? sum_some(sf, seen, mn) : 0.f; };
      const int at = told & 1;
      const float none = -CUDART_INF_F, own = seen >= kCols ? max_all(sf, none) : seen > 0 ? max_some(sf, seen, none) : none;
      S.visit_m[at][part][r] = own;
      if (part >= 2) S.visit_z[at][part & 1][r] = block_z;
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&S.visit[warp & 7]));
      if (!wait_for(smem_u32(&S.visit[warp & 7]), told & 1, abort, 51, P.status)) return false;
      ++told;
      const float other = S.visit_m[at][part ^ 2][r];
      if (part < 2) {
        if (m > -CUDART_INF_F) z = fmaf(z, ex2((mid - m) * sc), S.visit_z[at][part][r]);
        mid = fmaxf(m, own);
        if (mid > -CUDART_INF_F) z = fmaf(z, ex2((m - mid) * sc), sum(mid));
        m = fmaxf(mid, other);
      } else {
        m = fmaxf(fmaxf(m, other), own);
        block_z = sum(m);
      }
      return true;
    };

    float w1 = 0.f, w0 = 0.f;               // pass 2: the code is a rounded and clipped w1 (sf - m) + w0
    // Codes and operand words of the thread's 32 columns, stored over the columns the scores came from.
    auto codes = [&](const float (&sf)[kCols], int seen, uint32_t taddr) {
      const f32x2 nm2 = splat2(-m);
      if constexpr (!kLut) {
        // q = 15 - p: u = 15 - t times 2^-149 is a denormal whose bit pattern is round(u) (half to even; negative below zero), which the
        // pack instruction clips to [0, 15] and gathers, a nibble per key.  Turned right by one bit, a nibble is what the byte
        // selection takes: three bits that choose one of eight operand bytes, and a fourth that puts the sign of that byte, 0, in
        // its place where the parity is the other operand's.
        const f32x2 w12 = splat2(w1), w02 = splat2(w0), tiny2 = splat2(__uint_as_float(1u));
        uint32_t eo[16];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t q = 0u;
#pragma unroll
          for (int h = 3; h >= 0; --h) {
            const f32x2 d = add2(pack2(sf[8 * i + 2 * h], sf[8 * i + 2 * h + 1]), nm2);
            float u0, u1;
            unpack2(mul2(fma2(d, w12, w02), tiny2), u0, u1);
            q = push_pair_u4(__float_as_int(u0), __float_as_int(u1), q);
          }
          const uint32_t sel_o = ((q >> 1) & 0x77777777u) | ((q << 3) & 0x88888888u), sel_e = sel_o ^ 0x88888888u;
          eo[2 * i] = select_bytes(0x58504840u, 0x78706860u, sel_e);
          eo[2 * i + 1] = select_bytes(0x58504840u, 0x78706860u, sel_e >> 16);
          eo[8 + 2 * i] = select_bytes(0x50484038u, 0x70686058u, sel_o);
          eo[8 + 2 * i + 1] = select_bytes(0x50484038u, 0x70686058u, sel_o >> 16);
        }
        if (__builtin_expect(seen < kCols, 0)) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int n = seen - 4 * i;
            const uint32_t keep = n >= 4 ? 0xFFFFFFFFu : n > 0 ? (1u << (8 * n)) - 1u : 0u;
            eo[i] &= keep;
            eo[8 + i] &= keep;
          }
        }
        __syncwarp();
        tmem_st16(taddr, eo);
      } else {
        constexpr float kSteps = float(1 << kLutBits);
        const f32x2 steps2 = splat2(kSteps), magic2 = splat2(magic);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t eo[16], eow[16];
#pragma unroll
          for (int e = 0; e < 16; e += 2) {
            float d0, d1, u0, u1;
            unpack2(add2(pack2(sf[16 * h + e], sf[16 * h + e + 1]), nm2), d0, d1);
            unpack2(fma2(pack2(fma_sat(d0, w1, w0), fma_sat(d1, w1, w0)), steps2, magic2), u0, u1);
            asm("ld.shared.u32 %0, [%1];" : "=r"(eo[e]) : "r"(lut_addr + (__float_as_uint(u0) << 7)));
            asm("ld.shared.u32 %0, [%1];" : "=r"(eo[e + 1]) : "r"(lut_addr + (__float_as_uint(u1) << 7)));
          }
          if (__builtin_expect(seen < 16 * h + 16, 0)) {
#pragma unroll
            for (int e = 0; e < 16; ++e)
              if (16 * h + e >= seen) eo[e] = 0u;
          }
          // E pairs (even key in the low half) in words 0..7, O pairs in words 8..15
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            eow[e] = __byte_perm(eo[2 * e], eo[2 * e + 1], 0x5410);
            eow[8 + e] = __byte_perm(eo[2 * e], eo[2 * e + 1], 0x7632);
          }
          __syncwarp();
          tmem_st16(taddr + uint32_t(16 * h), eow);
        }
      }
    };

    // ---- epilogue of tile `it`: one row per thread (`roff`: its output offset, -1: past Lq), the 16-column chunks of the
    // accumulators dealt to the parts of a row
    auto finish = [&](int it, int64_t roff, int64_t sum_at) -> bool {
              if (!wait_for(smem_u32(&S.acc_full), it & 1, abort, 47, P.status)) return false;
              tc_fence_after();
              const float out_scale = kLut ? P.out_scale : -2.f * P.out_scale;  // 8-bit floats: 2^8 A times 2^-9 (z_v - v)
              const uint32_t taddr = tmem_base + (uint32_t(quarter * 32) << 16) + uint32_t(kAccCol);
              int code_sum = 0;
      #pragma unroll 1
              for (int c0 = part * 16; c0 < P.dh; c0 += kParts * 16) {
                uint32_t re[16], ro[16];
                __syncwarp();
                tmem_ld16(taddr + uint32_t(c0), re);
                tmem_ld16(taddr + uint32_t(P.n_pad + c0), ro);
                tmem_ld_wait(re);
                tmem_ld_wait(ro);
                if (c0 + kParts * 16 >= P.dh) {                 // the thread's last chunk: the accumulators may be written again
                  tc_fence_before();
                  __syncwarp();
                  if (lane == 0) mbar_arrive(smem_u32(&S.acc_empty));
                }
                float v[16];
                const f32x2 root2 = splat2(1.41421356237309504880f), scale2 = splat2(out_scale);
      #pragma unroll
                for (int e = 0; e < 16; e += 2)
                  unpack2(mul2(scale2, fma2(root2, pack2(__uint_as_float(ro[e]), __uint_as_float(ro[e + 1])),
                                            pack2(__uint_as_float(re[e]), __uint_as_float(re[e + 1])))), v[e], v[e + 1]);
                if (roff >= 0) {
                  if constexpr (kBytes) store_codes(P, v, roff, c0, code_sum);
                  else store_values(P, v, roff, c0, code_sum);
                }
              }
              if (part * 16 >= P.dh) {                          // no chunk for this thread
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&S.acc_empty));
              } else if (roff >= 0 && P.out_row_sum != nullptr && (kBytes || P.out_kind == REPQ_OUT_CODES)) {
                atomicAdd(P.out_row_sum + sum_at, code_sum);
              }
      return true;
    };

    // Where one CTA has the SM (wide heads), the epilogue waits until the next tile's pass 1 is through, under which the tile's
    // last MMAs complete; where two share it, the other one runs meanwhile and the epilogue follows at once (measured: 64 x 12
    // heads of 64 channels, 197 keys, 64 against 77 us; 4 x 32 heads of 128 channels, 2048 causal keys, 325 against 310).
    constexpr bool kDefer = NB != 1;
    bool ok = true, more = tile_at<kKeys>(P, 0, blockIdx.x, gridDim.x, t);
    int g = 0;                                            // visits, over both passes and all tiles
    uint32_t vs = 0, vp = 0;                              // V ring: stage and parity
    int64_t done_row = -1, done_sum = 0;                  // the tile before: output offset and row-sum index of the thread's row, -1: past Lq
    if (more) { fetch_q(t); stage_q(S.q[0]); }
    for (int it = 0; !*abort; ++it) {
      const int row = more ? t.q0 + r : P.Lq;
      const int valid = row < P.Lq ? (P.causal ? max(1, min(P.Lk, row + 1 + P.Lk - P.Lq)) : P.Lk) : 0;   // keys the row sees
      const int most = __reduce_max_sync(0xffffffffu, valid);                                             // ... any row of the warp
      // ---- pass 1
      if (more) {
        v_ptr = P.v + t.bo * P.v_so + t.bi * P.v_si + int64_t(v_key0) * P.ldv + v_g * kVChan;
        if (kDefer) fetch_v(0);
        m = mid = -CUDART_INF_F;
        z = block_z = 0.f;
        for (int b = 0; b < t.nb; ++b, ++g) {
          const int slot = g & 1, first = b * kKeys + part * kCols;
          if (!wait_for(smem_u32(&S.s_full[slot]), (g >> 1) & 1, abort, 44, P.status)) { ok = false; break; }
          if (first < most) {                             // (warps whose columns no row sees only hand the slot back)
            tc_fence_after();
            float sf[kCols];
            load_scores(slot, sf);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&S.s_empty[slot]));
            if constexpr (!kChains) stats(sf, valid - first);
            else if (!chain_stats(sf, valid - first)) { ok = false; break; }
          } else {
            if (lane == 0) mbar_arrive(smem_u32(&S.s_empty[slot]));
            if constexpr (kChains) {
              const float none[kCols] = {};
              if (!chain_stats(none, 0)) { ok = false; break; }
            }
          }
        }
        if (!ok || *abort) break;
        if (!kDefer) fetch_v(0);
        // the column parts of a row are merged below
        S.stat_m[part][r] = kChains && part < 2 ? mid : m;
        S.stat_z[part][r] = kChains && part >= 2 ? block_z : z;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&S.merged[quarter]));
      }
      if (kDefer && it > 0 && !finish(it - 1, done_row, done_sum)) break;
      if (!more) break;
      if (!wait_for(smem_u32(&S.merged[quarter]), it & 1, abort, 45, P.status)) break;
      // m = max, Z = sum of the rescaled partial sums (same order in every thread of the row, so that all hold the same Z)
      float zt = 0.f;
#pragma unroll
      for (int q = 0; q < kParts; ++q) m = fmaxf(m, S.stat_m[q][r]);
#pragma unroll
      for (int q = 0; q < (kChains ? 2 : kParts); ++q) {
        float mq = S.stat_m[q][r], zq = S.stat_z[q][r];
        if constexpr (kChains) {                            // the second part's last block
          const float mid_q = mq;
          mq = S.stat_m[q + 2][r];
          zq = fmaf(zq, ex2((mid_q - mq) * sc), S.stat_z[q + 2][r]);
        }
        if (mq > -CUDART_INF_F) zt = fmaf(zq, ex2((mq - m) * sc), zt);
      }
      {
        const float k0 = 2.f * (log2f(zt) + P.log2_s);
        if (kLut) {
          constexpr float kInv = 1.f / float(1 << (kLut ? kLutBits : 4));
          w1 = -2.f * sc * kInv;
          w0 = k0 * kInv;
        } else {
          w1 = 2.f * sc;
          w0 = 15.f - k0;
        }
      }
      // ---- pass 2
      for (int j = 0; j < t.nb; ++j, ++g) {
        const int slot = g & 1, first = j * kKeys + part * kCols;
        if (!wait_for(smem_u32(&S.v_empty[vs]), vp ^ 1u, abort, 46, P.status)) { ok = false; break; }
        stage_v(j, S.v[vs]);
        if (j + 1 < t.nb) fetch_v(j + 1);
        fence_async_smem();
        if (++vs == kV) { vs = 0; vp ^= 1u; }
        if (j == 0) {
          Tile next;
          more = tile_at<kKeys>(P, it + 1, blockIdx.x, gridDim.x, next);
          if (more) fetch_q(next);
        }
        if (!wait_for(smem_u32(&S.s_full[slot]), (g >> 1) & 1, abort, 44, P.status)) { ok = false; break; }
        // columns past the visit's last key are read by the MMAs only inside the step that holds it
        if (first < t.k_end) {
          tc_fence_after();
          const uint32_t taddr = taddr_s + uint32_t(slot * kKeys);
          if (first < most) {
            float sf[kCols];
            load_scores(slot, sf);
            codes(sf, valid - first, taddr);
          } else {
            const uint32_t zero[16] = {};
            __syncwarp();
            tmem_st16(taddr, zero);
            if (kLut) tmem_st16(taddr + 16u, zero);
          }
          tmem_st_wait();
          tc_fence_before();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&S.p_full[slot]));
        if (j == 0 && more) stage_q(S.q[(it + 1) & 1]);   // (the buffer's last reader: the S MMAs of the tile before this one)
      }
      if (!ok || *abort) break;
      done_row = row < P.Lq ? t.bo * P.o_so + t.bi * P.o_si + int64_t(row) * P.ldo : -1;
      done_sum = int64_t(t.bo) * P.Lq + row;
      if (!kDefer && !finish(it, done_row, done_sum)) break;
      if (more) tile_at<kKeys>(P, it + 1, blockIdx.x, gridDim.x, t);
    }
  }

  // ------------------------------------------------------------------ teardown
  if (warp < kWork) tmem_st_wait();               // an error path may leave a tensor-memory store in flight
  tc_fence_before();
  __syncthreads();
  if (warp == kWork) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(Sh::kTmem) : "memory");
  }
}

template <int NB, int kLutBits, bool kF8, bool kChains, bool kBytes>
repq_status launch_form_out(const AttnParams& P, int64_t pairs, cudaStream_t st) {
  using Sh = Shape<NB>;
  constexpr size_t smem = sizeof(PipeShared<NB, kLutBits, kChains>);
  static_assert(smem <= (NB == 1 ? 113 : 227) * 1024, "shared storage exceeds a CTA's share");
  REPQ_TRY((allow_smem<attention_pipe_kernel<NB, kLutBits, kF8, kChains, kBytes>>(int(smem))));
  AttnParams Q = P;
  Q.pairs = int(pairs);
  Q.tiles = (P.Lq + kRows - 1) / kRows;
  Q.by_pairs = fixed_div(uint32_t(pairs));
  Q.by_inner = fixed_div(uint32_t(P.batch_inner));
  if (kF8) Q.scale = P.scale * 262144.f;                  // the accumulators hold 2^-18 sum (q - z_q) k
  CUtensorMap map_k;
  REPQ_TRY(make_k_map(&map_k, P, int(pairs / P.batch_inner), Sh::kKeys));
  const int64_t tiles = int64_t(Q.tiles) * pairs, slots = int64_t(sm_count()) * Sh::kCtas;
  const dim3 grid{unsigned(tiles < slots ? tiles : slots)};
  REPQ_CUDA(launch_chained(attention_pipe_kernel<NB, kLutBits, kF8, kChains, kBytes>, grid, dim3(Sh::kThreads), smem, st, map_k, Q));
  note_launch();
  return REPQ_OK;
}

template <int NB, int kLutBits, bool kF8, bool kChains = false>
repq_status launch_kernel(const AttnParams& P, int64_t pairs, cudaStream_t st) {
  return P.out_kind == REPQ_OUT_CODES && !P.pack4 && P.vec_store ? launch_form_out<NB, kLutBits, kF8, kChains, true>(P, pairs, st)
                                                                 : launch_form_out<NB, kLutBits, kF8, kChains, false>(P, pairs, st);
}

template <bool kF8>
repq_status launch_form(const AttnParams& P, int64_t pairs, bool small_v, cudaStream_t st) {
  // Heads of up to 64 channels: two CTAs per SM with visits of 64 keys, except where every tile has an SM to itself; then the
  // tile's chain of visits is all there is, and half as many visits of 128 keys (16 worker warps) shorten it.  A pass of a
  // W4A4 block: one image of 577 tokens and 16 heads 62.5 -> 53.8 us, 8 of 197 and 6 heads 47.0 -> 41.4, one, float32 32.8 -> 32.2 (W6A6,
  // 2 of 197 and 12 heads 49.3 -> 45.6; of these 0.6 to 1.7 go to forming the sums as the 64-key form does).  Up to 64 keys there
  // is a single visit either way, and fewer than 32 tiles with up to 191 keys gain no whole visit of 128 (6 heads, 4-bit, one image of 129
  // keys 31.4 against 31.7, of 160 31.4 and 31.9, 6-bit 32.1 and 32.8; two images of 128 33.2 and 31.8).
  const int64_t tiles = int64_t((P.Lq + kRows - 1) / kRows) * pairs;
  const bool f8_pv = P.dh <= 64 && P.qmax_p <= 15 && small_v && P.log2_s >= 0.f;
  const bool short_keys = P.Lk <= 64 || (tiles < 32 && P.Lk < 192 && P.Lk != 128);
  if (P.dh <= 64 && (short_keys || tiles > sm_count())) {
    // 4-bit codes of 4-bit values: P.V in 8-bit floats (V rows by 16-byte loads; s >= 1 keeps t >= 0)
    if (P.qmax_p <= 15)
      return f8_pv ? launch_kernel<1, 0, kF8>(P, pairs, st) : launch_kernel<1, 4, kF8>(P, pairs, st);
    if (P.qmax_p <= 63) return launch_kernel<1, 6, kF8>(P, pairs, st);
    return launch_kernel<1, 8, kF8>(P, pairs, st);
  }
  if (P.dh <= 64) {
    if (P.qmax_p <= 15) return f8_pv ? launch_kernel<2, 0, kF8, true>(P, pairs, st) : launch_kernel<2, 4, kF8, true>(P, pairs, st);
    if (P.qmax_p <= 63) return launch_kernel<2, 6, kF8, true>(P, pairs, st);
    return launch_kernel<2, 8, kF8, true>(P, pairs, st);
  }
  if (P.qmax_p <= 15) return launch_kernel<2, 4, kF8>(P, pairs, st);
  if (P.qmax_p <= 63) return launch_kernel<2, 6, kF8>(P, pairs, st);
  return launch_kernel<2, 8, kF8>(P, pairs, st);
}

}  // namespace

// q - z_q as signed bytes (codes and zero points below 128) and row and batch strides of K usable as tensor-map strides
bool pipe_supported(const AttnParams& P, int qmax_qk) {
  return qmax_qk < 128 && P.zq >= 0 && P.zq < 128 && P.zk >= 0 && P.zk < 128 && P.k_so > 0 && P.ldk < (int64_t(1) << 40) &&
         P.k_so < (int64_t(1) << 40) && int64_t(P.batch_inner - 1) * P.k_si + P.dh <= P.ldk;
}

repq_status launch_pipe(const AttnParams& P, int64_t pairs, int qmax_qk, cudaStream_t st) {
  // 4-bit quantizers with the zero point of Q inside the code range: the tiles are also valid 8-bit floats
  const bool f8 = qmax_qk <= 15 && P.zq <= 15 && !P.no_f8;
  const bool small_v = qmax_qk <= 15 && P.z_v >= 0 && P.z_v <= 15 && aligned(P.v, 16) && P.ldv % 16 == 0 && P.v_so % 16 == 0 && P.v_si % 16 == 0;
  return f8 ? launch_form<true>(P, pairs, small_v, st) : launch_form<false>(P, pairs, small_v, st);
}

}  // namespace attn
}  // namespace repq
