// Integer GEMM for few tokens (decoding, short prompts, single images): the weights are the M = 128 operand of the
// tensor-core instruction and the tokens its N operand, so that a tile is 128 output channels x 16..128 tokens and no
// tensor-core row is spent on padding of the token side.
//
// What bounds it: with few tokens a layer is one pass over its weights, i.e. the HBM (or, for weights that fit, L2) copy
// rate, and below some 2 MB of weights the latency of one tile.  Both ask for many CTAs with many bytes in flight each:
//  - a tile's K range is split over the CTAs of a cluster (1, 2, 4 or 8); the int32 partial sums are exchanged through
//    distributed shared memory, every CTA finishing an equal share of the tile's tokens (integer sums: the result does
//    not depend on the split).  They are sent as soon as a CTA has them, by stores that a barrier of the receiver counts: 1.4 us from
//    the last MMA to the sums (48 x 4096 x 4096, clusters of four), 2.4 with two barriers of the cluster around plain stores;
//  - two CTAs per SM of 110 KB where the CTAs of a call do not all find an SM of their own.  Where they do they take 200 KB each: a deeper ring,
//    and no two CTAs on one SM while others idle (128 CTAs sat on 90 SMs; block pass of 48 tokens 72.1 -> 69.5 us);
//  - what stands behind the main loop is run through once before it ends where it is long enough (`dry` below): the code (24-45 KB, out of L2 since the
//    weights of a layer passed through it) and a chunk's residual and rotation values are near when the sums arrive;
//  - inside a block, while the kernel before it in the stream still runs, every CTA asks for its first weights
//    (activations and outputs, and weights that the kernel before may have written, are touched only behind the dependency).
// The epilogue has one output channel per thread (the channel's terms live in registers), tokens along the accumulator
// columns; for one token the 32 lanes of a warp are 32 neighbouring outputs, so loads and stores are coalesced without
// staging.  The arithmetic is epilogue.cuh's, element by element.
//
// Measured (block passes, 7B-shaped decoder layer of 48 tokens, one byte per weight code): 1860 -> 69.5 us against the warp-MMA
// kernel (2.9 TB/s of weights over the whole pass, all seven kernels included); one image through a ViT-S block 52 -> 30 us
// against 128-row tiles, of which so small a layer fills only a handful of SMs.  Of the 69.5, weights stream for 34 (at 4.9 to 6.7 TB/s);
// 16 to 96 MB of the widest layer's weights brought into L2 while attention runs changed nothing (-0.3 to +3.6).
//
// Every wait on an mbarrier is bounded as in the other tensor-core kernels; all threads reach the two cluster barriers, and every
// CTA sends its sums, whether or not a wait ran out.
#include <cuda.h>
#include <cuda_bf16.h>

#include <type_traits>

#include "kernels.h"
#include "tc_ptx.cuh"

namespace repq {
namespace {

using namespace tc;

constexpr int kRowsW = 128;                 // output channels per tile (MMA M)
constexpr int kBK = 128;                    // codes per k-block
constexpr int kEpiWarps = 8;                // two per tensor-memory lane quarter
constexpr int kThreads = 32 * (kEpiWarps + 2);
constexpr int kTok = 8;                     // tokens per tensor-memory load
constexpr int kMaxStages = 8;
constexpr uint32_t kWBytes = kRowsW * kBK;
constexpr uint32_t kChunkBytes = kTok * kRowsW * 4;      // partial sums of a chunk
constexpr int kMaxTokens = 128;           // tokens per tile at most
constexpr int kPrefetch = 8;                // k-blocks of weights brought into L2 ahead of the dependency wait (all of a
                                            // CTA's blocks at once crowd out the running kernel's own loads: 83 -> 88 us for
                                            // a 7B-shaped decoder block of 48 tokens)
constexpr int kSmemTwo = 110 * 1024;        // shared memory of a CTA, two resident (227 KB per SM less the static part)
constexpr int kSmemOne = 200 * 1024;        // ... where no SM needs to take two

struct SkinnyParams {
  int M, N, K;
  int mt;                      // tokens per tile (multiple of 16)
  int stages, kblocks, split;
  int weights_settled;         // the weights may be read ahead of the dependency wait
  int dry;                     // the epilogue's code and first values are brought near while the main loop runs
  int over_ring;               // the partial sums of a cluster's CTAs are exchanged over the ring instead of behind it
  uint32_t stage_bytes, a_bytes;
  uint32_t tmem_cols;
  const int32_t* asum;
  const int32_t* wsum;
  int32_t* status;
  EpilogueParams ep;
};

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}
// 16 bytes into the shared memory of a CTA of the cluster, counted by a barrier of that CTA
__device__ __forceinline__ void st_async_v4(uint32_t addr, uint32_t bar, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%2, %3, %4, %5}, [%1];"
               ::"r"(addr), "r"(bar), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* map, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(map), "r"(x), "r"(y) : "memory");
}

// The steps between the linear value and the output conversion that are compiled in only where asked for.
enum : int { kStepNone = 0, kStepGelu = 1, kStepResidual = 2, kStepRope = 3, kStepGlu = 4 };
enum : int { kOutF32 = 0, kOutBf16 = 1, kOutC4 = 2, kOutC8 = 3 };

// One chunk of kTok tokens of the thread's output channel j: the accumulators at `taddr` plus the partial sums the other
// CTAs of the cluster left (`part`, one block of `part_stride` pieces per CTA), then the epilogue of its first `live` tokens (those inside
// the matrix, at least one).  What an element needs from global memory (residual, rotation table) is requested for the whole chunk
// before any of it is used.  `dry`: what the chunk will need is brought near and nothing else happens.
template <int OUT, int STEP>
__device__ __forceinline__ void finish_chunk(const SkinnyParams& P, const ColumnTerms& ct, uint32_t taddr, const int32_t* asum,
                                             const uint4* part, int parts, int part_stride, int mc, int live, int j, bool col_ok, int lane, bool dry) {
  const EpilogueParams& ep = P.ep;
  float res[kTok];
  float2 cs[kTok];
  if constexpr (STEP == kStepResidual) {
#pragma unroll
    for (int e = 0; e < kTok; ++e) {
      const int64_t off = int64_t(mc + min(e, live - 1)) * ep.ld_residual + (col_ok ? j : 0);
      res[e] = ep.residual_bf16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(ep.residual)[off]) : static_cast<const float*>(ep.residual)[off];
    }
  }
  const bool turn = STEP == kStepRope && col_ok && j < ep.rope_cols;
  if constexpr (STEP == kStepRope) {
    const float2* line = ep.rope + ((j % ep.rope_dim) >> 1);
    int pos = mc % ep.rope_period;
#pragma unroll
    for (int e = 0; e < kTok; ++e) {
      if (turn) cs[e] = __ldg(line + int64_t(pos) * (ep.rope_dim >> 1));
      if (++pos == ep.rope_period) pos = 0;
    }
  }
  uint32_t r[kTok] = {};
  __syncwarp();
  if (!dry) {
    tmem_ld8(taddr, r);
    tmem_ld_wait();
  }
#pragma unroll 1
  for (int s = 0; s < parts; ++s) {
    const uint4 lo = part[s * part_stride], hi = part[s * part_stride + kRowsW];
    r[0] += lo.x; r[1] += lo.y; r[2] += lo.z; r[3] += lo.w;
    r[4] += hi.x; r[5] += hi.y; r[6] += hi.z; r[7] += hi.w;
  }
  if (ep.acc_debug != nullptr && col_ok && !dry) {
#pragma unroll
    for (int e = 0; e < kTok; ++e)
      if (e < live) ep.acc_debug[int64_t(mc + e) * P.N + j] = int32_t(r[e]);
  }
  float v[kTok];
  const int4 as0 = *reinterpret_cast<const int4*>(asum), as1 = *reinterpret_cast<const int4*>(asum + 4);
  const int32_t as[kTok] = {as0.x, as0.y, as0.z, as0.w, as1.x, as1.y, as1.z, as1.w};
#pragma unroll
  for (int e = 0; e < kTok; ++e) {
    const int32_t corr = int32_t(r[e] - uint32_t(ct.z_w) * uint32_t(as[e]) + uint32_t(ct.kzz));
    v[e] = fmaf(ct.scale, float(corr), ct.bias);
    if constexpr (STEP == kStepGelu) v[e] = gelu_erf(v[e]);
    if constexpr (STEP == kStepResidual) {
      if (ep.gelu) v[e] = gelu_erf(v[e]);
      v[e] += res[e];
    }
    if constexpr (STEP == kStepRope) {
      const float other = __shfl_xor_sync(0xffffffffu, v[e], 1);
      if (turn) {
        float a = (j & 1) ? other : v[e], b = (j & 1) ? v[e] : other;
        rope_rotate(cs[e], a, b);
        v[e] = (j & 1) ? b : a;
      }
    }
    if constexpr (STEP == kStepGlu) {                      // even channel: gate, odd: up; the even lane keeps the product
      const float up = __shfl_xor_sync(0xffffffffu, v[e], 1);
      v[e] = silu_mul(v[e], up);
    }
  }
  if (dry) live = 0;
  const bool store = col_ok && !(STEP == kStepGlu && (j & 1));
  const int64_t at0 = int64_t(mc) * ep.ldo + (STEP == kStepGlu || OUT == kOutC4 ? j >> 1 : j);
  if constexpr (OUT == kOutF32 || OUT == kOutBf16) {
    using T = typename std::conditional<OUT == kOutF32, float, __nv_bfloat16>::type;
    T* o = static_cast<T*>(ep.out) + at0;
#pragma unroll
    for (int e = 0; e < kTok; ++e) {
      if (store && e < live) {
        if constexpr (OUT == kOutF32) *o = v[e]; else *o = __float2bfloat16_rn(v[e]);
      }
      o += ep.ldo;
    }
  } else {
    uint8_t* o = static_cast<uint8_t*>(ep.out) + at0;
    int code[kTok];
#pragma unroll
    for (int e = 0; e < kTok; ++e) code[e] = store ? requantize(ct, v[e]) : 0;
#pragma unroll
    for (int e = 0; e < kTok; ++e) {
      if constexpr (OUT == kOutC4) {
        const int next = __shfl_down_sync(0xffffffffu, code[e], 1);
        if (col_ok && !(j & 1) && e < live) *o = uint8_t(code[e] | (next << 4));
      } else {
        if (store && e < live) *o = uint8_t(code[e]);
      }
      o += ep.ldo;
    }
    if (ep.out_row_sum != nullptr) {
      int sums = 0;                                        // lane e: code sum of token mc + e over the warp's channels
#pragma unroll
      for (int e = 0; e < kTok; ++e) {
        const int total = __reduce_add_sync(0xffffffffu, code[e]);
        if (lane == e) sums = total;
      }
      if (lane < live) atomicAdd(ep.out_row_sum + mc + lane, sums);
    }
  }
}

template <int OUT, int STEP>
__global__ void __launch_bounds__(kThreads, 2)
qgemm_skinny_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_a, const __grid_constant__ SkinnyParams P) {
  extern __shared__ __align__(1024) uint8_t ring[];
  __shared__ alignas(8) uint64_t s_full[kMaxStages], s_empty[kMaxStages], s_acc, s_done, s_part;
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ alignas(16) int32_t s_asum[kMaxTokens];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int split = P.split;
  const int rank = int(blockIdx.x) % split;
  const int n0 = int(blockIdx.x) / split * kRowsW, m0 = int(blockIdx.y) * P.mt;
  const int kb0 = rank * P.kblocks / split, kb1 = (rank + 1) * P.kblocks / split;
  const int stages = P.stages;
  // The tile's chunks of kTok tokens are dealt to the cluster's CTAs in contiguous shares; a CTA sends its partial sums of the other
  // shares to their owners, into a part of shared memory of their own: [source][chunk of the share][half of 4 tokens][channel] x 16 B.
  const int chunks = P.mt / kTok, share = (chunks + split - 1) / split;
  const int c_first = rank * share, c_end = min(chunks, c_first + share);
  // (or, where a ring of three stages leaves no room for that, over the ring, once all CTAs have finished with theirs).
  uint8_t* exchange = P.over_ring ? ring : ring + uint32_t(stages) * P.stage_bytes;

  if (warp == kEpiWarps && lane == 0) { tma_prefetch_map(&map_w); tma_prefetch_map(&map_a); }
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(smem_u32(&s_full[s]), 1); mbar_init(smem_u32(&s_empty[s]), 1); }
    mbar_init(smem_u32(&s_acc), 1);
    mbar_init(smem_u32(&s_done), 1);
    mbar_init(smem_u32(&s_part), 1);
    s_abort = 0;
    if (smem_u32(ring) & 1023u) {                          // the swizzled tiles need this alignment
      atomicCAS(P.status, 0, 69);
      s_abort = 1;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (c_end > c_first) mbar_expect_tx(smem_u32(&s_part), uint32_t((split - 1) * (c_end - c_first)) * kChunkBytes);
  }
  if (warp == kEpiWarps + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(P.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if (split > 1 && !P.over_ring) cluster_arrive();         // (this CTA's barriers are set up)
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  volatile int* abort = &s_abort;
  // Ahead of the dependency wait, while the kernel before this one finishes (inside a block, unless that kernel has just expanded
  // them): all of the CTA's weights where the ring holds them (ViT-S block of one image 33.0 -> 32.0 us), else the first
  // k-blocks into L2 (copies into the ring cost a 7B-shaped block of 48 tokens 1 us there).
  const int early = P.weights_settled && kb1 - kb0 <= stages && !*abort ? kb1 - kb0 : 0;
  if (warp == kEpiWarps) {
    if (early == 0 && P.weights_settled && blockIdx.y == 0 && lane < kPrefetch && kb0 + lane < kb1) tma_prefetch_2d(&map_w, (kb0 + lane) * kBK, n0);
    if (lane == 0) {
      for (int s = 0; s < early; ++s) {
        mbar_expect_only(smem_u32(&s_full[s]), kWBytes);   // (the activations of the stage bring the arrival)
        tma_load_2d(smem_u32(ring) + s * P.stage_bytes, &map_w, smem_u32(&s_full[s]), (kb0 + s) * kBK, n0);
      }
    }
  }
  grid_dependency_wait();
  grid_dependency_trigger();

  // the thread's output channel (epilogue warps)
  const EpilogueParams& ep = P.ep;
  const int quarter = warp & 3, half = warp >> 2;
  const int j = n0 + quarter * 32 + lane;
  const bool col_ok = j < P.N;
  ColumnTerms ct{};

  if (warp == kEpiWarps) {
    // ---------------------------------------------------------------- bulk copies (the warp walks the loop, one lane issues)
    const bool issues = elect_one();
    uint32_t stage = 0, phase = 0;
    int issued = 0;
    for (int kb = kb0; kb < kb1; ++kb) {
      const bool free = mbar_wait(smem_u32(&s_empty[stage]), phase ^ 1, abort, 61, P.status);
      if (!__all_sync(0xffffffffu, free)) break;
      const uint32_t bar = smem_u32(&s_full[stage]);
      const uint32_t base = smem_u32(ring) + stage * P.stage_bytes;
      if (issues) {
        mbar_expect_tx(bar, early ? P.a_bytes : kWBytes + P.a_bytes);
        if (early == 0) tma_load_2d(base, &map_w, bar, kb * kBK, n0);
        tma_load_2d(base + kWBytes, &map_a, bar, kb * kBK, m0);
      }
      __syncwarp();
      ++issued;
      if (++stage == uint32_t(stages)) { stage = 0; phase ^= 1; }
    }
    if (lane == 0) {
      // the copies issued last must have landed before the CTA may exit
      for (int i = issued < stages ? issued : stages; i > 0; --i) {
        if (stage == 0) { stage = uint32_t(stages) - 1; phase ^= 1; } else { --stage; }
        mbar_drain(smem_u32(&s_full[stage]), phase);
      }
      // weights asked for early whose activations were given up on
      for (int s = issued; s < early; ++s) mbar_drain_unjoined(smem_u32(&s_full[s]), 0);
    }
  } else if (warp == kEpiWarps + 1) {
    // ---------------------------------------------------------------- MMA issue: D = s32, A = B = unsigned bytes, K-major
    const bool issues = elect_one();
    const uint32_t idesc = (2u << 4) | (uint32_t(P.mt >> 3) << 17) | (uint32_t(kRowsW >> 4) << 24);
    uint32_t stage = 0, phase = 0;
    bool go = true;
    for (int kb = kb0; kb < kb1; ++kb) {
      go = mbar_wait(smem_u32(&s_full[stage]), phase, abort, 62, P.status);
      if (!(go = __all_sync(0xffffffffu, go))) break;
      tc_fence_after();
      const uint32_t base = smem_u32(ring) + stage * P.stage_bytes;
      const uint64_t dw = smem_desc_sw128(base), da = smem_desc_sw128(base + kWBytes);
      if (issues) {
#pragma unroll
        for (int k = 0; k < kBK / 32; ++k) umma_i8(tmem, dw + uint64_t(2 * k), da + uint64_t(2 * k), idesc, (kb != kb0 || k != 0) ? 1u : 0u);
        umma_commit(smem_u32(&s_empty[stage]));
      }
      __syncwarp();
      if (++stage == uint32_t(stages)) { stage = 0; phase ^= 1; }
    }
    if (issues) {
      if (go) umma_commit(smem_u32(&s_acc));
      umma_commit(smem_u32(&s_done));                      // all MMAs have completed before tensor memory is freed
    }
    __syncwarp();
    mbar_drain(smem_u32(&s_done), 0);
  } else {
    // ---------------------------------------------------------------- epilogue
    // the tile's token sums and the channel's terms, behind the main loop
    for (int i = threadIdx.x; i < P.mt; i += 32 * kEpiWarps) s_asum[i] = m0 + i < P.M ? __ldg(P.asum + m0 + i) : 0;
    if (col_ok) ct = column_terms(ep, j, __ldg(P.wsum + j));
    if (ep.glu) { const ColumnTerms q = column_terms(ep, 0, 0); ct.inv_so = q.inv_so; ct.zo_lo = q.zo_lo; ct.zo_hi = q.zo_hi; ct.zo = q.zo; }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory");
    const uint32_t tquarter = tmem + (uint32_t(quarter * 32) << 16);
    const int row = quarter * 32 + lane;
    // The first round runs dry, while the main loop waits for its operands: its code, and the residual and rotation values of the first
    // chunk, are then near (48 tokens x 12288 x 4096 with rotation: last MMA to end of the kernel 3.1 -> 1.1 us).  Short main loops have
    // no time for it, and start with the second.  Codes two per byte do without the code for it: products of a block have no such output,
    // and by themselves they lose 4 to 11 % by it (2000 x 1000 x 512 6.0 and 6.4 us, 1000 x 1000 x 1024 with GELU 6.5 and 6.9).
    constexpr bool kDry = OUT != kOutC4;
#pragma unroll 1
    for (int round = kDry && P.dry ? 0 : 1; round < 2; ++round) {
      if (round != 0) {
        bool ok = mbar_wait(smem_u32(&s_acc), 0, abort, 63, P.status);
        tc_fence_after();
        if (split > 1) {
          __syncwarp();
          if (P.over_ring) cluster_arrive();               // (this CTA's main loop is through)
          cluster_wait();                                  // (and so far are the others)
#pragma unroll 1
          for (int c = half; c < chunks; c += kEpiWarps / 4) {
            const int owner = c / share;
            if (owner == rank) continue;
            uint32_t r[kTok];
            __syncwarp();
            tmem_ld8(tquarter + uint32_t(c * kTok), r);
            tmem_ld_wait();
            const int src = rank - (rank > owner ? 1 : 0);     // 0 .. split - 2
            const uint32_t at = smem_u32(exchange) + uint32_t((src * (min(chunks, (owner + 1) * share) - owner * share) + (c - owner * share)) * 2 * kRowsW + row) * 16u;
            const uint32_t to = map_to_rank(at, uint32_t(owner)), bar = map_to_rank(smem_u32(&s_part), uint32_t(owner));
            st_async_v4(to, bar, r[0], r[1], r[2], r[3]);
            st_async_v4(to + kRowsW * 16u, bar, r[4], r[5], r[6], r[7]);
          }
          if (c_end > c_first && !mbar_wait(smem_u32(&s_part), 0, abort, 64, P.status)) {
            // given up, here or by a role that raised the flag: the sums still come (every CTA sends), and have to land before this one leaves
            mbar_drain(smem_u32(&s_part), 0);
            ok = false;
          }
          __syncwarp();
          cluster_arrive();                                // (nothing more comes to this CTA, and it sends nothing more)
        }
        if (!__all_sync(0xffffffffu, ok && !*abort)) break;      // (all lanes leave together)
      }
      for (int c = c_first + half; c < c_end; c += kEpiWarps / 4) {
        const int mc = m0 + c * kTok;
        if (mc >= P.M) break;
        const uint4* part = reinterpret_cast<const uint4*>(exchange) + (c - c_first) * 2 * kRowsW + row;
        finish_chunk<OUT, STEP>(P, ct, tquarter + uint32_t(c * kTok), s_asum + c * kTok, part, round != 0 ? split - 1 : 0,
                                (c_end - c_first) * 2 * kRowsW, mc, min(kTok, P.M - mc), j, col_ok, lane, kDry && round == 0);
        if (round == 0) break;
      }
    }
  }
  __syncwarp();
  if (split > 1) {
    // no CTA leaves before the sums sent to it have arrived, whether or not a wait ran out
    if (warp >= kEpiWarps) {
      if (P.over_ring) cluster_arrive();
      cluster_wait();
      cluster_arrive();
    }
    cluster_wait();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kEpiWarps + 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(P.tmem_cols) : "memory");
  }
}

repq_status make_map(CUtensorMap* map, const uint8_t* base, int64_t rows, int64_t k, int64_t ld, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  REPQ_REQUIRE(fn != nullptr, REPQ_CUDA_ERROR, "qgemm: cuTensorMapEncodeTiled is not available");
  const cuuint64_t dims[2] = {cuuint64_t(k), cuuint64_t(rows)};
  const cuuint64_t strides[1] = {cuuint64_t(ld)};
  const cuuint32_t box[2] = {kBK, cuuint32_t(box_rows)};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  REPQ_REQUIRE(r == CUDA_SUCCESS, REPQ_CUDA_ERROR, "qgemm: cuTensorMapEncodeTiled failed with code %d", int(r));
  return REPQ_OK;
}

template <int OUT, int STEP>
repq_status launch(dim3 grid, uint32_t smem, const CUtensorMap& map_w, const CUtensorMap& map_a, const SkinnyParams& P, cudaStream_t st) {
  REPQ_TRY((allow_smem<qgemm_skinny_kernel<OUT, STEP>>(kSmemOne)));
  REPQ_CUDA(launch_chained_cluster(qgemm_skinny_kernel<OUT, STEP>, grid, dim3(kThreads), smem, st, P.split, map_w, map_a, P));
  note_launch();
  return REPQ_OK;
}

template <int OUT>
repq_status launch_step(int step, dim3 grid, uint32_t smem, const CUtensorMap& map_w, const CUtensorMap& map_a, const SkinnyParams& P, cudaStream_t st) {
  switch (step) {
    case kStepGelu: return launch<OUT, kStepGelu>(grid, smem, map_w, map_a, P, st);
    case kStepResidual: return launch<OUT, kStepResidual>(grid, smem, map_w, map_a, P, st);
    case kStepRope: return launch<OUT, kStepRope>(grid, smem, map_w, map_a, P, st);
    case kStepGlu:
      if constexpr (OUT != kOutC4) return launch<OUT, kStepGlu>(grid, smem, map_w, map_a, P, st);   // (packed codes are refused)
    default: return launch<OUT, kStepNone>(grid, smem, map_w, map_a, P, st);
  }
}

}  // namespace

// Tokens per tile and CTAs per tile by the least estimated time, in microseconds:
//   a launch                1.9
//   operands                k-blocks of a CTA x 0.295 (a ring's latency over its stages) or, with two CTAs on an SM, x (16 KB of
//                           weights + tokens) at 160 KB per us and SM; or all weights at 4.6 TB/s, whichever is longer
//   epilogue                0.024 per token of a CTA's share, 0.039 with GELU or a step on column pairs, 0.046 with a residual
//   exchange in a cluster   1.15 and 0.031 per token that leaves the CTA (fitted to the exchange behind two barriers of the cluster)
//   two CTAs on an SM       0.5, and 1.53 x the epilogue and the exchange
// Clusters fill the SMs less evenly: those of four and eight share SMs from 0.91 and 0.75 CTAs per SM on, and beyond 1.8 and 1.62
// per SM (two without a cluster) the last ones wait for a second wave, which costs more than it brings.
// The best plan's time is within 0.6 % of the fastest form's on average (4.8 % with the terms used before, which had no cost per
// token exchanged: 48 x 4096 x 4096 with residual 11.7 -> 7.9 us, 197 x 768 x 3072 11.2 -> 6.7).
SkinnyPlan qgemm_skinny_plan(const repq_gemm_desc& d) {
  SkinnyPlan best;
  if (d.batch_outer != 1 || d.batch_inner != 1 || d.N < 64 || d.K < 64) return best;
  if (!d.a_row_sum || !d.w_row_sum) return best;           // (the sums are not taken here; no workspace)
  if (packed4(d.bits_a) || packed4(d.bits_w) || packed6(d.bits_w)) return best;
  if (!(aligned(d.a_codes, 16) && d.lda_bytes % 16 == 0 && aligned(d.w_codes, 16) && d.ldw_bytes % 16 == 0)) return best;
  const int sms = sm_count();
  const int n_tiles = (d.N + kRowsW - 1) / kRowsW, kblocks = (d.K + kBK - 1) / kBK;
  const float hbm = float(d.N) * float(d.K) / 4.6e6f;
  const float per_token = d.residual ? 0.0461f : d.gelu || d.glu || d.rope_cos_sin ? 0.0386f : 0.0243f;
  for (int mt : {16, 32, 48, 64, 96, 128}) {
    const int64_t m_tiles = (int64_t(d.M) + mt - 1) / mt;
    for (int split = 1; split <= 8; split *= 2) {
      const float ctas = float(n_tiles) * float(m_tiles) * float(split);
      const float single = float(sms) * (split == 8 ? 0.75f : split == 4 ? 0.91f : 1.f);
      const float most = float(sms) * (split == 8 ? 1.62f : split == 4 ? 1.8f : 2.f);
      if (ctas > most || (split > 1 && kblocks < 2 * split)) continue;
      const bool two = ctas > single;
      const float kb = float((kblocks + split - 1) / split), share = float((mt / kTok + split - 1) / split * kTok);
      const float wide = (two ? 2.f : 1.f) * (16.f + float(mt) / 8.f) / 160.f;
      float load = kb * (wide > 0.295f ? wide : 0.295f);
      if (load < hbm) load = hbm;
      float us = 1.9f + load + (two ? 0.49f : 0.f) + (two ? 1.53f : 1.f) * share * per_token;
      if (split > 1) us += 1.15f + (two ? 1.53f : 1.f) * 0.0314f * float(mt) * (1.f - 1.f / float(split));
      if (best.mt == 0 || us < best.us) { best.mt = mt; best.split = split; best.two = two; best.us = us; }
    }
    if (mt >= d.M) break;
  }
  return best;
}

repq_status qgemm_skinny(const repq_gemm_desc& d, const EpilogueParams& ep, const SkinnyPlan& plan, Params params, cudaStream_t st) {
  SkinnyParams P{};
  P.M = d.M; P.N = d.N; P.K = d.K;
  P.asum = d.a_row_sum; P.wsum = d.w_row_sum;
  P.ep = ep;
  P.weights_settled = params == Params::settled;
  P.status = device_status_word();
  REPQ_REQUIRE(P.status != nullptr, REPQ_CUDA_ERROR, "qgemm: device status word unavailable");
  const int n_tiles = (d.N + kRowsW - 1) / kRowsW, mt = plan.mt, split = plan.split;
  const int m_tiles = (d.M + mt - 1) / mt;
  P.kblocks = (d.K + kBK - 1) / kBK;
  P.mt = mt;
  P.split = split;
  P.a_bytes = uint32_t(mt) * kBK;
  P.stage_bytes = kWBytes + P.a_bytes;
  const int per = (P.kblocks + split - 1) / split;         // k-blocks of a CTA
  // behind the ring: the partial sums that the other CTAs of the cluster send
  const uint32_t exchange = uint32_t(split - 1) * uint32_t((mt / kTok + split - 1) / split) * kChunkBytes;
  auto ring_of = [&](uint32_t bytes) {
    const int n = int(bytes / P.stage_bytes), useful = per < kMaxStages ? per : kMaxStages;
    return n < useful ? n : useful;
  };
  // (by the plan's limits: fewer CTAs than SMs do not all fit one per SM in clusters, and with 200 KB each the rest wait for a second wave,
  // 16 x 2048 x 8192, 128 CTAs in clusters of eight, 12.2 us; with 110 KB 7.4)
  const uint32_t most = plan.two ? kSmemTwo : kSmemOne;
  int stages = ring_of(most - exchange);
  P.over_ring = stages < 3 && stages < per;
  if (P.over_ring) stages = ring_of(most);                 // (at least three, or all k-blocks)
  P.stages = stages;
  // Where the dry round pays: never, always, this line; 197 x 1536 x 384 with GELU 3.84, 4.08, 3.92 us, 64 x 1024 x 128 with residual 2.99, 3.68,
  // 2.91, 48 x 4096 x 4096 with residual 8.43, 8.20, 8.08, 197 x 2304 x 768 with residual 6.48, 6.22, 6.02; block passes of 197 x 384 27.5, 28.4,
  // 27.7, of 16 tokens x 4096 60.3, 59.8, 59.7.
  P.dry = per >= (d.residual ? 6 : 8);
  uint32_t smem = uint32_t(stages) * P.stage_bytes;
  if (!P.over_ring) smem += exchange;
  else if (smem < exchange) smem = exchange;
  P.tmem_cols = 32;
  while (P.tmem_cols < uint32_t(mt)) P.tmem_cols *= 2;
  CUtensorMap map_w, map_a;
  REPQ_TRY(make_map(&map_w, d.w_codes, d.N, d.K, d.ldw_bytes, kRowsW));
  REPQ_TRY(make_map(&map_a, d.a_codes, d.M, d.K, d.lda_bytes, mt));
  const int out = ep.out_kind == REPQ_OUT_F32 ? kOutF32 : ep.out_kind == REPQ_OUT_BF16 ? kOutBf16 : ep.pack4 ? kOutC4 : kOutC8;
  const int step = ep.rope ? kStepRope : ep.glu ? kStepGlu : ep.residual ? kStepResidual : ep.gelu ? kStepGelu : kStepNone;
  const dim3 grid(unsigned(n_tiles * split), unsigned(m_tiles));
  switch (out) {
    case kOutF32: return launch_step<kOutF32>(step, grid, smem, map_w, map_a, P, st);
    case kOutBf16: return launch_step<kOutBf16>(step, grid, smem, map_w, map_a, P, st);
    case kOutC4: return launch_step<kOutC4>(step, grid, smem, map_w, map_a, P, st);
    default: return launch_step<kOutC8>(step, grid, smem, map_w, map_a, P, st);
  }
}

}  // namespace repq
