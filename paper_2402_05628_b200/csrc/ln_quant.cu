// Fused LayerNorm + layer-wise uniform quantization (Eq. 9 with the reparameterized affine factors of
// Eq. 12, then Eq. 4 with the scalar (s~, z~)).
//
// Every input element is read once with 128-bit loads and leaves as a 4-bit (or 8-bit) code.  A row is owned by a group
// of TPR threads which keeps its slice of the row in registers, so mean and centred variance are two register passes with
// shuffle reductions.  Each group works on one or two rows at a time, and the rows of its next iteration are requested before
// the current ones are reduced, so that loads stay in flight all the time.  Rows of several warps meet at one barrier: every
// warp centres its slice on the slice's own mean, the means and squares are merged behind the barrier, and the code sums wait
// for the next one.
//
// What bounds it: HBM for float input and for rows of one warp (5.1-6.3 TB/s of 6.46); for longer bf16 rows instructions and the latencies
// of a row's chain at the 16 warps per SM that the registers leave (ncu, 32768 x 4096: 10.9 instructions per element, DRAM 43 % of its peak,
// issue slots 56 %).  Calls of many rows of 2048 or 4096 elements take ln_rows_kernel below.
// Measured against three barriers per iteration: 65536 bf16 rows of 1536 53 -> 45 us, 32768 float rows of 2048 83 -> 48, 16384 of
// 4096 76 -> 49; 32768 bf16 rows of 4096 gained nothing (80).
// The per-channel factors gamma~/s~ and beta~/s~ are staged once per CTA in shared memory (halves of the 8-element
// chunks apart, so that a warp's 16-byte reads are free of bank conflicts).
//
// The float work runs on packed pairs (two elements per add / mul / fma issue slot).  Rounding is done by the
// float adder: t + 1.5 * 2^23 leaves rint(t) (half to even, on t itself, as Eq. 4 has it) in the low mantissa
// bits while |t| < 2^22; inputs that cannot guarantee that bound are clamped and converted with cvt.rni
// instead.  z is added as an integer and the clip of Eq. 4 is the saturation of the packing instruction.  (t times 2^-149, a denormal whose
// bits are rint(t), plus z as another denormal saves two integer additions per pair, but the compiler makes one fused operation of the packed
// product and the packed sum, although both ask for their own rounding: t + z is then rounded, and a tie falls the other way for odd z.)
#include <cuda_bf16.h>

#include <type_traits>

#include "f32x2.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace repq {
namespace {

constexpr int kChunk = 8;   // elements per 128-bit bf16 load
constexpr int kMagicBits = 0x4B400000;   // float 1.5 * 2^23

// Rows a thread group works on at a time (the loads of the next ones are always in flight as well): two, except where the
// chunks per thread leave the registers for one.  bf16: from four chunks on in groups that share an SM with others (2048 / 4096
// elements, 64 x 4 / 128 x 4 threads x chunks, 69 / 73 us in short runs with one row, 97 / 101 with two); groups of 256 and 512 threads have no
// more than two blocks on an SM either way and hide a row's latencies behind the second (268 MB of rows, one -> two: 6152
// elements 122 -> 116 us, 8192 93 -> 85, 12296 130 -> 118, 16384 103 -> 95).  float: from three chunks on (768, 32 x 3, 21 and 28),
// from four in groups of 512 (8200, 512 x 3, 88 with one, 83 with two; 12296, 512 x 4, 78 and 107).
__host__ __device__ constexpr int rows_in_flight(int vpt, int tpr, int elem_bytes) {
  if (elem_bytes == 2) return vpt < 4 || tpr >= 256 ? 2 : 1;
  return vpt < (tpr >= 512 ? 4 : 3) ? 2 : 1;
}

// Blocks per SM that the register budget is cut for (0: left to the compiler): two where the compiler would take a few registers
// too many for the second.  float rows of one warp or less: up to five chunks per thread (268 MB of rows, without -> with: 512
// elements 85 -> 65 us, 1024 83 -> 63, 1280 78 -> 66); six (1536 elements) would spill, 69 -> 77.
constexpr int min_blocks(int vpt, int tpr, int elem_bytes) { return tpr == 256 || (elem_bytes == 4 && tpr <= 32 && vpt <= 5) ? 2 : 0; }

// A chunk of 8 elements as it is loaded (kept in this form while the rows before it are processed), and
// its expansion into 4 packed float pairs.
template <typename T> struct RawChunk;
template <> struct RawChunk<float> { float4 a, b; };
template <> struct RawChunk<__nv_bfloat16> { uint4 a; };

__device__ __forceinline__ void load_raw(const float* p, bool on, RawChunk<float>& r) {
  r.a = r.b = make_float4(0.f, 0.f, 0.f, 0.f);
  if (on) {
    r.a = __ldcs(reinterpret_cast<const float4*>(p));
    r.b = __ldcs(reinterpret_cast<const float4*>(p) + 1);
  }
}
__device__ __forceinline__ void load_raw(const __nv_bfloat16* p, bool on, RawChunk<__nv_bfloat16>& r) {
  r.a = make_uint4(0u, 0u, 0u, 0u);
  if (on) r.a = __ldcs(reinterpret_cast<const uint4*>(p));
}
__device__ __forceinline__ void expand(const RawChunk<float>& r, f32x2 (&v)[kChunk / 2]) {
  v[0] = pack2(r.a.x, r.a.y); v[1] = pack2(r.a.z, r.a.w); v[2] = pack2(r.b.x, r.b.y); v[3] = pack2(r.b.z, r.b.w);
}
__device__ __forceinline__ void expand(const RawChunk<__nv_bfloat16>& r, f32x2 (&v)[kChunk / 2]) {
  const uint32_t w[4] = {r.a.x, r.a.y, r.a.z, r.a.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = pack2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
}

// Reductions inside a warp are xor shuffles (integers of a whole warp take the warp-wide reduction instruction).
// Barrier of one thread group: the whole block where a group is the block, else a named barrier of the group's own (the
// groups of a block then no longer wait for one another).
template <int TPR>
__device__ __forceinline__ void group_sync(int group_first_warp) {
  if constexpr (TPR >= 256) __syncthreads();
  else asm volatile("bar.sync %0, %1;" ::"r"(1 + group_first_warp / (TPR / 32)), "n"(TPR) : "memory");
}

template <int TPR, int kRows>
__device__ __forceinline__ void warp_reduce(float (&v)[kRows]) {
  const bool odd = threadIdx.x & 1;
  if constexpr (kRows == 2 && TPR >= 4) {
    // neighbouring lanes split the two rows between them (one shuffle for both rows), every further step then moves one
    // value per lane, and a last exchange hands each lane the other row's total: log(TPR) + 1 shuffles instead of
    // twice the log.  All lanes of a parity add the same pairs at every step, so they end with the same bits.
    float t = (odd ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, odd ? v[0] : v[1], 1);
#pragma unroll
    for (int o = TPR / 2; o > 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    const float u = __shfl_xor_sync(0xffffffffu, t, 1);
    v[0] = odd ? u : t;
    v[1] = odd ? t : u;
  } else {
#pragma unroll
    for (int o = TPR / 2; o > 0; o >>= 1)
#pragma unroll
      for (int r = 0; r < kRows; ++r) v[r] += __shfl_xor_sync(0xffffffffu, v[r], o);
  }
}
template <int TPR, int kRows>
__device__ __forceinline__ void group_sum(int (&v)[kRows]) {
  if constexpr (TPR == 32) {
#pragma unroll
    for (int r = 0; r < kRows; ++r) v[r] = __reduce_add_sync(0xffffffffu, v[r]);
  } else {
#pragma unroll
    for (int o = TPR / 2; o > 0; o >>= 1)
#pragma unroll
      for (int r = 0; r < kRows; ++r) v[r] += __shfl_xor_sync(0xffffffffu, v[r], o);
  }
}

template <typename T, int TPR, int kVPT, bool kPack4, bool kFull>
__global__ void __launch_bounds__((TPR > 256 ? TPR : 256), min_blocks(kVPT, TPR, sizeof(T)))
ln_quant_kernel(const T* __restrict__ x, int64_t rows, int D, int64_t ldx,
                const float* __restrict__ gamma_t, const float* __restrict__ beta_t, float eps, int rms,
                float inv_s, int z, int qmax, uint8_t* __restrict__ codes, int64_t ldc,
                int32_t* __restrict__ row_sum, int32_t* __restrict__ clear, int64_t n_clear, Params params) {
  const bool settled = params == Params::settled, beside = params == Params::beside;
  constexpr int kRows = rows_in_flight(kVPT, TPR, sizeof(T));
  constexpr int kBlock = TPR > 256 ? TPR : 256;
  constexpr int kGroups = kBlock / TPR;
  constexpr int kRowsPerBlock = kGroups * kRows;
  extern __shared__ __align__(16) float s_gb[];          // g[D] then b[D]: gamma~/s~ and beta~/s~
  // Rows of several warps: one barrier per iteration.  A warp reduces its own slice twice (sum, then squares centred on the
  // slice's own mean) and leaves both in `red`; behind the barrier every warp merges the slices' means and squares
  // (M2 = sum M2_w + n_w (mean_w - mean)^2).  Code sums wait in `red_c` for the next iteration's barrier.  Both alternate by
  // iteration parity: a slot written in iteration k is read before the barrier of k + 1 (`red`) or of k + 2 (`red_c`), and
  // written again in k + 2, behind the barrier of k + 1 or, for `red_c`, behind that of k + 2.
  constexpr bool kWide = TPR > 32;
  constexpr int kWarps = kWide ? TPR / 32 : 1;             // warps of a row
  __shared__ float2 red[kWide ? 2 : 1][kBlock / 32 * kRows];
  __shared__ int red_c[kWide ? 2 : 1][kBlock / 32 * kRows];

  const int tig = threadIdx.x % TPR;             // thread in group
  const int group = threadIdx.x / TPR;
  const int group_first_warp = (group * TPR) >> 5;
  const int nchunks = D / kChunk;

  // The rows of the next iteration are requested while those of the current one are processed, so that loads
  // stay in flight through the reductions and the packing.
  RawChunk<T> raw[kRows][kVPT];
  auto fetch = [&](int64_t first_row) {
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      // rows past the end re-read the last row (their codes are never stored); when the row fills the group
      // exactly (kFull) no load is predicated
      const int64_t row = first_row + r < rows ? first_row + r : rows - 1;
      const T* xr = x + row * ldx;
#pragma unroll
      for (int i = 0; i < kVPT; ++i) {
        const int c = tig + i * TPR;
        load_raw(xr + c * kChunk, kFull || c < nchunks, raw[r][i]);
      }
    }
  };
  // Factors that the kernel ahead in the stream may have written are read behind the wait, together with the first rows; settled
  // ones while that kernel finishes.  (Loads past L1: what that kernel wrote must not meet an older line.)  The next kernel's start
  // is allowed as soon as everything ahead has completed, so that its prologue runs beside the staging.
  // Pieces of 4 factors, all of a thread's in flight at once; a block starts at a piece of its own, since all blocks read the same
  // 8 D bytes at the same moment and would queue for the same lines of L2.
  // What reading behind the wait costs, back to back against a settled start: 0.3-1.3 us per launch up to 4096 elements (32768 x 4096
  // 76.0 -> 76.4, 4239 x 4096 11.8 -> 12.9), 2-3 at 8192 (9950 rows 47.5 -> 50.4); in a block pass 0.2-1.3 (one ViT-S image 31.9 -> 32.1,
  // 64 DeiT-B images 208.6 -> 209.9).  With factors one by one behind the first rows 1-3.
  constexpr int kPieces = (TPR * kVPT * kChunk / 4 + kBlock - 1) / kBlock;
  const int n4 = D / 4, rot = int(blockIdx.x * 32u % uint32_t(n4));
  const bool vec = ((reinterpret_cast<uintptr_t>(gamma_t) | reinterpret_cast<uintptr_t>(beta_t)) & 15) == 0;
  auto load4 = [&](const float* p) {
    return vec ? __ldcg(reinterpret_cast<const float4*>(p)) : make_float4(__ldcg(p), __ldcg(p + 1), __ldcg(p + 2), __ldcg(p + 3));
  };
  auto piece = [&](int k) {
    const int q = k * kBlock + int(threadIdx.x) + rot;
    return q < n4 ? q : q - n4;
  };
  if (!settled) {
    if (!beside) grid_dependency_wait();
    grid_dependency_trigger();
  }
  float4 g4[kPieces], b4[kPieces];
#pragma unroll
  for (int k = 0; k < kPieces; ++k) {
    g4[k] = b4[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k * kBlock + int(threadIdx.x) < n4) {
      g4[k] = load4(gamma_t + 4 * piece(k));
      b4[k] = load4(beta_t + 4 * piece(k));
    }
  }
  const int64_t first_rows = int64_t(blockIdx.x) * kRowsPerBlock + group * kRows;
  const int64_t stride = int64_t(gridDim.x) * kRowsPerBlock;
  // Float rows of one warp without gaps between them: a block's rows of the iteration after the next one are brought into L2 by one
  // bulk request (inputs new from pass to pass, 400 MB of them: 80000 x 768 53.5 -> 48.4 us, 131072 x 384 45.4 -> 40.0, 80000 x 1024 68.7 ->
  // 64.6, 262144 x 64 19.6 -> 15.8; rows of several warps gained nothing, 30000 x 2048 48.1 -> 50.4, and bf16 rows, which wait for
  // instructions, lost 6 to 12 %).  Fewer rows ask for nothing; 20000 and 40000 rows of 64 elements take 0.3 to 0.4 us longer than without this
  // code, of 128 and more 6 to 20 % less (other registers, another number of blocks).
  constexpr bool kToL2 = sizeof(T) == 4 && TPR <= 32;
  const bool deep = kToL2 && ldx == D && rows > 3 * stride;
  auto to_l2 = [&](int64_t first) {
    if (deep && threadIdx.x == 0 && first < rows)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(x + first * ldx), "r"(uint32_t(min(int64_t(kRowsPerBlock), rows - first)) * uint32_t(D) * uint32_t(sizeof(T))) : "memory");
  };
  auto begin = [&] {
    fetch(first_rows);
    if constexpr (kToL2) to_l2(int64_t(blockIdx.x) * kRowsPerBlock + stride);
  };
  if (!settled) begin();

  float* s_g = s_gb;
  float* s_b = s_gb + D;
  // |t| <= sqrt(D) |gamma~/s~| + |beta~/s~|.  Where that bound may reach 2^22, t is clamped and converted instead, which gives a NaN the
  // lowest code (a whole-kernel decision, taken here once).
  const float root_d = sqrtf(float(D));
  bool wide = false;
  // layout: the first halves (4 floats) of all chunks, then the second halves, so that the 16-byte reads of
  // neighbouring lanes are neighbours in shared memory (chunk by chunk they would sit 32 bytes apart: two-way
  // bank conflicts)
#pragma unroll
  for (int k = 0; k < kPieces; ++k) {
    if (k * kBlock + int(threadIdx.x) < n4) {
      const int q = piece(k), at = (q & 1) * (D / 2) + (q >> 1) * 4;
      const float gi[4] = {g4[k].x * inv_s, g4[k].y * inv_s, g4[k].z * inv_s, g4[k].w * inv_s};
      const float bi[4] = {b4[k].x * inv_s, b4[k].y * inv_s, b4[k].z * inv_s, b4[k].w * inv_s};
      *reinterpret_cast<float4*>(s_g + at) = make_float4(gi[0], gi[1], gi[2], gi[3]);
      *reinterpret_cast<float4*>(s_b + at) = make_float4(bi[0], bi[1], bi[2], bi[3]);
#pragma unroll
      for (int e = 0; e < 4; ++e) wide = wide || !(fabsf(gi[e]) * root_d + fabsf(bi[e]) < 4.0e6f);
    }
  }
  const bool guard = __syncthreads_or(wide) != 0;
  // The branch to the second form is taken once per row, around the chunks (per chunk and per row: bf16, 16384 x 8192 74.6 and 72.5 us,
  // 10000 x 6152 52.9 and 46.7, 12608 x 768 8.6 and 8.4, 131072 x 1024 66.1 and 65.2, but 18464 x 1024 13.1 and 13.6); float rows of one
  // warp take it per chunk (12608 x 384 7.1 and 7.2, 30000 x 1536 36.0 and 36.8).
  constexpr bool kPerRow = kWide || sizeof(T) == 2;
  // x and the outputs belong to the chain of kernels
  if (settled) {
    grid_dependency_wait();
    grid_dependency_trigger();
    begin();
  }
  for (int64_t i = int64_t(blockIdx.x) * kBlock + threadIdx.x; i < n_clear; i += int64_t(gridDim.x) * kBlock) clear[i] = 0;

  const float inv_d = 1.f / float(D);
  const uint32_t qmax4 = uint32_t(qmax) * 0x01010101u;
  const f32x2 magic2 = splat2(__int_as_float(kMagicBits));
  const int z_less_magic = z - kMagicBits;

  // the warp's slice of a row, and the slice its lane merges
  const int lane_w = threadIdx.x & 31;
  const int slice_of_lane = (lane_w / kRows) & (kWarps - 1);
  constexpr bool kConst = kFull && sizeof(T) == 2;         // (float rows: known sizes cost registers instead, 146 against 108)
  auto slice_size = [&](int w) {                           // elements of a row that warp w of its group holds
    if constexpr (kConst) return float(32 * kVPT * kChunk);
    int n = 0;
#pragma unroll
    for (int i = 0; i < kVPT; ++i) n += max(0, min(32, nchunks - (w * 32 + i * TPR)));
    return float(n * kChunk);
  };
  auto inverse = [](float n) { return kConst ? 1.f / float(32 * kVPT * kChunk) : n > 0.f ? 1.f / n : 0.f; };
  const float n_slice_of_lane = kWide ? slice_size(slice_of_lane) : 0.f, inv_slice_of_lane = inverse(n_slice_of_lane);
  const float inv_slice = kWide ? inverse(slice_size((threadIdx.x >> 5) - group_first_warp)) : 0.f;
  bool parity_seen = false;
  int64_t last_row0 = 0;
  int parity = 0;
  for (int64_t base = int64_t(blockIdx.x) * kRowsPerBlock; base < rows; base += stride, parity ^= 1) {
    const int64_t row0 = base + group * kRows;

    f32x2 v[kRows][kVPT][kChunk / 2];
    float sum[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r)
#pragma unroll
      for (int i = 0; i < kVPT; ++i) expand(raw[r][i], v[r][i]);
    fetch(row0 + stride);
    if constexpr (kToL2) to_l2(base + 2 * stride);
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      f32x2 acc = 0ull;
#pragma unroll
      for (int i = 0; i < kVPT; ++i)
#pragma unroll
        for (int e = 0; e < kChunk / 2; ++e) acc = add2(acc, v[r][i][e]);
      float lo, hi;
      unpack2(acc, lo, hi);
      sum[r] = lo + hi;
    }

    float mu[kRows], var[kRows];
    if constexpr (!kWide) {
      if (!rms) {
        warp_reduce<TPR, kRows>(sum);
#pragma unroll
        for (int r = 0; r < kRows; ++r) mu[r] = sum[r] * inv_d;
      } else {
#pragma unroll
        for (int r = 0; r < kRows; ++r) mu[r] = 0.f;
      }
    } else {
      if (!rms) warp_reduce<32, kRows>(sum);
#pragma unroll
      for (int r = 0; r < kRows; ++r) mu[r] = rms ? 0.f : sum[r] * inv_slice;       // mean of the warp's slice
    }

    float ss[kRows], slice_mean[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      slice_mean[r] = mu[r];
      const f32x2 neg_mu = splat2(-mu[r]);
      f32x2 acc = 0ull;
#pragma unroll
      for (int i = 0; i < kVPT; ++i) {
        if (kFull || tig + i * TPR < nchunks) {
#pragma unroll
          for (int e = 0; e < kChunk / 2; ++e) {
            v[r][i][e] = add2(v[r][i][e], neg_mu);
            acc = fma2(v[r][i][e], v[r][i][e], acc);
          }
        }
      }
      float lo, hi;
      unpack2(acc, lo, hi);
      ss[r] = lo + hi;
    }
    if constexpr (!kWide) {
      warp_reduce<TPR, kRows>(ss);
#pragma unroll
      for (int r = 0; r < kRows; ++r) var[r] = ss[r] * inv_d;
    } else {
      warp_reduce<32, kRows>(ss);
      const int lane = threadIdx.x & 31;
      if (lane < kRows) red[parity][(threadIdx.x >> 5) * kRows + lane] = make_float2(lane ? sum[kRows - 1] : sum[0], lane ? ss[kRows - 1] : ss[0]);
      group_sync<TPR>(group_first_warp);
      // the code sums of the iteration before
      if (row_sum != nullptr && parity_seen && tig < kRows) {
        int t = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) t += red_c[parity ^ 1][(group_first_warp + w) * kRows + tig];
        const int64_t row = row0 - stride + tig;
        if (row < rows) row_sum[row] = t;
      }
      parity_seen = true;
      // lane l merges slice (l / kRows mod kWarps) of row (l mod kRows): xor steps over the slice index
      const float2 p = red[parity][(group_first_warp + slice_of_lane) * kRows + (lane & (kRows - 1))];
      float total = p.x;
#pragma unroll
      for (int o = kWarps * kRows / 2; o >= kRows; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
      const float mean = rms ? 0.f : total * inv_d;
      const float off = rms ? 0.f : p.x * inv_slice_of_lane - mean;
      float m2 = fmaf(n_slice_of_lane * off, off, p.y);
#pragma unroll
      for (int o = kWarps * kRows / 2; o >= kRows; o >>= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, o);
      if constexpr (kRows == 2) {
        const float mean1 = __shfl_xor_sync(0xffffffffu, mean, 1), m21 = __shfl_xor_sync(0xffffffffu, m2, 1);
        const bool odd = lane & 1;
        mu[0] = odd ? mean1 : mean;
        mu[1] = odd ? mean : mean1;
        var[0] = (odd ? m21 : m2) * inv_d;
        var[1] = (odd ? m2 : m21) * inv_d;
      } else {
        mu[0] = mean;
        var[0] = m2 * inv_d;
      }
    }
    // rows of several warps: v is centred on the slice's mean, the rest of the way to the row's mean is one more product
    f32x2 rstd[kRows], rest[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const float rs = rsqrtf(var[r] + eps);
      rstd[r] = splat2(rs);
      if constexpr (kWide) rest[r] = splat2((slice_mean[r] - mu[r]) * rs);
    }
    auto normalised = [&](f32x2 x, int r) {
      if constexpr (kWide) return fma2(x, rstd[r], rest[r]);
      else return mul2(x, rstd[r]);
    };

    int csum[kRows];
    bool live[kRows];
    uint8_t* out[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      csum[r] = 0;
      live[r] = row0 + r < rows;
      out[r] = codes + (row0 + r) * ldc;
    }
    auto chunks = [&](auto guarded) {
#pragma unroll
    for (int i = 0; i < kVPT; ++i) {
      const int c = tig + i * TPR;
      if (kFull || c < nchunks) {
        f32x2 g[kChunk / 2], b[kChunk / 2];
        const float4 g0 = *reinterpret_cast<const float4*>(s_g + c * 4);
        const float4 g1 = *reinterpret_cast<const float4*>(s_g + D / 2 + c * 4);
        const float4 b0 = *reinterpret_cast<const float4*>(s_b + c * 4);
        const float4 b1 = *reinterpret_cast<const float4*>(s_b + D / 2 + c * 4);
        g[0] = pack2(g0.x, g0.y); g[1] = pack2(g0.z, g0.w); g[2] = pack2(g1.x, g1.y); g[3] = pack2(g1.z, g1.w);
        b[0] = pack2(b0.x, b0.y); b[1] = pack2(b0.z, b0.w); b[2] = pack2(b1.x, b1.y); b[3] = pack2(b1.z, b1.w);
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
          // Eq. 4: clip(round(t) + z, 0, qmax): round half to even by the float -> int conversion, then the
          // packing instruction saturates to the container ([0, 15] or [0, 255])
          int q[kChunk];
          if (kPerRow ? !decltype(guarded)::value : !guard) {
#pragma unroll
            for (int e = 0; e < kChunk / 2; ++e) {
              float u0, u1;
              unpack2(add2(fma2(normalised(v[r][i][e], r), g[e], b[e]), magic2), u0, u1);
              q[2 * e] = __float_as_int(u0) + z_less_magic;
              q[2 * e + 1] = __float_as_int(u1) + z_less_magic;
            }
          } else {
            float t[kChunk];
#pragma unroll
            for (int e = 0; e < kChunk / 2; ++e) unpack2(fma2(normalised(v[r][i][e], r), g[e], b[e]), t[2 * e], t[2 * e + 1]);
#pragma unroll
            for (int e = 0; e < kChunk; ++e) q[e] = __float2int_rn(fminf(fmaxf(t[e], -1.0e9f), 1.0e9f)) + z;
          }
          // rows past the end compute on a copy of the last row; only the stores are predicated
          if constexpr (kPack4) {
            uint32_t w = 0;
#pragma unroll
            for (int e = kChunk - 2; e >= 0; e -= 2) w = push_pair_u4(q[e], q[e + 1], w);
            if (live[r]) reinterpret_cast<uint32_t*>(out[r])[c] = w;
            csum[r] = int(__dp4a(w & 0x0F0F0F0Fu, 0x01010101u, __dp4a((w >> 4) & 0x0F0F0F0Fu, 0x01010101u, uint32_t(csum[r]))));
          } else {
            uint2 w;
            w.x = push_pair_u8(q[0], q[1], push_pair_u8(q[2], q[3], 0u));
            w.y = push_pair_u8(q[4], q[5], push_pair_u8(q[6], q[7], 0u));
            w.x = __vminu4(w.x, qmax4);          // 4- and 6-bit quantizers in byte containers
            w.y = __vminu4(w.y, qmax4);
            if (live[r]) reinterpret_cast<uint2*>(out[r])[c] = w;
            csum[r] = int(__dp4a(w.x, 0x01010101u, __dp4a(w.y, 0x01010101u, uint32_t(csum[r]))));
          }
        }
      }
    }
    };
    if (kPerRow && guard) chunks(std::true_type{});
    else chunks(std::false_type{});
    if (row_sum != nullptr) {
      if constexpr (!kWide) {
        group_sum<TPR, kRows>(csum);
        if (tig == 0) {
#pragma unroll
          for (int r = 0; r < kRows; ++r)
            if (row0 + r < rows) row_sum[row0 + r] = csum[r];
        }
      } else {
        group_sum<32, kRows>(csum);
        if ((threadIdx.x & 31) == 0) {
#pragma unroll
          for (int r = 0; r < kRows; ++r) red_c[parity][(threadIdx.x >> 5) * kRows + r] = csum[r];
        }
        last_row0 = row0;
      }
    }
  }
  if constexpr (kWide) {
    if (row_sum != nullptr && parity_seen) {
      group_sync<TPR>(group_first_warp);
      if (tig < kRows) {
        int t = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) t += red_c[parity ^ 1][(group_first_warp + w) * kRows + tig];
        if (last_row0 + tig < rows) row_sum[last_row0 + tig] = t;
      }
    }
  }
  if (beside) grid_dependency_wait();
}


// ---- bf16 rows of 2048 or 4096 elements, many of them: a row per warp
//
// With a row over several warps 4.4 of 10.9 instructions per element were what a row costs beside its elements (shuffles, merges, a barrier,
// addresses, paid per warp), and 16 warps per SM waited for one another.  Here a lane holds all of a row's chunks of 8 elements that
// its namesakes in the kSlices warps of ln_quant_kernel hold, as packed float pairs (64 or 128 registers), and there is no barrier in the
// loop.  The registers leave no room for a row in flight, so a warp's next two rows are under way in shared memory, by one bulk copy
// each.  A buffer is filled again one iteration after it was read: by then everything computed from it has been issued, so its loads
// have returned.  The sums are formed slice by slice in the order of ln_quant_kernel, so that a row's codes do not depend on how many
// rows share the call.
// New inputs, groups of warps -> this: 32768 x 4096 to packed codes 77.1 -> 63.4 us, to bytes 83.1 -> 69.4, 20000 x 4096 RMS 46.5 -> 40.1,
// 65536 x 2048 73.5 -> 63.1.  The form for large factors is chosen once per row: a branch per chunk cost 10 us at 4096.  Eight warps of 200
// registers took 66 us where this took 59.0.  Two rows per warp with half of a row each, which reads the factors half as
// often, took 89 us: twelve warps are few, and each then waits on twice the work of one iteration.
template <int kSlices> constexpr int row_warps() { return kSlices == 4 ? 12 : 20; }      // by 168 and 96 registers a thread
template <int kSlices, bool kPack4>
__global__ void __launch_bounds__(32 * row_warps<kSlices>(), 1)
ln_rows_kernel(const __nv_bfloat16* __restrict__ x, uint32_t rows, int64_t ldx, const float* __restrict__ gamma_t,
               const float* __restrict__ beta_t, float eps, int rms, float inv_s, int z, int qmax, uint8_t* __restrict__ codes, int64_t ldc,
               int32_t* __restrict__ row_sum, int32_t* __restrict__ clear, int64_t n_clear, Params params, int32_t* status) {
  const bool settled = params == Params::settled, beside = params == Params::beside;
  constexpr int kWarps = row_warps<kSlices>(), kBlock = 32 * kWarps, kPer = 4, kVPT = kSlices * kPer;
  constexpr int D = 32 * kVPT * kChunk;
  constexpr uint32_t kRowBytes = D * 2u;
  extern __shared__ __align__(128) float s_gb[];         // gamma~/s~, beta~/s~ (halves of chunks apart), then two rows per warp
  __shared__ alignas(8) uint64_t full[kWarps][2];
  __shared__ volatile int abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t buf = tc::smem_u32(s_gb + 2 * D) + uint32_t(warp) * 2u * kRowBytes;
  if (lane < 2) tc::mbar_init(tc::smem_u32(&full[warp][lane]), 1);
  if (tid == 0) abort = 0;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncwarp();

  constexpr int kPieces = D / 4;
  const int rot = int(blockIdx.x * 32u % uint32_t(kPieces));
  const bool vec = ((reinterpret_cast<uintptr_t>(gamma_t) | reinterpret_cast<uintptr_t>(beta_t)) & 15) == 0;
  auto load4 = [&](const float* p) {
    return vec ? __ldcg(reinterpret_cast<const float4*>(p)) : make_float4(__ldcg(p), __ldcg(p + 1), __ldcg(p + 2), __ldcg(p + 3));
  };
  const uint32_t stride = gridDim.x * kWarps, first = uint32_t(warp) * gridDim.x + blockIdx.x;
  auto request = [&](uint32_t row, int k) {
    if (lane == 0 && row < rows) {
      const uint32_t bar = tc::smem_u32(&full[warp][k & 1]);
      tc::mbar_expect_tx(bar, kRowBytes);
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   ::"r"(buf + uint32_t(k & 1) * kRowBytes), "l"(x + int64_t(row) * ldx), "r"(kRowBytes), "r"(bar) : "memory");
    }
  };
  auto begin = [&] {
    if (!beside) grid_dependency_wait();
    grid_dependency_trigger();
    request(first, 0);
    request(first + stride, 1);
  };
  if (!settled) begin();               // (factors that the kernel ahead may have written are read behind the wait, as in ln_quant_kernel)
  constexpr int kOwn = (kPieces + kBlock - 1) / kBlock;  // a thread's pieces, all in flight at once
  float4 g4[kOwn], b4[kOwn];
  const float root_d = sqrtf(float(D));
  bool wide = false;
#pragma unroll
  for (int i = 0; i < kOwn; ++i) {
    const int q = (tid + i * kBlock + rot) % kPieces;
    if (tid + i * kBlock < kPieces) { g4[i] = load4(gamma_t + 4 * q); b4[i] = load4(beta_t + 4 * q); }
  }
#pragma unroll
  for (int i = 0; i < kOwn; ++i) {
    const int q = (tid + i * kBlock + rot) % kPieces, at = (q & 1) * (D / 2) + (q >> 1) * 4;
    if (tid + i * kBlock < kPieces) {
      const float gi[4] = {g4[i].x * inv_s, g4[i].y * inv_s, g4[i].z * inv_s, g4[i].w * inv_s};
      const float bi[4] = {b4[i].x * inv_s, b4[i].y * inv_s, b4[i].z * inv_s, b4[i].w * inv_s};
      *reinterpret_cast<float4*>(s_gb + at) = make_float4(gi[0], gi[1], gi[2], gi[3]);
      *reinterpret_cast<float4*>(s_gb + D + at) = make_float4(bi[0], bi[1], bi[2], bi[3]);
#pragma unroll
      for (int e = 0; e < 4; ++e) wide = wide || !(fabsf(gi[e]) * root_d + fabsf(bi[e]) < 4.0e6f);
    }
  }
  const bool guard = __syncthreads_or(wide) != 0;          // (as in ln_quant_kernel)
  if (settled) begin();
  for (int64_t i = int64_t(blockIdx.x) * kBlock + tid; i < n_clear; i += int64_t(gridDim.x) * kBlock) clear[i] = 0;

  // Totals over the lanes for every slice: the first steps of the tree split the slices between the halves of the warp (the pairs that
  // are added are those of a tree per slice); lane l ends with slice l / 8 or l / 16.
  auto totals = [&](const float (&t)[kSlices]) {
    const bool high = lane & 16;
    float u;
    if constexpr (kSlices == 4) {
      const float a = (high ? t[2] : t[0]) + __shfl_xor_sync(0xffffffffu, high ? t[0] : t[2], 16);
      const float b = (high ? t[3] : t[1]) + __shfl_xor_sync(0xffffffffu, high ? t[1] : t[3], 16);
      const bool next = lane & 8;
      u = (next ? b : a) + __shfl_xor_sync(0xffffffffu, next ? a : b, 8);
    } else {
      u = (high ? t[1] : t[0]) + __shfl_xor_sync(0xffffffffu, high ? t[0] : t[1], 16);
      u += __shfl_xor_sync(0xffffffffu, u, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
    return u;
  };
  auto over_slices = [&](float u) {    // sum over the slices, in the order of their distance
    u += __shfl_xor_sync(0xffffffffu, u, 16);
    if constexpr (kSlices == 4) u += __shfl_xor_sync(0xffffffffu, u, 8);
    return u;
  };
  constexpr float kSliceSize = float(32 * kPer * kChunk);
  const float inv_d = 1.f / float(D);
  const uint32_t qmax4 = uint32_t(qmax) * 0x01010101u;
  const f32x2 magic2 = splat2(__int_as_float(kMagicBits));
  const int z_less_magic = z - kMagicBits;
  int k = 0;
  uint32_t row = first;
  for (; row < rows; row += stride, ++k) {
    if (k > 0) request(row + stride, k + 1);
    const bool came = tc::mbar_wait(tc::smem_u32(&full[warp][k & 1]), (k >> 1) & 1, &abort, 91, status);
    if (!__all_sync(0xffffffffu, came)) break;
    f32x2 v[kVPT][kChunk / 2];
    const uint32_t at = buf + uint32_t(k & 1) * kRowBytes + uint32_t(lane) * 16u;
#pragma unroll
    for (int i = 0; i < kVPT; ++i) {
      RawChunk<__nv_bfloat16> raw;
      asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(raw.a.x), "=r"(raw.a.y), "=r"(raw.a.z), "=r"(raw.a.w) : "r"(at + uint32_t(i) * 512u));
      expand(raw, v[i]);
    }
    // (a slice's mean, and later the rest of the way to the row's, stays with the lanes that own the slice and is fetched where it is
    // used: 128 registers of values leave no room for all of them)
    float t[kSlices], own_sum = 0.f;
    if (!rms) {
#pragma unroll
      for (int w = 0; w < kSlices; ++w) {
        f32x2 acc = 0ull;
#pragma unroll
        for (int i = w; i < kVPT; i += kSlices)
#pragma unroll
          for (int e = 0; e < kChunk / 2; ++e) acc = add2(acc, v[i][e]);
        float lo, hi;
        unpack2(acc, lo, hi);
        t[w] = lo + hi;
      }
      own_sum = totals(t);
    }
    const float own_mean = own_sum * (1.f / kSliceSize);
#pragma unroll
    for (int w = 0; w < kSlices; ++w) {
      const f32x2 neg_mu = splat2(-__shfl_sync(0xffffffffu, own_mean, (32 / kSlices) * w));
      f32x2 acc = 0ull;
#pragma unroll
      for (int i = w; i < kVPT; i += kSlices)
#pragma unroll
        for (int e = 0; e < kChunk / 2; ++e) {
          v[i][e] = add2(v[i][e], neg_mu);
          acc = fma2(v[i][e], v[i][e], acc);
        }
      float lo, hi;
      unpack2(acc, lo, hi);
      t[w] = lo + hi;
    }
    const float mean = rms ? 0.f : over_slices(own_sum) * inv_d;
    const float off = rms ? 0.f : own_mean - mean;
    const float m2 = over_slices(fmaf(kSliceSize * off, off, totals(t)));
    const float rs = rsqrtf(m2 * inv_d + eps);
    const f32x2 rstd = splat2(rs);
    const float own_rest = (own_mean - mean) * rs;
    int csum[1] = {0};
    uint8_t* out = codes + int64_t(row) * ldc;
    auto chunks = [&](auto guarded) {
#pragma unroll
    for (int w = 0; w < kSlices; ++w) {
      const f32x2 rest = splat2(__shfl_sync(0xffffffffu, own_rest, (32 / kSlices) * w));
#pragma unroll
      for (int i = w; i < kVPT; i += kSlices) {
        const int c = lane + 32 * i;
        const float4 g0 = *reinterpret_cast<const float4*>(s_gb + c * 4), g1 = *reinterpret_cast<const float4*>(s_gb + D / 2 + c * 4);
        const float4 b0 = *reinterpret_cast<const float4*>(s_gb + D + c * 4), b1 = *reinterpret_cast<const float4*>(s_gb + D + D / 2 + c * 4);
        const f32x2 g[kChunk / 2] = {pack2(g0.x, g0.y), pack2(g0.z, g0.w), pack2(g1.x, g1.y), pack2(g1.z, g1.w)};
        const f32x2 b[kChunk / 2] = {pack2(b0.x, b0.y), pack2(b0.z, b0.w), pack2(b1.x, b1.y), pack2(b1.z, b1.w)};
        int q[kChunk];
#pragma unroll
        for (int e = 0; e < kChunk / 2; ++e) {
          const f32x2 u = fma2(fma2(v[i][e], rstd, rest), g[e], b[e]);
          float u0, u1;
          if constexpr (decltype(guarded)::value) {
            unpack2(u, u0, u1);
            q[2 * e] = __float2int_rn(fminf(fmaxf(u0, -1.0e9f), 1.0e9f)) + z;
            q[2 * e + 1] = __float2int_rn(fminf(fmaxf(u1, -1.0e9f), 1.0e9f)) + z;
          } else {
            unpack2(add2(u, magic2), u0, u1);
            q[2 * e] = __float_as_int(u0) + z_less_magic;
            q[2 * e + 1] = __float_as_int(u1) + z_less_magic;
          }
        }
        if constexpr (kSlices == 4) __syncwarp();        // keeps the chunks apart: interleaved, they spill (67.7 us instead of 59.0)
        if constexpr (kPack4) {
          uint32_t p = 0;
#pragma unroll
          for (int e = kChunk - 2; e >= 0; e -= 2) p = push_pair_u4(q[e], q[e + 1], p);
          reinterpret_cast<uint32_t*>(out)[c] = p;
          csum[0] = int(__dp4a(p & 0x0F0F0F0Fu, 0x01010101u, __dp4a((p >> 4) & 0x0F0F0F0Fu, 0x01010101u, uint32_t(csum[0]))));
        } else {
          uint2 p;
          p.x = __vminu4(push_pair_u8(q[0], q[1], push_pair_u8(q[2], q[3], 0u)), qmax4);      // 4- and 6-bit quantizers in byte containers
          p.y = __vminu4(push_pair_u8(q[4], q[5], push_pair_u8(q[6], q[7], 0u)), qmax4);
          reinterpret_cast<uint2*>(out)[c] = p;
          csum[0] = int(__dp4a(p.x, 0x01010101u, __dp4a(p.y, 0x01010101u, uint32_t(csum[0]))));
        }
      }
    }
    };
    if (guard) chunks(std::true_type{});
    else chunks(std::false_type{});
    if (row_sum != nullptr) {
      group_sum<32, 1>(csum);
      if (lane == 0) row_sum[row] = csum[0];
    }
  }
  // given up: the copies under way must have landed before the block may exit
  if (row < rows && lane == 0) {
    tc::mbar_drain(tc::smem_u32(&full[warp][k & 1]), (k >> 1) & 1);
    if (row + stride < rows) tc::mbar_drain(tc::smem_u32(&full[warp][(k + 1) & 1]), ((k + 1) >> 1) & 1);
  }
  if (beside) grid_dependency_wait();
}

template <typename T>
struct Call {
  const T* x;
  int64_t rows;
  int D;
  int64_t ldx;
  const float *gamma_t, *beta_t;
  float eps;
  int rms;
  float s_t;
  int z, bits;
  uint8_t* codes;
  int64_t ldc;
  int32_t* row_sum;
  ClearWords clear;
  Params params;
};

template <typename T, int TPR, int kVPT, bool kPack4, bool kFull>
repq_status launch(const Call<T>& c, cudaStream_t st) {
  constexpr int kBlock = TPR > 256 ? TPR : 256;
  constexpr int kRowsPerBlock = kBlock / TPR * rows_in_flight(kVPT, TPR, sizeof(T));
  constexpr int kMostSmem = TPR * kVPT * kChunk * 2 * int(sizeof(float));
  auto kern = ln_quant_kernel<T, TPR, kVPT, kPack4, kFull>;
  const int64_t need = (c.rows + kRowsPerBlock - 1) / kRowsPerBlock;
  const size_t smem = size_t(c.D) * 2 * sizeof(float);
  if constexpr (kMostSmem > 40 * 1024) REPQ_TRY((allow_smem<ln_quant_kernel<T, TPR, kVPT, kPack4, kFull>>(kMostSmem)));
  static Residency memo;
  // persistent grid: exactly the blocks that are resident at once, so that every block keeps its load pipeline
  // running over all of its rows
  int resident = 0;
  REPQ_TRY(resident_blocks(memo, kern, kBlock, smem, &resident));
  const int64_t cap = int64_t(sm_count()) * resident;
  const int grid = int(need < cap ? need : cap);
  REPQ_CUDA(launch_chained(kern, dim3(grid), dim3(kBlock), smem, st, c.x, c.rows, c.D, c.ldx, c.gamma_t, c.beta_t, c.eps, c.rms, 1.f / c.s_t,
                           c.z, code_max(c.bits), c.codes, c.ldc, c.row_sum, c.clear.at, c.clear.n, c.params));
  note_launch();
  return REPQ_OK;
}

template <int kSlices, bool kPack4>
repq_status launch_rows(const Call<__nv_bfloat16>& c, cudaStream_t st) {
  constexpr int kWarps = row_warps<kSlices>(), kD = 1024 * kSlices, kSmem = kD * 8 + kWarps * 2 * kD * 2;
  static_assert(kSmem <= 226 * 1024, "rows and factors exceed shared memory");
  REPQ_TRY((allow_smem<ln_rows_kernel<kSlices, kPack4>>(kSmem)));
  int32_t* status = device_status_word();
  REPQ_REQUIRE(status != nullptr, REPQ_CUDA_ERROR, "ln_quant: device status word unavailable");
  REPQ_CUDA(launch_chained(ln_rows_kernel<kSlices, kPack4>, dim3(sm_count()), dim3(32 * kWarps), size_t(kSmem), st, c.x, uint32_t(c.rows), c.ldx, c.gamma_t,
                           c.beta_t, c.eps, c.rms, 1.f / c.s_t, c.z, code_max(c.bits), c.codes, c.ldc, c.row_sum, c.clear.at, c.clear.n,
                           c.params, status));
  note_launch();
  return REPQ_OK;
}
// Rows of a call from which a row per warp is ahead: about four and a half turns of the warps at 4096 elements (new inputs, packed codes, by groups
// of warps and by single ones: 4096 rows 12.9 and 14.6 us, 7000 19.7 and 19.8, 7992 22.2 and 21.5, 10000 26.7 and 25.0), five at 2048 (12000 16.4 and
// 16.6, 14000 18.8 and 18.0, 14800 19.9 and 18.6, 16000 21.1 and 19.7).  3072 elements gained nothing (63.9 and 63.8), rows that do not fill the chunks lost.
template <int kSlices>
bool many_rows(int64_t rows) { return rows < (int64_t(1) << 31) && 2 * rows >= int64_t(kSlices == 4 ? 9 : 10) * row_warps<kSlices>() * sm_count(); }

// Chunks per thread kVPT .. kMost, the row lengths that narrower groups leave to groups of TPR threads.
template <typename T, int TPR, int kVPT, int kMost>
repq_status launch_group(const Call<T>& c, cudaStream_t st) {
  if constexpr (kVPT < kMost) {
    if (c.D > TPR * kVPT * kChunk) return launch_group<T, TPR, kVPT + 1, kMost>(c, st);
  }
  const bool full = c.D == TPR * kVPT * kChunk;   // the row fills the group exactly: no chunk is predicated
  if (packed4(c.bits)) return full ? launch<T, TPR, kVPT, true, true>(c, st) : launch<T, TPR, kVPT, true, false>(c, st);
  return full ? launch<T, TPR, kVPT, false, true>(c, st) : launch<T, TPR, kVPT, false, false>(c, st);
}

template <typename T>
repq_status dispatch(const Call<T>& c, cudaStream_t st) {
  const int nchunks = c.D / kChunk;
  // The fewest warps whose threads hold the row in at most six chunks: a row of one warp has no barrier, and what a row costs
  // beside its elements (shuffles, merges, barrier) is paid per thread (measured, 1536 elements: 45 us with one warp, 59 with
  // two; 3072: 49 and 61).  Eight chunks leave too few warps on the SM (2048 float elements: 56 against 48).
  if (nchunks <= 8 * 4) return launch_group<T, 8, 1, 4>(c, st);
  if (nchunks <= 16 * 4) return launch_group<T, 16, 3, 4>(c, st);
  if (nchunks <= 32 * 6) return launch_group<T, 32, 3, 6>(c, st);
  if constexpr (sizeof(T) == 2) {
    if (c.D == 2048 && many_rows<2>(c.rows)) return packed4(c.bits) ? launch_rows<2, true>(c, st) : launch_rows<2, false>(c, st);
    if (c.D == 4096 && many_rows<4>(c.rows)) return packed4(c.bits) ? launch_rows<4, true>(c, st) : launch_rows<4, false>(c, st);
  }
  if (nchunks <= 64 * 6) return launch_group<T, 64, 4, 6>(c, st);
  if (nchunks <= 128 * 6) return launch_group<T, 128, 4, 6>(c, st);
  if (nchunks <= 256 * 4) return launch_group<T, 256, 4, 4>(c, st);
  if (nchunks <= 512 * 4) return launch_group<T, 512, 3, 4>(c, st);
  return fail(REPQ_UNSUPPORTED, "ln_quant: D = %d exceeds 16384", c.D);
}

}  // namespace

repq_status launch_ln_quant(const void* x, int x_dtype, int64_t rows, int D, int64_t ldx, const float* gamma_t,
                            const float* beta_t, float eps, int norm_kind, float s_t, int z_t, int bits, uint8_t* codes,
                            int64_t ld_codes_bytes, int32_t* row_sum, ClearWords clear, Params params, cudaStream_t st) {
  REPQ_REQUIRE(rows >= 0 && D > 0, REPQ_INVALID_ARG, "ln_quant: rows must be >= 0 and D > 0");
  if (rows == 0) return REPQ_OK;
  REPQ_REQUIRE(x && gamma_t && beta_t && codes, REPQ_INVALID_ARG, "ln_quant: NULL pointer");
  REPQ_REQUIRE(x_dtype == REPQ_F32 || x_dtype == REPQ_BF16, REPQ_INVALID_ARG, "ln_quant: x_dtype must be REPQ_F32 or REPQ_BF16");
  REPQ_REQUIRE(norm_kind == REPQ_NORM_LAYERNORM || norm_kind == REPQ_NORM_RMS, REPQ_INVALID_ARG, "ln_quant: unknown norm_kind");
  REPQ_REQUIRE(bits_ok(bits), REPQ_INVALID_ARG, "ln_quant: bits must be 4, 6 or 8");
  REPQ_REQUIRE(s_t > 0.f && eps >= 0.f, REPQ_INVALID_ARG, "ln_quant: s_t must be positive and eps non-negative");
  REPQ_REQUIRE(z_t > -(1 << 20) && z_t < (1 << 20), REPQ_INVALID_ARG, "ln_quant: |z_t| must be below 2^20");
  REPQ_REQUIRE(D % 8 == 0, REPQ_UNSUPPORTED, "ln_quant: D = %d must be a multiple of 8", D);
  REPQ_REQUIRE(D <= 16384, REPQ_UNSUPPORTED, "ln_quant: D = %d exceeds 16384", D);
  REPQ_REQUIRE(ldx >= D, REPQ_INVALID_ARG, "ln_quant: ldx < D");
  const size_t esz = x_dtype == REPQ_F32 ? 4 : 2;
  REPQ_REQUIRE(aligned(x, 16) && (size_t(ldx) * esz) % 16 == 0, REPQ_ALIGNMENT, "ln_quant: x rows must be 16-byte aligned");
  const int64_t unit = packed4(bits) ? 4 : 8;
  REPQ_REQUIRE(ld_codes_bytes >= code_row_bytes(D, bits), REPQ_INVALID_ARG, "ln_quant: ld_codes_bytes shorter than a row");
  REPQ_REQUIRE(aligned(codes, unit) && ld_codes_bytes % unit == 0, REPQ_ALIGNMENT,
               "ln_quant: codes rows must be %d-byte aligned", int(unit));
  auto run = [&](auto* typed) {
    return dispatch(Call<std::remove_const_t<std::remove_pointer_t<decltype(typed)>>>{
        typed, rows, D, ldx, gamma_t, beta_t, eps, norm_kind == REPQ_NORM_RMS, s_t, z_t, bits, codes, ld_codes_bytes, row_sum, clear,
        params}, st);
  };
  return x_dtype == REPQ_F32 ? run(static_cast<const float*>(x)) : run(static_cast<const __nv_bfloat16*>(x));
}

}  // namespace repq

extern "C" repq_status repq_ln_quant(const void* x, int x_dtype, int64_t rows, int D, int64_t ldx,
                                     const float* gamma_t, const float* beta_t, float eps, int norm_kind,
                                     float s_t, int z_t, int bits, uint8_t* codes, int64_t ld_codes_bytes,
                                     int32_t* row_sum, void* stream) {
  return repq::launch_ln_quant(x, x_dtype, rows, D, ldx, gamma_t, beta_t, eps, norm_kind, s_t, z_t, bits, codes, ld_codes_bytes,
                               row_sum, repq::ClearWords{}, repq::Params::streamed, static_cast<cudaStream_t>(stream));
}
