// Per-channel dual clipping (Sec. III-D, Eqs. 18-20): the step that hands the channel-wise quantizer of the
// LayerNorm activations its bounds, just before the scale reparameterization.  Every channel d learns two factors,
//     x_up = max_d * sigmoid(alpha1_d),   x_low = min_d * sigmoid(alpha2_d)                      (Eqs. 18-19)
// by Adam on ||X'_{:,d} - X^'_{:,d}||^2 (Eq. 20), X^' the de-quantized channel-wise quantization (Eqs. 4-6) on those
// bounds.  The round operations are passed straight through in the backward direction and the clip passes the
// gradient on [0, 2^b - 1] inclusive: with u = x/s, zc = -x_low/s, r = round(u), z = round(zc), q = clip(r + z),
//     inside the clip   dx^/ds = r - u            dx^/dx_low (s fixed) = 0
//     clipped           dx^/ds = q - z + zc       dx^/dx_low (s fixed) = 1
// and s = (x_up - x_low) / (2^b - 1).
//
// Inside the clip dx^/ds = (x^ - x)/s, so the gradient with respect to s is 2/s times the squared error of those values;
// with d = q - z - u (the error in units of s) one pass over a channel has to sum d^2 over the values inside the clip and d
// over the values clipped at either end, and the objective is s^2 sum d^2.
//
// Channels are independent, so the whole optimisation of a channel stays inside one CTA (1 to 16 warps), which holds the
// channel's values in shared memory from the first pass to the last.  Two forms:
//  - passes over the values in every step.  What bounds them is the float64 pipe (64 lanes per cycle and SM: five operations per
//    value and step) and, for few values per channel, the chain of one step: reduction, exp, square root, divisions (ncu, 6304 x
//    384: float64 pipe 34 % busy, conversions to double 23 % of theirs, first stall the barrier around the reduction and the
//    update).  Hence the quotient by a reciprocal taken once per step, the round operation by adding 1.5 * 2^52 (its integer,
//    in the low word, also decides the clip, on the integer pipe), and several CTAs per SM, so that one channel's chain runs
//    under the others' passes.
//  - values sorted once, a step's sums from prefix sums at the edges between the 16 codes of a 4-bit quantizer.  What bounds it is the
//    chain of a step alone (1.15 us: 16 cycles per float64 operation, 90 to 220 for a square root, a division, the sigmoid), one warp per
//    channel without a barrier.  100 steps, passes -> this: 6304 x 384 294 -> 158 us, 12608 x 768 823 -> 557, 591 x 4096 398 -> 250,
//    20000 x 1024 1754 -> 1219, 64 x 384 136 -> 125; the objective adds 2 to 45.  The learned bounds are the same floats.
//    A full merge sort took 85 us of 6304 x 384 against 25 for buckets and ranks.
// Arithmetic is float64 throughout (the decisions of the two round operations steer the gradient).
// No scratch memory, no inter-CTA traffic, no atomics outside the counting of the sort (whose result does not depend on their order).
// Channels of more values than shared memory holds take the kernel that re-reads them: a CTA owns 8 neighbouring channels
// (one 32-byte sector per token row) and 32 token lanes, every step is one pass over the CTA's slab.
#include <cuda_bf16.h>
#include <math_constants.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.h"

namespace repq {
namespace {

constexpr int kCh = 8;            // channels per CTA
constexpr int kLanes = 32;        // token lanes per channel
constexpr int kThreads = kCh * kLanes;

struct ClipParams {
  const float* x; int64_t n, ldx; int D;
  double Q; int iters; double lr, alpha0, beta1, beta2, eps;
  float* x_low; float* x_up; double* loss;
};

constexpr int kMaxResident = 50 * 1024;        // values of a channel that fit the shared memory of one CTA


// Sorted form: most values of a channel (its 10 bytes per value fill shared memory), values of a bucket above which the channel
// counts as crowded (ranks cost a bucket's square; the densest of a normal channel's buckets holds three times the average of
// 1 << shift and its scatter), buckets of n values, shared memory.
constexpr int kMaxSorted = 22 * 1024;
__host__ __device__ constexpr int crowd(int shift) { return 16 + (4 << shift); }
__host__ __device__ constexpr int sorted_buckets(int n, int shift) { return (n >> shift) + 8; }
constexpr size_t sorted_bytes(int64_t n, int shift) {
  const int64_t n8 = (n + 7) / 8 * 8;
  return size_t(2 * n8 + 4 + sorted_buckets(int(n), shift) + 1) * 4;
}

__device__ __forceinline__ double sigmoid(double a) { return 1.0 / (1.0 + exp(-a)); }

__global__ void __launch_bounds__(kThreads) dual_clip_kernel(ClipParams P) {
  __shared__ double red[3][kLanes][kCh];
  __shared__ double sh_s[kCh], sh_low[kCh];
  const int ch = threadIdx.x % kCh, lane = threadIdx.x / kCh;
  const int d = blockIdx.x * kCh + ch;
  const bool on = d < P.D;
  const float* col = P.x + (on ? d : 0);

  // ---- extremes of the channel
  double mx = -INFINITY, mn = INFINITY;
  if (on)
    for (int64_t t = lane; t < P.n; t += kLanes) {
      const double v = double(__ldg(col + t * P.ldx));
      mx = fmax(mx, v);
      mn = fmin(mn, v);
    }
  red[0][lane][ch] = mx;
  red[1][lane][ch] = mn;
  __syncthreads();
  double x_max = 0.0, x_min = 0.0;
  // state of the channel's first thread
  double a1 = P.alpha0, a2 = P.alpha0, m1 = 0.0, v1 = 0.0, m2 = 0.0, v2 = 0.0, sg1 = 0.0, sg2 = 0.0;
  double b1t = 1.0, b2t = 1.0;
  if (lane == 0) {
    x_max = red[0][0][ch];
    x_min = red[1][0][ch];
    for (int l = 1; l < kLanes; ++l) {
      x_max = fmax(x_max, red[0][l][ch]);
      x_min = fmin(x_min, red[1][l][ch]);
    }
  }
  double loss_first = 0.0;
  for (int it = 0; it <= P.iters; ++it) {
    // the channel's quantizer for this iteration (Eq. 6 on the bounds of Eqs. 18-19)
    if (lane == 0) {
      sg1 = sigmoid(a1);
      sg2 = sigmoid(a2);
      const double up = x_max * sg1, low = x_min * sg2;
      sh_s[ch] = (up - low) / P.Q;
      sh_low[ch] = low;
    }
    __syncthreads();
    const double s = sh_s[ch], low = sh_low[ch];
    const double zc = -low / s, z = rint(zc);
    double acc_loss = 0.0, acc_ds = 0.0, acc_dl = 0.0;
    // a channel whose bounds coincide (a constant channel, or extremes of 0) has no quantizer to learn: its sums stay
    // 0, its factors keep their starting value and the contracted extremes are returned as they are
    if (on && s > 0.0)
      for (int64_t t = lane; t < P.n; t += kLanes) {
        const double x = double(__ldg(col + t * P.ldx));
        const double u = x / s, r = rint(u), pre = r + z;
        const double q = fmin(fmax(pre, 0.0), P.Q);
        const double e = s * (q - z) - x;
        const bool inside = pre >= 0.0 && pre <= P.Q;
        acc_loss += e * e;
        acc_ds += 2.0 * e * (inside ? r - u : q - z + zc);
        acc_dl += inside ? 0.0 : 2.0 * e;
      }
    red[0][lane][ch] = acc_loss;
    red[1][lane][ch] = acc_ds;
    red[2][lane][ch] = acc_dl;
    __syncthreads();
    if (lane == 0) {
      double loss = 0.0, dL_ds = 0.0, dL_dl = 0.0;
      for (int l = 0; l < kLanes; ++l) {
        loss += red[0][l][ch];
        dL_ds += red[1][l][ch];
        dL_dl += red[2][l][ch];
      }
      if (it == 0) loss_first = loss;
      if (it == P.iters) {
        // the pass after the last update: the objective that the returned bounds reach
        if (on) {
          P.x_up[d] = float(x_max * sg1);
          P.x_low[d] = float(x_min * sg2);
          if (P.loss) {
            P.loss[d] = loss_first;
            P.loss[P.D + d] = loss;
          }
        }
      } else {
        const double g1 = dL_ds / P.Q * x_max * sg1 * (1.0 - sg1);
        const double g2 = (dL_dl - dL_ds / P.Q) * x_min * sg2 * (1.0 - sg2);
        m1 = P.beta1 * m1 + (1.0 - P.beta1) * g1;
        v1 = P.beta2 * v1 + (1.0 - P.beta2) * g1 * g1;
        m2 = P.beta1 * m2 + (1.0 - P.beta1) * g2;
        v2 = P.beta2 * v2 + (1.0 - P.beta2) * g2 * g2;
        b1t *= P.beta1;
        b2t *= P.beta2;
        a1 -= P.lr * (m1 / (1.0 - b1t)) / (sqrt(v1 / (1.0 - b2t)) + P.eps);
        a2 -= P.lr * (m2 / (1.0 - b1t)) / (sqrt(v2 / (1.0 - b2t)) + P.eps);
      }
    }
    // the next iteration's writes of sh_s / red follow this barrier
    __syncthreads();
  }
}

// Sums of one pass over a channel.
struct ClipSums { double in2, low, high, out2; };      // sum d^2 inside the clip, sum d clipped at 0 / at Q, sum d^2 clipped

// kN values at once: the operations of all of them side by side, one branch for the common case that none is clipped.
// kSmall: every quotient and zero point is below 2^30 in magnitude, so that integers decide the clip.
template <bool kSmall, int kN>
__device__ __forceinline__ void clip_values(const float (&xs)[kN], double inv, double lo, double hi, int zi, uint32_t qi, ClipSums& a,
                                            double& in2b) {
  double u[kN], d[kN];
  bool inside[kN], all = true;
#pragma unroll
  for (int i = 0; i < kN; ++i) {
    u[i] = double(xs[i]) * inv;
    if (kSmall) {
      const double t = u[i] + 6755399441055744.0;       // 1.5 * 2^52: round half to even, the integer in the low word
      d[i] = (t - 6755399441055744.0) - u[i];
      inside[i] = uint32_t(__double2loint(t) + zi) <= qi;
    } else {
      const double r = rint(u[i]);
      d[i] = r - u[i];
      inside[i] = r >= lo && r <= hi;
    }
    all = all && inside[i];
  }
  if (all) {
#pragma unroll
    for (int i = 0; i < kN; ++i) {
      if (i & 1) in2b = fma(d[i], d[i], in2b); else a.in2 = fma(d[i], d[i], a.in2);
    }
  } else {
#pragma unroll
    for (int i = 0; i < kN; ++i) {
      if (inside[i]) {
        a.in2 = fma(d[i], d[i], a.in2);
      } else if (u[i] < lo) {                           // (a rounded value below lo, an integer, comes from u < lo)
        const double e = lo - u[i];
        a.low += e;
        a.out2 = fma(e, e, a.out2);
      } else {
        const double e = hi - u[i];
        a.high += e;
        a.out2 = fma(e, e, a.out2);
      }
    }
  }
}

// Sum over the warp of four values per lane: two exchanges that halve the values a lane carries, three plain steps.  Lane l
// returns the total of value l mod 4 (in2, low, high, out2).
__device__ __forceinline__ double warp_sum4(const ClipSums& a, int lane) {
  const bool p = lane & 1, q = lane & 2;
  const double k0 = p ? a.low : a.in2, k1 = p ? a.out2 : a.high;
  const double x0 = k0 + __shfl_xor_sync(0xffffffffu, p ? a.in2 : a.low, 1), x1 = k1 + __shfl_xor_sync(0xffffffffu, p ? a.high : a.out2, 1);
  double t = (q ? x1 : x0) + __shfl_xor_sync(0xffffffffu, q ? x0 : x1, 2);
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// One channel per CTA of kWarps warps, its values resident in shared memory.
template <int kWarps>
__global__ void __launch_bounds__(32 * kWarps, kWarps == 16 ? 2 : 28 / kWarps) dual_clip_resident_kernel(ClipParams P) {
  constexpr int T = 32 * kWarps;
  extern __shared__ __align__(16) float val[];
  __shared__ double part[kWarps * 4];
  __shared__ double sh_inv, sh_lo, sh_hi, sh_c1, sh_c2;
  __shared__ int sh_zi, sh_mode;                       // 0: no quantizer (bounds coincide), 1: integer clip, 2: general
  __shared__ float ext[2][kWarps];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int d = blockIdx.x, n = int(P.n);
  const float* col = P.x + d;

  float mxf = -INFINITY, mnf = INFINITY;
#pragma unroll 8
  for (int t = tid; t < n; t += T) {
    const float v = __ldg(col + int64_t(t) * P.ldx);
    val[t] = v;
    mxf = fmaxf(mxf, v);
    mnf = fminf(mnf, v);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mxf = fmaxf(mxf, __shfl_xor_sync(0xffffffffu, mxf, o));
    mnf = fminf(mnf, __shfl_xor_sync(0xffffffffu, mnf, o));
  }
  if (lane == 0) { ext[0][warp] = mxf; ext[1][warp] = mnf; }
  __syncthreads();
  // warp 0 keeps the channel's state; even lanes the upper factor, odd lanes the lower one (every pair of lanes holds the
  // same numbers, so that the whole warp goes through one update)
  const bool upper = (lane & 1) == 0;
  double bound = 0.0, other = 0.0, sg = 0.0, mine = 0.0, a = P.alpha0, m = 0.0, v = 0.0, b1t = 1.0, b2t = 1.0;
  double s = 0.0, z = 0.0, zc = 0.0, big = 0.0, loss_first = 0.0;
  if (warp == 0) {
    for (int w = 0; w < kWarps; ++w) { mxf = fmaxf(mxf, ext[0][w]); mnf = fminf(mnf, ext[1][w]); }
    mine = upper ? double(mxf) : double(mnf);
    big = fmax(fabs(double(mxf)), fabs(double(mnf)));
  }
  const uint32_t qi = uint32_t(P.Q);
  const double inv_q = 1.0 / P.Q;
  for (int it = 0; it <= P.iters; ++it) {
    // the channel's quantizer for this step (Eq. 6 on the bounds of Eqs. 18-19)
    if (warp == 0) {
      sg = sigmoid(a);
      bound = mine * sg;
      other = __shfl_xor_sync(0xffffffffu, bound, 1);
      const double up = upper ? bound : other, low = upper ? other : bound;
      s = (up - low) * inv_q;
      const double inv = 1.0 / s;
      zc = -low * inv;
      z = rint(zc);
      if (lane == 0) {
        sh_inv = inv;
        sh_lo = -z;
        sh_hi = P.Q - z;
        const bool small = big * inv < 1073741824.0 && fabs(z) < 1073741824.0;
        sh_zi = small ? int(z) : 0;
        sh_mode = !(s > 0.0) ? 0 : small ? 1 : 2;
      }
    }
    if (it == P.iters && P.loss == nullptr) break;     // the pass after the last update serves the objective alone
    if (kWarps > 1) __syncthreads(); else __syncwarp();
    const double inv = sh_inv, lo = sh_lo, hi = sh_hi;
    const int zi = sh_zi, mode = sh_mode;
    ClipSums acc{0.0, 0.0, 0.0, 0.0};
    // a channel whose bounds coincide (a constant channel, or extremes of 0) has no quantizer to learn: its sums stay
    // 0, its factors keep their starting value and the contracted extremes are returned as they are
    double in2b = 0.0;
    if (mode == 1) {
      for (int t = tid * 4; t + 3 < n; t += T * 4) {
        const float4 p = *reinterpret_cast<const float4*>(val + t);
        const float x[4] = {p.x, p.y, p.z, p.w};
        clip_values<true, 4>(x, inv, lo, hi, zi, qi, acc, in2b);
      }
      if (tid < (n & 3)) {
        const float x[1] = {val[(n & ~3) + tid]};
        clip_values<true, 1>(x, inv, lo, hi, zi, qi, acc, in2b);
      }
    } else if (mode == 2) {
      for (int t = tid; t < n; t += T) {
        const float x[1] = {val[t]};
        clip_values<false, 1>(x, inv, lo, hi, zi, qi, acc, in2b);
      }
    }
    acc.in2 += in2b;
    double total = warp_sum4(acc, lane);
    if (kWarps > 1) {
      if (lane < 4) part[warp * 4 + lane] = total;
      if (warp == kWarps - 1) {                        // Adam's bias corrections of this step, off warp 0's chain
        b1t *= P.beta1;
        b2t *= P.beta2;
        if (lane == 0) { sh_c1 = P.lr / (1.0 - b1t); sh_c2 = 1.0 / (1.0 - b2t); }
      }
      __syncthreads();
    }
    if (warp == 0) {
      double c1, c2;
      if (kWarps > 1) {
        total = part[lane & (kWarps * 4 - 1)];
        if (kWarps == 16) total += part[lane + 32];
#pragma unroll
        for (int o = 4; o < kWarps * 4 && o < 32; o <<= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
        c1 = sh_c1;
        c2 = sh_c2;
      } else {
        b1t *= P.beta1;
        b2t *= P.beta2;
        c1 = P.lr / (1.0 - b1t);
        c2 = 1.0 / (1.0 - b2t);
      }
      acc.in2 = __shfl_sync(0xffffffffu, total, 0);
      acc.low = __shfl_sync(0xffffffffu, total, 1);
      acc.high = __shfl_sync(0xffffffffu, total, 2);
      acc.out2 = __shfl_sync(0xffffffffu, total, 3);
      const bool live = s > 0.0;
      const double loss = live ? s * s * (acc.in2 + acc.out2) : 0.0;
      if (it == 0) loss_first = loss;
      if (it == P.iters) {
        if (lane == 0) { P.loss[d] = loss_first; P.loss[P.D + d] = loss; }
      } else {
        const double dL_ds = live ? 2.0 * s * (acc.in2 + (zc - z) * acc.low + (P.Q - z + zc) * acc.high) : 0.0;
        const double dL_dl = live ? 2.0 * s * (acc.low + acc.high) : 0.0;
        const double g = (upper ? dL_ds * inv_q : dL_dl - dL_ds * inv_q) * mine * sg * (1.0 - sg);
        m = P.beta1 * m + (1.0 - P.beta1) * g;
        v = P.beta2 * v + (1.0 - P.beta2) * g * g;
        a -= c1 * m / (sqrt(c2 * v) + P.eps);
      }
    }
  }
  if (tid == 0) {
    P.x_up[d] = float(bound);
    P.x_low[d] = float(other);
  }
}

template <int kWarps>
repq_status launch_resident(const ClipParams& P, cudaStream_t st) {
  const size_t smem = size_t(P.n) * sizeof(float);
  REPQ_TRY(allow_smem<dual_clip_resident_kernel<kWarps>>(kMaxResident * 4));
  dual_clip_resident_kernel<kWarps><<<P.D, 32 * kWarps, smem, st>>>(P);
  REPQ_CUDA(cudaGetLastError());
  return REPQ_OK;
}

// ---- sorted form

__device__ __forceinline__ void order(float& a, float& b) {
  const float t = fminf(a, b);
  b = fmaxf(a, b);
  a = t;
}

// Ascending sort of the n values (n8 with the infinities that fill the last group of eight).  Every merge of two sorted runs starts by
// comparing mirrored positions, so that each comparison leaves the smaller value at the lower index and positions past n8 act
// as infinities that never move: any n is sorted in place.  A thread takes eight values through up to three steps at a time.
template <int T>
__device__ __forceinline__ void sort_channel(float* val, int n8, int tid) {
  auto sync = [] { if (T > 32) __syncthreads(); else __syncwarp(); };
  auto load8 = [&](int i, float (&v)[8]) {
    const float4 a = *reinterpret_cast<const float4*>(val + i), b = *reinterpret_cast<const float4*>(val + i + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  };
  auto store8 = [&](int i, const float (&v)[8]) {
    *reinterpret_cast<float4*>(val + i) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4*>(val + i + 4) = make_float4(v[4], v[5], v[6], v[7]);
  };
  auto steps = [](float (&v)[8], int first) {            // distances 4, 2, 1 from `first` on
    if (first >= 4) { order(v[0], v[4]); order(v[1], v[5]); order(v[2], v[6]); order(v[3], v[7]); }
    if (first >= 2) { order(v[0], v[2]); order(v[1], v[3]); order(v[4], v[6]); order(v[5], v[7]); }
    order(v[0], v[1]); order(v[2], v[3]); order(v[4], v[5]); order(v[6], v[7]);
  };
  const int groups = n8 >> 3;
  for (int t = tid; t < groups; t += T) {                // runs of eight
    float v[8];
    load8(8 * t, v);
    order(v[0], v[1]); order(v[2], v[3]); order(v[4], v[5]); order(v[6], v[7]);
    order(v[0], v[3]); order(v[1], v[2]); order(v[4], v[7]); order(v[5], v[6]);
    order(v[0], v[1]); order(v[2], v[3]); order(v[4], v[5]); order(v[6], v[7]);
    order(v[0], v[7]); order(v[1], v[6]); order(v[2], v[5]); order(v[3], v[4]);
    steps(v, 2);
    store8(8 * t, v);
  }
  for (int k = 4; (8 << (k - 4)) < n8; ++k) {            // runs of 2^k out of runs of 2^(k-1)
    sync();
    {
      // mirrored step and distances 2^(k-2), 2^(k-3): the upper four of a thread's values come from the mirrored offset
      const int lh = k - 3, h = 1 << lh;
      for (int t = tid; t < ((n8 + (1 << k) - 1) >> k) << lh; t += T) {
        const int base = (t >> lh) << k, o = t & (h - 1);
        float v[8];
        int i[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          i[j] = base + j * h + (j < 4 ? o : h - 1 - o);
          v[j] = i[j] < n8 ? val[i[j]] : INFINITY;
        }
        order(v[0], v[7]); order(v[1], v[6]); order(v[2], v[5]); order(v[3], v[4]);
        steps(v, 2);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (i[j] < n8) val[i[j]] = v[j];
      }
    }
    int lt = k - 4;                                      // log2 of the next distance
    for (; lt >= 3; lt -= 3) {
      sync();
      const int lh = lt - 2, h = 1 << lh;
      for (int t = tid; t < ((n8 + (8 << lh) - 1) >> (lh + 3)) << lh; t += T) {
        const int base = ((t >> lh) << (lh + 3)) + (t & (h - 1));
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = base + j * h < n8 ? val[base + j * h] : INFINITY;
        steps(v, 4);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (base + j * h < n8) val[base + j * h] = v[j];
      }
    }
    if (lt >= 0) {
      sync();
      for (int t = tid; t < groups; t += T) {
        float v[8];
        load8(8 * t, v);
        steps(v, 1 << lt);
        store8(8 * t, v);
      }
    }
  }
  sync();
}

// Bucket of a value, monotone in x (every operation rounds once): equal parts of the channel's range or, `spread`, of the range of
// u / (1 + |u|), u = (x - low) scale, whose parts grow with the distance from `low` like the density of a long tail falls.
struct Buckets {
  float low, scale;
  int last;
  bool spread;
  __device__ __forceinline__ int of(float x) const {
    float u = __fmul_rn(__fsub_rn(x, low), scale);
    if (spread) {
      const float half = 0.5f * float(last + 1);
      u = __fmaf_rn(copysignf(__fsub_rn(1.f, __frcp_rn(__fadd_rn(1.f, fabsf(u)))), u), half, half);
    }
    return max(0, min(last, __float2int_rz(u)));
  }
};

// One channel per CTA of kWarps warps.  All of them load the channel's values, sort them (by bucket, then by rank inside
// the bucket; where values crowd in few buckets, by buckets that widen with the distance from the middle, and where they crowd there too,
// as values that repeat do, by merging) and form prefix sums of every fourth; the first
// warp then runs the optimisation alone, since a step no longer passes over the values: those of code q lie between two edges of
// the sorted order, and with y = x - pivot, kappa_q = q - z - pivot/s,
//     sum over a code of (q - z - x/s)^2 = n kappa^2 - 2 (kappa/s) sum y + (1/s^2) sum y^2
// from counts and prefix sums at the edges.  The prefix sums run outwards from the pivot, the channel's median, in both directions, so
// that the sums between two inner edges never contain a tail; what cancels is kappa^2 per value against at most 1/4.  |kappa| is at
// most Q where the median lies inside the clip, and about Q (1 + 1 / sigmoid(alpha)) where it does not and any value does.  The three
// sums that steer a step, float64 against 80-bit floats, 6304 values, alpha from 6 down to -3: 1e-13 of the sum of squares inside the clip
// (one value at -3000 among normal ones 9e-14, normal values 2e-14; summed from the least value on 1e-11 and 3e-13; value by value 1e-16),
// where the squares inside are a part of the gradient.  Only the float32 bounds, 6e-8 apart, leave the kernel with it.
// An edge is the smallest float whose rounded quotient reaches the next code, so every value has the code that its own quotient
// rounds to.
template <int kWarps>
__global__ void __launch_bounds__(32 * kWarps, kWarps == 16 ? 2 : 28 / kWarps) dual_clip_sorted_kernel(ClipParams P, int bucket_shift) {
  constexpr int T = 32 * kWarps;
  extern __shared__ __align__(16) float smem[];
  __shared__ float ext[2][kWarps];
  __shared__ int part_n[kWarps];
  __shared__ double2 part[2][kWarps];
  __shared__ double learned[2];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int d = blockIdx.x, n = int(P.n), n8 = (n + 7) & ~7;
  const int middle = (n >> 1) & ~3;                      // the prefix sums start here
  // values (raw, then sorted), values by bucket (later the prefix sums, 16 bytes per four values), starts of the buckets
  float* val = smem;
  float* by_bucket = smem + n8;
  double2* pre = reinterpret_cast<double2*>(by_bucket);
  int* start = reinterpret_cast<int*>(by_bucket + n8 + 4);
  const int nb = sorted_buckets(n, bucket_shift), blocks = (n >> 2) + 1;
  const float* col = P.x + d;
  auto sync = [] { if (kWarps > 1) __syncthreads(); else __syncwarp(); };
  auto bar = [] { asm volatile("bar.sync 1, %0;" ::"n"(T) : "memory"); };   // the same, from more than one place

  float mxf = -INFINITY, mnf = INFINITY;
  bool odd_value = false;                                // an infinity or a NaN: no order, and no finite sums either
#pragma unroll 8
  for (int t = tid; t < n; t += T) {
    const float v = __ldg(col + int64_t(t) * P.ldx);
    val[t] = v;
    mxf = fmaxf(mxf, v);
    mnf = fminf(mnf, v);
    odd_value = odd_value || !(fabsf(v) < INFINITY);
  }
  if (tid < n8 - n) val[n + tid] = INFINITY;
  for (int i = tid; i <= nb; i += T) start[i] = 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mxf = fmaxf(mxf, __shfl_xor_sync(0xffffffffu, mxf, o));
    mnf = fminf(mnf, __shfl_xor_sync(0xffffffffu, mnf, o));
  }
  if (lane == 0) { ext[0][warp] = mxf; ext[1][warp] = mnf; }
  const bool finite = __syncthreads_or(odd_value) == 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) { mxf = fmaxf(mxf, ext[0][w]); mnf = fminf(mnf, ext[1][w]); }
  Buckets B{mnf, float(nb) / (mxf - mnf), nb - 1, false};
  if (!(B.scale < INFINITY)) B.scale = 0.f;              // one value, or a range below the normal numbers: a single bucket

  double pivot = 0.0;
  if (finite) {
    // counts of the buckets; where they are crowded, again in spread ones around the middle of 32 of the values
    const int run_b = (nb + T - 1) / T, first_b = min(nb, tid * run_b), last_b = min(nb, first_b + run_b);
    bool crowded = false;
    int own = 0;
    for (;;) {
      for (int t = tid; t < n; t += T) atomicAdd(&start[B.of(val[t])], 1);
      sync();
      own = 0;
      crowded = false;
      for (int b = first_b; b < last_b; ++b) { own += start[b]; crowded = crowded || start[b] > crowd(bucket_shift); }
      crowded = __syncthreads_or(crowded) != 0;
      if (!crowded || B.spread) break;
      const float w = val[int(int64_t(n) * lane >> 5)];
      int rank = 0;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float o = __shfl_sync(0xffffffffu, w, i);
        rank += o < w || (o == w && i < lane) ? 1 : 0;
      }
      auto ranked = [&](int r) { return __shfl_sync(0xffffffffu, w, __ffs(__ballot_sync(0xffffffffu, rank == r)) - 1); };
      const float middle_w = ranked(16), scale = 2.f / (ranked(24) - ranked(8));
      if (!(scale < INFINITY)) break;
      B = Buckets{middle_w, scale, nb - 1, true};
      for (int i = tid; i <= nb; i += T) start[i] = 0;
      sync();
    }
    {
      // inclusive scan of the counts, a run of buckets per thread
      int sum = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, sum, o);
        if (lane >= o) sum += t;
      }
      if (lane == 31) part_n[warp] = sum;
      sync();
      int at = sum - own;
      for (int w = 0; w < warp; ++w) at += part_n[w];
      for (int b = first_b; b < last_b; ++b) start[b] = at += start[b];
      if (tid == 0) start[nb] = n;
    }
    sync();
    for (int t = tid; t < n; t += T) {                   // leaves every bucket's start behind
      const float v = val[t];
      const int at = atomicSub(&start[B.of(v)], 1) - 1;
      by_bucket[at] = v;
    }
    sync();
    if (crowded) {
      sort_channel<T>(val, n8, tid);
    } else {
      for (int t = tid; t < n; t += T) {
        const float v = by_bucket[t];
        const int b = B.of(v), first = start[b], last = start[b + 1];
        int rank = first;
        for (int i = first; i < last; ++i) {
          const float w = by_bucket[i];
          rank += (w < v || (w == v && i < t)) ? 1 : 0;
        }
        val[rank] = v;
      }
      sync();
    }
    pivot = double(val[n >> 1]);
    // prefix sums at every fourth value, those below `middle` negative: a run of blocks of four values per thread, summed twice
    // (total, then block by block beyond the threads nearer to the middle)
    const int run = (blocks + T - 1) / T, first = min(blocks, tid * run), last = min(blocks, first + run);
    const int up0 = max(first, middle >> 2), down1 = min(last, middle >> 2);
    auto add_block = [&](int b, double2& t) {
      for (int i = 4 * b; i < min(n, 4 * b + 4); ++i) {
        const double y = double(val[i]) - pivot;
        t.x += y;
        t.y = fma(y, y, t.y);
      }
    };
    double2 up = make_double2(0.0, 0.0), down = up;
    for (int b = up0; b < last; ++b) add_block(b, up);
    for (int b = down1 - 1; b >= first; --b) add_block(b, down);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double ux = __shfl_up_sync(0xffffffffu, up.x, o), uy = __shfl_up_sync(0xffffffffu, up.y, o);
      const double dx = __shfl_down_sync(0xffffffffu, down.x, o), dy = __shfl_down_sync(0xffffffffu, down.y, o);
      if (lane >= o) { up.x += ux; up.y += uy; }
      if (lane + o < 32) { down.x += dx; down.y += dy; }
    }
    if (lane == 31) part[0][warp] = up;
    if (lane == 0) part[1][warp] = down;
    sync();
    up = make_double2(__shfl_up_sync(0xffffffffu, up.x, 1), __shfl_up_sync(0xffffffffu, up.y, 1));
    down = make_double2(__shfl_down_sync(0xffffffffu, down.x, 1), __shfl_down_sync(0xffffffffu, down.y, 1));
    if (lane == 0) up = make_double2(0.0, 0.0);
    if (lane == 31) down = make_double2(0.0, 0.0);
    for (int w = 0; w < warp; ++w) { up.x += part[0][w].x; up.y += part[0][w].y; }
    for (int w = kWarps - 1; w > warp; --w) { down.x += part[1][w].x; down.y += part[1][w].y; }
    for (int b = up0; b < last; ++b) {
      pre[b] = up;
      add_block(b, up);
    }
    for (int b = down1 - 1; b >= first; --b) {
      add_block(b, down);
      pre[b] = make_double2(-down.x, -down.y);
    }
    sync();
  }
  // The objective goes to the caller in float64: value by value, as in the other form, by all warps.
  const double inv_q = 1.0 / P.Q;
  auto objective = [&](double up, double low, double* out) {
    const double s = (up - low) * inv_q, inv = 1.0 / s, z = rint(-low * inv), lo = -z, hi = P.Q - z;
    double sum[2] = {0.0, 0.0};
#pragma unroll 4
    for (int i = 2 * tid; i < n8; i += 2 * T) {
      const float2 x2 = *reinterpret_cast<const float2*>(val + i);
      const double u0 = double(x2.x) * inv, u1 = double(x2.y) * inv;
      const double d0 = fmin(fmax(rint(u0), lo), hi) - u0, d1 = fmin(fmax(rint(u1), lo), hi) - u1;
      sum[0] = i < n ? fma(d0, d0, sum[0]) : sum[0];
      sum[1] = i + 1 < n ? fma(d1, d1, sum[1]) : sum[1];
    }
    sum[0] += sum[1];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], o);
    if (kWarps > 1) {
      if (lane == 0) part[0][warp].x = sum[0];
      bar();
      if (tid == 0) {
        for (int w = 1; w < kWarps; ++w) sum[0] += part[0][w].x;
      }
    }
    // (bounds that coincide: no quantizer, no objective)
    if (tid == 0) *out = !(s > 0.0) ? 0.0 : finite ? s * s * sum[0] : CUDART_NAN;
  };
  if (P.loss != nullptr) {
    const double sg = sigmoid(P.alpha0);
    objective(__dmul_rn(double(mxf), sg), __dmul_rn(double(mnf), sg), P.loss + d);   // (equal extremes: equal bounds, both rounded)
  }

  // ---- the optimisation: even lanes carry the upper factor, odd lanes the lower one (every pair of lanes holds the same numbers)
  // (The other warps wait in a branch that ends there: with a common barrier behind an `if (warp == 0)` a step took 4.6 us, not 1.15.)
  if (warp != 0) {
    if (P.loss != nullptr) {
      bar();
      objective(learned[0], learned[1], P.loss + P.D + d);
    }
    return;
  }
  const int top_lane = int(P.Q) + 1;                     // a lane per edge: below code 0, between the codes, above code Q
  struct Below { double c, y, yy; };                     // number of the values below an edge, sums of y and y^2 from the middle to it
  auto sums_to = [&](int c) {
    // from the prefix sums on the middle's side of the edge, and up to three values more
    const bool up = c >= middle;
    const double2 t = pre[(up ? c : c + 3) >> 2];
    const float4 q = *reinterpret_cast<const float4*>(val + max(0, min((up ? c : c - 1) & ~3, n8 - 4)));
    const int r = (up ? c : -c) & 3;
    const float f0 = up ? q.x : q.w, f1 = up ? q.y : q.z, f2 = up ? q.z : q.y;
    const double y0 = r > 0 ? double(f0) - pivot : 0.0, y1 = r > 1 ? double(f1) - pivot : 0.0, y2 = r > 2 ? double(f2) - pivot : 0.0;
    const double sign = up ? 1.0 : -1.0;
    return Below{double(c), fma(sign, (y0 + y1) + y2, t.x), fma(sign, fma(y0, y0, y1 * y1) + y2 * y2, t.y)};
  };
  Below none{0.0, 0.0, 0.0}, all = none;
  if (finite) { none = sums_to(0); all = sums_to(n); }

  const bool upper = (lane & 1) == 0;
  const double mine = upper ? double(mxf) : double(mnf);
  double bound = 0.0, other = 0.0, a = P.alpha0, m = 0.0, v = 0.0, b1t = 1.0, b2t = 1.0, c1s = 0.0, c2s = 0.0;
  for (int it = 0; it <= P.iters; ++it) {
    // the channel's quantizer for this step (Eq. 6 on the bounds of Eqs. 18-19)
    const double sg = sigmoid(a);
    bound = mine * sg;
    other = __shfl_xor_sync(0xffffffffu, bound, 1);
    if (it == P.iters) break;
    if ((it & 31) == 0) {                                // Adam's bias corrections of the next 32 steps, one per lane
      double p1 = 1.0, p2 = 1.0;
#pragma unroll 1
      for (int i = 0; i < 32; ++i) {
        b1t *= P.beta1;
        b2t *= P.beta2;
        if (i == lane) { p1 = b1t; p2 = b2t; }
      }
      c1s = P.lr / (1.0 - p1);
      c2s = 1.0 / (1.0 - p2);
    }
    const double up = upper ? bound : other, low = upper ? other : bound;
    const double s = (up - low) * inv_q, inv = 1.0 / s, zc = -low * inv, z = rint(zc), lo = -z;
    // a channel whose bounds coincide (a constant channel, or extremes of 0) has no quantizer to learn: its sums stay
    // 0, its factors keep their starting value and the contracted extremes are returned as they are
    const bool live = s > 0.0;
    double in2 = 0.0, sum_low = 0.0, sum_high = 0.0;
    if (live && finite) {
      const double shift_p = pivot * inv, k_lo = lo - shift_p, k_hi = (P.Q - z) - shift_p;
      const double k = lo + double(lane);                // first code at or above the lane's edge
      float edge = float((k - 0.5) * s);
      const int bucket = B.of(edge);                     // (no value of a later bucket is below the next float either)
      int first = start[bucket], last = start[bucket + 1];
      if (rint(double(edge) * inv) < k) edge = nextafterf(edge, INFINITY);
      while (first < last) {
        const int mid = (first + last) >> 1;
        if (val[mid] < edge) first = mid + 1; else last = mid;
      }
      const Below t = sums_to(first);
      // the code between the lane's edge and the one before; its squares without those of y, which add up over the codes
      const double kappa = k_lo + double(lane - 1), inv2 = inv * inv;
      const double dc = t.c - __shfl_up_sync(0xffffffffu, t.c, 1), dy = t.y - __shfl_up_sync(0xffffffffu, t.y, 1);
      if (lane > 0 && lane <= top_lane) in2 = kappa * (kappa * dc - 2.0 * inv * dy);
      // what is clipped, beyond the first and the last edge
      const bool top = lane == top_lane;
      const double c = top ? all.c - t.c : t.c, y = top ? all.y - t.y : t.y - none.y, end = top ? k_hi : k_lo;
      const double linear = end * c - inv * y;
      if (top) in2 = fma(inv2, t.yy, in2);
      if (lane == 0) in2 = -inv2 * t.yy;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) in2 += __shfl_xor_sync(0xffffffffu, in2, o);
      sum_low = __shfl_sync(0xffffffffu, linear, 0);
      sum_high = __shfl_sync(0xffffffffu, linear, top_lane);
    } else if (live) {
      in2 = sum_low = sum_high = CUDART_NAN;
    }
    const double dL_ds = live ? 2.0 * s * (in2 + (zc - z) * sum_low + (P.Q - z + zc) * sum_high) : 0.0;
    const double dL_dl = live ? 2.0 * s * (sum_low + sum_high) : 0.0;
    const double g = (upper ? dL_ds * inv_q : dL_dl - dL_ds * inv_q) * (mine * sg * (1.0 - sg));
    m = P.beta1 * m + (1.0 - P.beta1) * g;
    v = P.beta2 * v + (1.0 - P.beta2) * g * g;
    const double c1 = __shfl_sync(0xffffffffu, c1s, it & 31), c2 = __shfl_sync(0xffffffffu, c2s, it & 31);
    a -= c1 * m / (sqrt(c2 * v) + P.eps);
  }
  if (lane == 0) {
    P.x_up[d] = float(bound);
    P.x_low[d] = float(other);
    learned[0] = bound;
    learned[1] = other;
  }
  if (P.loss != nullptr) {
    bar();
    objective(learned[0], learned[1], P.loss + P.D + d);
  }
}

template <int kWarps>
repq_status launch_sorted(const ClipParams& P, int shift, cudaStream_t st) {
  REPQ_TRY((allow_smem<dual_clip_sorted_kernel<kWarps>>(int(sorted_bytes(kMaxSorted, 1)))));
  dual_clip_sorted_kernel<kWarps><<<P.D, 32 * kWarps, sorted_bytes(P.n, shift), st>>>(P, shift);
  REPQ_CUDA(cudaGetLastError());
  return REPQ_OK;
}

// Full-precision normalisation of the calibration batch (Eq. 9; mean-free variant for RMS): the activations the
// clipping factors are learned on.  One CTA per row at a time, mean and centred variance in float32 with a
// float64 block reduction, float32 output.  Calibration-time only: the inference path never forms X'.
template <typename T>
__global__ void __launch_bounds__(256) layernorm_kernel(const T* __restrict__ x, int64_t rows, int D, int64_t ldx,
                                                        const float* __restrict__ gamma, const float* __restrict__ beta,
                                                        float eps, int rms, float* __restrict__ y, int64_t ldy) {
  __shared__ double red[8];
  __shared__ float bc;
  auto block_sum = [&](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();                               // the previous use of red / bc is over
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int i = 0; i < 8; ++i) t += red[i];
      bc = float(t / double(D));
    }
    __syncthreads();
    return bc;
  };
  auto ld = [](const T* p) {
    if constexpr (sizeof(T) == 2) return __bfloat162float(*p);
    else return float(*p);
  };
  for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
    const T* xr = x + r * ldx;
    double acc = 0.0;
    if (!rms)
      for (int c = threadIdx.x; c < D; c += 256) acc += double(ld(xr + c));
    const float mu = rms ? 0.f : block_sum(acc);
    acc = 0.0;
    for (int c = threadIdx.x; c < D; c += 256) {
      const float dlt = ld(xr + c) - mu;
      acc += double(dlt) * double(dlt);
    }
    const float rstd = rsqrtf(block_sum(acc) + eps);
    for (int c = threadIdx.x; c < D; c += 256)
      y[r * ldy + c] = fmaf((ld(xr + c) - mu) * rstd, __ldg(gamma + c), __ldg(beta + c));
  }
}

}  // namespace
}  // namespace repq

using namespace repq;

extern "C" repq_status repq_layernorm(const void* x, int x_dtype, int64_t rows, int D, int64_t ldx, const float* gamma,
                                      const float* beta, float eps, int norm_kind, float* y, int64_t ldy, void* stream) {
  REPQ_REQUIRE(rows >= 0 && D > 0 && ldx >= D && ldy >= D, REPQ_INVALID_ARG, "layernorm: bad sizes");
  if (rows == 0) return REPQ_OK;
  REPQ_REQUIRE(x && gamma && beta && y, REPQ_INVALID_ARG, "layernorm: NULL pointer");
  REPQ_REQUIRE(x_dtype == REPQ_F32 || x_dtype == REPQ_BF16, REPQ_INVALID_ARG, "layernorm: x_dtype must be REPQ_F32 or REPQ_BF16");
  REPQ_REQUIRE(norm_kind == REPQ_NORM_LAYERNORM || norm_kind == REPQ_NORM_RMS, REPQ_INVALID_ARG, "layernorm: unknown norm_kind");
  REPQ_REQUIRE(eps >= 0.f, REPQ_INVALID_ARG, "layernorm: eps must be non-negative");
  const int grid = int(rows < 4096 ? rows : 4096);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int rms = norm_kind == REPQ_NORM_RMS;
  if (x_dtype == REPQ_F32)
    layernorm_kernel<float><<<grid, 256, 0, st>>>(static_cast<const float*>(x), rows, D, ldx, gamma, beta, eps, rms, y, ldy);
  else
    layernorm_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(x), rows, D, ldx, gamma, beta, eps, rms, y, ldy);
  REPQ_CUDA(cudaGetLastError());
  note_launch();
  return REPQ_OK;
}

extern "C" repq_status repq_dual_clip(const float* x, int64_t n, int D, int64_t ldx, int bits, int iters, float lr,
                                      float alpha0, float* x_low, float* x_up, double* loss, void* stream) {
  REPQ_REQUIRE(x && x_low && x_up, REPQ_INVALID_ARG, "dual_clip: NULL pointer");
  REPQ_REQUIRE(n > 0 && D > 0 && ldx >= D, REPQ_INVALID_ARG, "dual_clip: n and D must be positive, ldx >= D");
  REPQ_REQUIRE(bits == 4 || bits == 6 || bits == 8, REPQ_INVALID_ARG, "dual_clip: bits must be 4, 6 or 8");
  REPQ_REQUIRE(iters >= 0 && iters <= 100000 && lr > 0.f, REPQ_INVALID_ARG, "dual_clip: iters must be 0..100000 and lr positive");
  ClipParams P{};
  P.x = x; P.n = n; P.ldx = ldx; P.D = D;
  P.Q = double((1 << bits) - 1);
  P.iters = iters; P.lr = double(lr); P.alpha0 = double(alpha0);
  P.beta1 = 0.9; P.beta2 = 0.999; P.eps = 1e-8;
  P.x_low = x_low; P.x_up = x_up; P.loss = loss;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (n <= kMaxResident) {
    const int sms = sm_count();
    const int share = (D + sms - 1) / sms;                                  // channels of an SM
    // channels that an SM holds at a time, at so many bytes each, and its turns
    auto held = [&](size_t bytes) { return std::max(1, int(228 * 1024 / int64_t(bytes + 1536))); };
    auto turns = [&](int shift) { return (share + held(sorted_bytes(n, shift)) - 1) / held(sorted_bytes(n, shift)); };
    const int held_resident = int(int64_t(kMaxResident) * 4 / (n * 4 + 1024));
    // Sorted form: 16 codes (a lane per edge; 64 and 256 codes were slower than passes over the values, 1182 x 2048 430 against 389
    // and 6304 x 384 1360 against 346), no long queue of channels behind one another (16384 x 4096, 28 turns: 4600 against 4566) and
    // enough steps to pay for the sort: a step of all channels that an SM holds at a time takes 1.1 us against 1.3 to 2.9, the sort 35
    // to 70 us a turn (6304 x 384 46 against 11, and from the 20th step on, or the 28th with outliers, it is ahead); beyond one
    // turn the passes of three times as many channels run side by side (12608 x 768 ahead from the 39th or 52nd step, 20000 x 1024 the 41st or 54th).
    const bool sorted = bits == 4 && n <= kMaxSorted && turns(3) <= 16 && iters >= (turns(3) > 1 ? 72 : 32);
    int shift = 3;                                          // as many buckets as do not cost a further turn
    while (shift > 1 && turns(shift - 1) <= turns(3)) --shift;
    // warps per channel: about 28 warps on every SM over all channels, and as many where shared memory limits the
    // channels an SM holds at a time
    const int want = std::max(28 * sms / D, 24 / std::max(1, sorted ? held(sorted_bytes(n, shift)) : held_resident));
    auto launch = [&](auto warps) {
      constexpr int kWarps = decltype(warps)::value;
      return sorted ? launch_sorted<kWarps>(P, shift, st) : launch_resident<kWarps>(P, st);
    };
    if (want >= 16) REPQ_TRY(launch(std::integral_constant<int, 16>()));
    else if (want >= 8) REPQ_TRY(launch(std::integral_constant<int, 8>()));
    else if (want >= 4) REPQ_TRY(launch(std::integral_constant<int, 4>()));
    else if (want >= 2) REPQ_TRY(launch(std::integral_constant<int, 2>()));
    else REPQ_TRY(launch(std::integral_constant<int, 1>()));
  } else {
    const int grid = (D + kCh - 1) / kCh;
    dual_clip_kernel<<<grid, kThreads, 0, st>>>(P);
    REPQ_CUDA(cudaGetLastError());
  }
  note_launch();
  return REPQ_OK;
}
