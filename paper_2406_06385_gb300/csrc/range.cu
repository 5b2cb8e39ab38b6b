// Range setting (App. B) and the downcast of the frozen base (Eq. 6 / Eq. 7): the passes over
// the pretrained weights that prepare a layer.  Min-max and the downcast are bound by HBM (the
// fp32 weights are read once); the L^p search evaluates every candidate scale on every weight
// and is bound by the FP32 and ALU pipes.
#include <cuda_runtime.h>
#include <cstdint>

#include "kernels.h"
#include "quant.cuh"

namespace lrqat {
namespace {

constexpr int kThreads = 256;
constexpr float kMagic = 12582912.0f;   // 1.5 * 2^23: adding it rounds |x| <= 2^22 half to even

// ------------------------------------------------------------ range setting --
// Min and max over one (row, group) segment of `seg` values (a multiple of 128, 16-byte
// aligned), spread over `step` threads of which this is number `t`: 16-byte loads, four in
// flight.  (One 4-byte load per thread and iteration read a 5120 x 5120 layer in 51.1 us, this
// takes 15.5 us.)
__device__ __forceinline__ void segment_min_max(const float* __restrict__ src, int seg, int t, int step, float& lo,
                                                float& hi) {
  const float4* v4 = reinterpret_cast<const float4*>(src);
  const int n4 = seg / 4;
  auto take = [&](const float4& v) {
    lo = fminf(lo, fminf(fminf(v.x, v.y), fminf(v.z, v.w)));
    hi = fmaxf(hi, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
  };
  int j = t;
  for (; j + 3 * step < n4; j += 4 * step) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = __ldg(v4 + j + u * step);
#pragma unroll
    for (int u = 0; u < 4; ++u) take(v[u]);
  }
  for (; j < n4; j += step) take(__ldg(v4 + j));
}

__device__ __forceinline__ void warp_min_max(float& lo, float& hi) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
}

// max |w| of a segment from its minimum and maximum; 0 when nothing but NaN was seen.
__device__ __forceinline__ float abs_max(float lo, float hi) { return fmaxf(fmaxf(-lo, hi), 0.0f); }

// Symmetric (z0 null): s0 = max|w| / p, 1 for an all-zero segment.  Asymmetric (zero offsets,
// Eq. 1): s0 = (max - min) / (2^b - 1) in fp32 (1 if max == min) and
// z0 = clip(round(n - min / s0), n, p), min / s0 one fp32 division, the rest exact.
__device__ __forceinline__ void write_range(float lo, float hi, int bits, int64_t e, float* __restrict__ s0,
                                            float* __restrict__ z0) {
  if (z0 == nullptr) {
    const float a = abs_max(lo, hi);
    s0[e] = a > 0.0f ? __fdiv_rn(a, static_cast<float>((1 << (bits - 1)) - 1)) : 1.0f;
    return;
  }
  const float span = __fsub_rn(hi, lo);
  const float s = span > 0.0f ? __fdiv_rn(span, static_cast<float>((1 << bits) - 1)) : 1.0f;
  const double n = -static_cast<double>(1 << (bits - 1)), p = static_cast<double>((1 << (bits - 1)) - 1);
  s0[e] = s;
  z0[e] = static_cast<float>(fmin(fmax(rint(n - static_cast<double>(__fdiv_rn(lo, s))), n), p));
}

// WARP: one warp per segment (short segments: a group of 128 is one 16-byte load per lane);
// otherwise one block per segment.
template <bool WARP>
__global__ void __launch_bounds__(kThreads) range_minmax_kernel(const float* __restrict__ W0, int64_t nseg, int seg,
                                                                int bits, float* __restrict__ s0,
                                                                float* __restrict__ z0) {
  float lo = INFINITY, hi = -INFINITY;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (WARP) {
    const int64_t e = static_cast<int64_t>(blockIdx.x) * (kThreads / 32) + warp;
    if (e >= nseg) return;
    segment_min_max(W0 + e * seg, seg, lane, 32, lo, hi);
    warp_min_max(lo, hi);
    if (lane == 0) write_range(lo, hi, bits, e, s0, z0);
    return;
  }
  segment_min_max(W0 + static_cast<int64_t>(blockIdx.x) * seg, seg, threadIdx.x, kThreads, lo, hi);
  warp_min_max(lo, hi);
  __shared__ float warp_lo[kThreads / 32], warp_hi[kThreads / 32];
  if (lane == 0) {
    warp_lo[warp] = lo;
    warp_hi[warp] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
      lo = fminf(lo, warp_lo[w]);
      hi = fmaxf(hi, warp_hi[w]);
    }
    write_range(lo, hi, bits, blockIdx.x, s0, z0);
  }
}

// ---------------------------------------------------------------- L^p search --
// s_j = fl32(s_max (j + 1) / N), j < N, s_max = max|w| / p as in min-max;
// loss_j = sum |w - s_j clip(round(w / s_j), n, p)|^p, w / s_j decided as one fp32 division, the
// error formed with one fused multiply-add, |err|^p by multiplication for integer p, even and
// odd positions summed apart in order.  The smallest loss wins, the smaller j on a tie.
//
// A block takes R segments; thread t evaluates candidate t % N of segment t / N, so nearly every
// lane has a candidate (one block per segment with a thread per candidate left 156 of 256 lanes
// idle at N = 100).  The segments pass through shared memory in chunks of kLpChunk values,
// which all threads of a segment read at the same address (broadcast); rows kLpChunk + 4
// values apart keep the segments that one warp spans on different banks.  Two neighbouring
// values are one packed fp32x2 step but for the clip, which is the saturation of an FMA: with
// r = fl32(1 / s) and W = p - n, t = sat(w r / W - n / W) and t W + n is the clipped quotient (clip and
// round commute, n and p being integers) within 3 W 2^-24 of the IEEE one; the magic add rounds
// it.  Only when one of eight values lies within W 2^-20 of a half-integer are they redone with the
// IEEE division: a margin of 2^-12 for every width sent one warp step in eight there, this one in
// 140 at 4 bits.  Measured on a 5120 x 5120 layer, N = 100, p = 2: 4232 us with a block per segment,
// 962 us with clips by fminf / fmaxf and the fixed margin, 798 us now (the FP32 pipe: 7 operations per
// weight and candidate).
constexpr int kLpPairs = 4;             // packed pairs per step: one near-tie test for all of them
constexpr int kLpChunk = 512;
constexpr int kLpRow = kLpChunk + 4;
constexpr int kLpMaxCand = 256;
constexpr int kLpMaxSegs = 8;
constexpr int kLpMaxThreads = 512;
constexpr int kLpSmemFloats = kLpMaxSegs * kLpRow > kLpMaxSegs * kLpMaxCand * 2 ? kLpMaxSegs * kLpRow
                                                                                : kLpMaxSegs * kLpMaxCand * 2;

// |err|^p of two errors; IP: the integer p (1 .. 8), 0: any other p.  The last product is two
// scalar ones: a packed product whose result is added next was fused with that sum by the
// compiler (the inline mul.rn.f32x2 and add.rn.f32x2 too), and losses that differ in the last
// bit order nearly equal candidates differently (2 of 204,800 rows).
template <int IP>
__device__ __forceinline__ float2 lp_power(float2 err, float p_norm) {
  err = make_float2(fabsf(err.x), fabsf(err.y));
  if (IP == 0) return make_float2(err.x > 0.0f ? powf(err.x, p_norm) : 0.0f, err.y > 0.0f ? powf(err.y, p_norm) : 0.0f);
  float2 t = err;
#pragma unroll
  for (int i = 1; i < IP - 1; ++i) t = __fmul2_rn(t, err);
  return IP > 1 ? make_float2(__fmul_rn(t.x, err.x), __fmul_rn(t.y, err.y)) : t;
}

template <int IP>
__global__ void __launch_bounds__(kLpMaxThreads) range_lp_kernel(const float* __restrict__ W0, int64_t nseg, int seg,
                                                                 int segs_per_block, int bits, float p_norm,
                                                                 int n_cand, float* __restrict__ s0) {
  __shared__ __align__(16) float buf[kLpSmemFloats];   // the chunk, then the losses
  __shared__ float seg_max[kLpMaxSegs];
  const int64_t e0 = static_cast<int64_t>(blockIdx.x) * segs_per_block;
  const int nloc = static_cast<int>(nseg - e0 < segs_per_block ? nseg - e0 : segs_per_block);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const float pmax = static_cast<float>((1 << (bits - 1)) - 1), nmin = -static_cast<float>(1 << (bits - 1));
  for (int g = warp; g < nloc; g += nwarps) {
    float lo = INFINITY, hi = -INFINITY;
    segment_min_max(W0 + (e0 + g) * seg, seg, lane, 32, lo, hi);
    warp_min_max(lo, hi);
    const float a = abs_max(lo, hi);
    if (lane == 0) seg_max[g] = a > 0.0f ? __fdiv_rn(a, pmax) : 1.0f;
  }
  __syncthreads();
  const int g = threadIdx.x / n_cand, j = threadIdx.x % n_cand;
  const bool live = g < nloc;
  const float s = live ? static_cast<float>(static_cast<double>(seg_max[g]) * (j + 1) / n_cand) : 1.0f;
  const float r = __frcp_rn(s), width = pmax - nmin, c = -nmin / width, rw = r / width;
  const float2 s2 = make_float2(-s, -s), width2 = make_float2(width, width);
  const float2 up = make_float2(kMagic + nmin, kMagic + nmin);
  // a scale whose reciprocal overflows or comes near the subnormals takes the division for every value
  const float tie = r < INFINITY && r > 0x1p-100f ? 0.5f - width * 0x1p-20f : -1.0f;
  float2 acc = make_float2(0.0f, 0.0f);
  for (int c0 = 0; c0 < seg; c0 += kLpChunk) {
    const int len = seg - c0 < kLpChunk ? seg - c0 : kLpChunk;   // a multiple of 128
    const int len4 = len / 4;
    for (int i = threadIdx.x; i < nloc * len4; i += blockDim.x) {
      const int gg = i / len4, q = i % len4;
      *reinterpret_cast<float4*>(&buf[gg * kLpRow + 4 * q]) =
          __ldg(reinterpret_cast<const float4*>(W0 + (e0 + gg) * seg + c0) + q);
    }
    __syncthreads();
    if (live) {
      const float4* row = reinterpret_cast<const float4*>(&buf[g * kLpRow]);
      for (int i = 0; i < len4; i += kLpPairs / 2) {
        float2 w[kLpPairs], q[kLpPairs];
        float dmax = 0.0f;
#pragma unroll
        for (int h = 0; h < kLpPairs; h += 2) {
          const float4 w4 = row[i + h / 2];
          w[h] = make_float2(w4.x, w4.y);
          w[h + 1] = make_float2(w4.z, w4.w);
        }
#pragma unroll
        for (int h = 0; h < kLpPairs; ++h) {
          const float2 t = make_float2(__saturatef(__fmaf_rn(w[h].x, rw, c)), __saturatef(__fmaf_rn(w[h].y, rw, c)));
          const float2 m = __fadd2_rn(__ffma2_rn(t, width2, up), make_float2(-kMagic, -kMagic));   // the code
          q[h] = m;
          const float2 d = __ffma2_rn(t, width2, make_float2(nmin - m.x, nmin - m.y));
          dmax = fmaxf(dmax, fmaxf(fabsf(d.x), fabsf(d.y)));
        }
        if (dmax > tie) {
#pragma unroll
          for (int h = 0; h < kLpPairs; ++h)
            q[h] = make_float2(fminf(fmaxf(rintf(__fdiv_rn(w[h].x, s)), nmin), pmax),
                               fminf(fmaxf(rintf(__fdiv_rn(w[h].y, s)), nmin), pmax));
        }
#pragma unroll
        for (int h = 0; h < kLpPairs; ++h) acc = __fadd2_rn(acc, lp_power<IP>(__ffma2_rn(s2, q[h], w[h]), p_norm));
      }
    }
    __syncthreads();
  }
  // the losses and their candidates, 256 per segment (absent ones infinite), and a fixed tree
  // over them per segment
  float* best_loss = buf;
  int* best_j = reinterpret_cast<int*>(buf + kLpMaxSegs * kLpMaxCand);
  for (int i = threadIdx.x; i < nloc * kLpMaxCand; i += blockDim.x) {
    best_loss[i] = INFINITY;
    best_j[i] = i % kLpMaxCand;
  }
  __syncthreads();
  if (live) best_loss[g * kLpMaxCand + j] = acc.x + acc.y;
  __syncthreads();
  for (int gg = warp; gg < nloc; gg += nwarps) {
    float* bl = best_loss + gg * kLpMaxCand;
    int* bj = best_j + gg * kLpMaxCand;
    for (int h = kLpMaxCand / 2; h > 0; h >>= 1) {
      for (int i = lane; i < h; i += 32) {
        const float lo = bl[i + h];
        const int jo = bj[i + h];
        if (lo < bl[i] || (lo == bl[i] && jo < bj[i])) {
          bl[i] = lo;
          bj[i] = jo;
        }
      }
      __syncwarp();
    }
    if (lane == 0) s0[e0 + gg] = static_cast<float>(static_cast<double>(seg_max[gg]) * (bj[0] + 1) / n_cand);
  }
}

// ----------------------------------------------------------------- downcast --
// A block converts kDownCols columns of one row, 8 values per thread (two 16-byte loads), so a
// thread knows its row without a division.  The quotient W0 / s0 is one IEEE fp32 division by
// definition (its rounding decides integers); the integer formats form y = w r with r =
// fl32(1 / s), which lies within |y| 2^-22 of it, and divide only when a value of the eight
// comes close to a rounding boundary.  Measured on a 5120 x 5120 layer, Q4.4: 4 values per
// thread with 64-bit index divisions and IEEE divisions 44.4 us, this 24.0 us.
constexpr int kDownCols = 8 * 128;
constexpr int kDownThreads = 128;

// One value by the definitions (Q-fixed: round(2^f clip(x, n, p)); INT-b: clip(round(x), n, p)).
template <int FMT>
__device__ __forceinline__ int quantize_div(float x, float n, float p, float two_f) {
  if (FMT == FMT_Q8) return __float2int_rn(fminf(fmaxf(x, n), p) * two_f);
  const int c = __float2int_rn(x);
  return min(max(c, static_cast<int>(n)), static_cast<int>(p));
}

// Eight values (f = 0 for INT-b; clip and round commute, n and p being integers).  Scaled, |2^f y|
// <= 128, so the product lies within 2^-14 of the quotient and a value more than 2^-12 away
// from a half-integer rounds like it.
template <int FMT>
__device__ __forceinline__ void quantize8(const float (&w)[8], float s, float n, float p, float two_f, int (&q)[8]) {
  const float r = __frcp_rn(s);
  float y[8], dmax = 0.0f, finite = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float x = w[i] * r;
    finite = __fmaf_rn(x, 0.0f, finite);   // NaN once a product is not finite
    const float v = fminf(fmaxf(x, n), p) * two_f;
    y[i] = __fadd_rn(v, kMagic);
    dmax = fmaxf(dmax, fabsf(v - (y[i] - kMagic)));
  }
  if (dmax > 0.499755859375f || !(finite == 0.0f)) {
#pragma unroll
    for (int i = 0; i < 8; ++i) q[i] = quantize_div<FMT>(__fdiv_rn(w[i], s), n, p, two_f);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) q[i] = __float_as_int(y[i]) - __float_as_int(kMagic);
  }
}

// With zero offsets: round(2^f clip(w / s + z, n, p)) (INT-b: clip(round(w / s + z), n, p)), the
// integer offset added exactly in double precision.
template <int FMT>
__device__ __forceinline__ void quantize8_offset(const float (&w)[8], float s, double z, float n, float p, float two_f,
                                                 int (&q)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const double x = static_cast<double>(__fdiv_rn(w[i], s)) + z;
    if (FMT == FMT_Q8) q[i] = __double2int_rn(fmin(fmax(x, static_cast<double>(n)), static_cast<double>(p)) * two_f);
    else q[i] = min(max(__double2int_rn(x), static_cast<int>(n)), static_cast<int>(p));
  }
}

// Floating-point storage (Sec. 3, the cast choices of phi): Phi0 = cast(fl32(W0 / s0))
// with round-to-nearest-even, no clipping inside phi, FP16 and FP8 saturating at their
// largest finite value.
template <int FMT>
__device__ __forceinline__ uint32_t pack_fp8x2(float lo, float hi) {
  unsigned short r;
  if (FMT == FMT_E4M3) asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  else asm("cvt.rn.satfinite.e5m2x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return r;
}

// Saturating: values beyond 65504 (which round-to-nearest would turn into infinities)
// are clamped to it first.
__device__ __forceinline__ uint32_t pack_sat_f16x2(float lo, float hi) {
  uint32_t r;
  lo = fminf(fmaxf(lo, -65504.0f), 65504.0f);
  hi = fminf(fmaxf(hi, -65504.0f), 65504.0f);
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

template <int FMT>
__global__ void __launch_bounds__(kDownThreads) downcast_kernel(const float* __restrict__ W0,
                                                                const float* __restrict__ s0,
                                                                const float* __restrict__ z0, int64_t k,
                                                                int group_size, int ngroups, float n, float p,
                                                                float two_f, void* __restrict__ out) {
  const int64_t row = blockIdx.x;
  for (int64_t col = (static_cast<int64_t>(blockIdx.y) * kDownThreads + threadIdx.x) * 8; col < k;
       col += static_cast<int64_t>(gridDim.y) * kDownCols) {
    const int64_t e = row * k + col;   // a multiple of 8
    const int64_t sidx = group_size ? row * ngroups + col / group_size : row;
    const float s = s0[sidx];
    const float4 a = __ldg(reinterpret_cast<const float4*>(W0 + e)), b = __ldg(reinterpret_cast<const float4*>(W0 + e) + 1);
    const float w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    if constexpr (FMT == FMT_Q8 || FMT == FMT_I4) {
      int q[8];
      if (z0 == nullptr) quantize8<FMT>(w, s, n, p, two_f, q);
      else quantize8_offset<FMT>(w, s, static_cast<double>(z0[sidx]), n, p, two_f, q);
      if (FMT == FMT_Q8) {
        auto word = [&](int i) {
          return __byte_perm(__byte_perm(q[i], q[i + 1], 0x0040u), __byte_perm(q[i + 2], q[i + 3], 0x0040u), 0x5410u);
        };
        reinterpret_cast<uint2*>(out)[e / 8] = make_uint2(word(0), word(4));
      } else {
        uint32_t word = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) word |= (static_cast<uint32_t>(q[i]) & 0xFu) << (4 * i);
        reinterpret_cast<uint32_t*>(out)[e / 8] = word;
      }
    } else {
      float x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = __fdiv_rn(w[i], s);
      if (FMT == FMT_BF16) {
        reinterpret_cast<uint4*>(out)[e / 8] = make_uint4(pack_rn_bf16x2(x[0], x[1]), pack_rn_bf16x2(x[2], x[3]),
                                                          pack_rn_bf16x2(x[4], x[5]), pack_rn_bf16x2(x[6], x[7]));
      } else if (FMT == FMT_F16) {
        reinterpret_cast<uint4*>(out)[e / 8] = make_uint4(pack_sat_f16x2(x[0], x[1]), pack_sat_f16x2(x[2], x[3]),
                                                          pack_sat_f16x2(x[4], x[5]), pack_sat_f16x2(x[6], x[7]));
      } else {
        reinterpret_cast<uint2*>(out)[e / 8] =
            make_uint2(pack_fp8x2<FMT>(x[0], x[1]) | (pack_fp8x2<FMT>(x[2], x[3]) << 16),
                       pack_fp8x2<FMT>(x[4], x[5]) | (pack_fp8x2<FMT>(x[6], x[7]) << 16));
      }
    }
  }
}

}  // namespace

cudaError_t launch_range_minmax(const float* W0, int64_t m, int64_t k, int group_size, int bits, float* s0, float* z0,
                                cudaStream_t stream) {
  const int seg = group_size ? group_size : static_cast<int>(k);
  const int64_t nseg = m * (k / seg);
  // up to 1024 values a warp's lanes have at most eight 16-byte loads each
  if (seg <= 1024) {
    constexpr int per = kThreads / 32;
    range_minmax_kernel<true><<<static_cast<unsigned>((nseg + per - 1) / per), kThreads, 0, stream>>>(W0, nseg, seg,
                                                                                                    bits, s0, z0);
  } else {
    range_minmax_kernel<false><<<static_cast<unsigned>(nseg), kThreads, 0, stream>>>(W0, nseg, seg, bits, s0, z0);
  }
  return cudaGetLastError();
}

cudaError_t launch_range_lp(const float* W0, int64_t m, int64_t k, int group_size, int bits, float p_norm, int n_cand,
                            float* s0, int sms, cudaStream_t stream) {
  const int seg = group_size ? group_size : static_cast<int>(k);
  const int64_t nseg = m * (k / seg);
  if (n_cand < 1 || n_cand > kLpMaxCand || bits > 8) return cudaErrorInvalidValue;
  // Segments per block: the fewest warp rounds on the busiest SM (a block's threads are its
  // segments' candidates, padded to whole warps).  At most 512 threads, so that several blocks
  // share an SM and one computes while another fetches its chunk (5120 x 5120, N = 100, the last
  // product still fused with the sum: 814 us with 512 threads, 936 us with 704); segments of a single chunk have less work between
  // barriers and take smaller blocks (groups of 128: 1101 us with 320 threads, 1312 us with 512).
  const int max_threads = seg <= kLpChunk ? 320 : kLpMaxThreads;
  int best = 1;
  int64_t best_cost = -1;
  for (int R = 1; R <= kLpMaxSegs && (R == 1 || R * n_cand <= max_threads); ++R) {
    const int64_t blocks = (nseg + R - 1) / R;
    const int64_t cost = (blocks + sms - 1) / sms * ((R * n_cand + 31) / 32);
    if (best_cost < 0 || cost <= best_cost) {
      best_cost = cost;
      best = R;
    }
  }
  const unsigned blocks = static_cast<unsigned>((nseg + best - 1) / best);
  const unsigned threads = static_cast<unsigned>((best * n_cand + 31) / 32 * 32);
  const int ip = static_cast<int>(p_norm);
  const bool int_p = static_cast<float>(ip) == p_norm && ip >= 1 && ip <= 8;
  auto kernel = !int_p    ? range_lp_kernel<0>
                : ip == 1 ? range_lp_kernel<1>
                : ip == 2 ? range_lp_kernel<2>
                : ip == 3 ? range_lp_kernel<3>
                : ip == 4 ? range_lp_kernel<4>
                : ip == 5 ? range_lp_kernel<5>
                : ip == 6 ? range_lp_kernel<6>
                : ip == 7 ? range_lp_kernel<7>
                          : range_lp_kernel<8>;
  kernel<<<blocks, threads, 0, stream>>>(W0, nseg, seg, best, bits, p_norm, n_cand, s0);
  return cudaGetLastError();
}

cudaError_t launch_downcast(const float* W0, const float* s0, const float* z0, int64_t m, int64_t k, int group_size,
                            int bits, int fmt, void* phi0, cudaStream_t stream) {
  if (fmt_float(fmt) && z0 != nullptr) return cudaErrorInvalidValue;
  const int ngroups = group_size ? static_cast<int>(k / group_size) : 1;
  const float n = -static_cast<float>(1 << (bits - 1)), p = static_cast<float>((1 << (bits - 1)) - 1);
  const float two_f = fmt == FMT_Q8 ? static_cast<float>(1 << (8 - bits)) : 1.0f;
  const int64_t col_blocks = (k + kDownCols - 1) / kDownCols;
  const dim3 grid(static_cast<unsigned>(m), static_cast<unsigned>(col_blocks < 65535 ? col_blocks : 65535));
  auto kernel = fmt == FMT_Q8     ? downcast_kernel<FMT_Q8>
                : fmt == FMT_I4   ? downcast_kernel<FMT_I4>
                : fmt == FMT_BF16 ? downcast_kernel<FMT_BF16>
                : fmt == FMT_F16  ? downcast_kernel<FMT_F16>
                : fmt == FMT_E4M3 ? downcast_kernel<FMT_E4M3>
                                  : downcast_kernel<FMT_E5M2>;
  kernel<<<grid, kDownThreads, 0, stream>>>(W0, s0, z0, k, group_size, ngroups, n, p, two_f, phi0);
  return cudaGetLastError();
}

}  // namespace lrqat
