// Optimizer step on the trainable parameters of an LR-QAT layer (App. B, Table B1):
// AdamW with decoupled weight decay over A, B (fp32 master copies, bf16 copies for the
// GEMMs) and the scales s, after clipping the global L2 norm of all trainable
// gradients.  The norm is accumulated layer by layer into one device scalar.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <atomic>
#include <cstdint>
#include <utility>

#include "kernels.h"
#include "quant.cuh"

namespace lrqat {
namespace {

namespace cg = cooperative_groups;

// ---- squared gradient norm ------------------------------------------------------------------
// One cluster of up to 16 CTAs (the gradients of one layer are 1-6 MB: one SM alone takes over
// 100 us to read them, and an entry point without a workspace has no place for the partial sums
// of a grid; a cluster adds its CTAs' sums through distributed shared memory).  The squares are
// summed as unevaluated pairs of floats (Knuth's two-sum, the square's rounding error by one FMA):
// about 48 bits at the FP32 rate, where the FP64 pipe of this GPU (about two lanes per SM and
// clock) made a sum in doubles cost 150 us of the 253 us that a 13824 x 5120 layer at r = 32 took.
// Measured on that layer: 253 us (one CTA, doubles) -> 7.8 us
// (20 us while every thread still added its four sums in doubles).
constexpr int kNormThreads = 1024;
constexpr int kNormCluster = 16;         // CTAs; 8 (the portable size) where 16 cannot be resident
// 2^48: sums of squares of values up to it stay finite.  A warp adds 128 squares per item of its
// threads before it goes to doubles, and 128 x items x 2^96 < 2^127 up to 2^24 items per thread, which would be
// 2^39 gradients on eight CTAs.  (With 2^60 the warps' sums left fp32 from about 2^58 on, and the
// two-sum then makes inf - inf: a NaN norm, which AdamW does not clip by.)
constexpr float kNormBig = 2.8147498e14f;
constexpr float kNormSmall = 9.094947e-13f;  // 2^-40: the squares' rounding errors stay normal above it

// hi + lo += x^2, exactly up to the rounding of lo.
__device__ __forceinline__ void add_square(float x, float& hi, float& lo) {
  const float p = __fmul_rn(x, x);
  const float e = __fmaf_rn(x, x, -p);
  const float s = __fadd_rn(hi, p);
  const float b = __fsub_rn(s, hi);
  const float r = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(p, b));
  hi = s;
  lo = __fadd_rn(lo, __fadd_rn(r, e));
}

struct NormSeg {
  const float* g;
  int64_t n;       // a multiple of 4 (m and k are multiples of 128)
  int aligned;     // 16-byte aligned: read as float4
};

__device__ __forceinline__ float4 load4(const NormSeg& s, int64_t i) {
  if (s.aligned) return __ldg(reinterpret_cast<const float4*>(s.g) + i);
  const float* p = s.g + 4 * i;
  return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}

// The pair (hi, lo) += the pair (h, l).
__device__ __forceinline__ void add_pair(float h, float l, float& hi, float& lo) {
  const float s = __fadd_rn(hi, h);
  const float b = __fsub_rn(s, hi);
  const float r = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(h, b));
  hi = s;
  lo = __fadd_rn(lo, __fadd_rn(r, l));
}

// Four independent sums (one per element of a 16-byte load) and the largest magnitude seen.
struct NormAcc {
  float hi[4], lo[4], amax;
};

// The gradients of a layer as one range of 16-byte items.
struct NormRange {
  NormSeg a, b, c;
  int64_t n;   // items
};
__device__ __forceinline__ float4 load_item(const NormRange& r, int64_t i) {
  const int64_t na = r.a.n / 4, nb = r.b.n / 4;
  return i < na ? load4(r.a, i) : i < na + nb ? load4(r.b, i - na) : load4(r.c, i - na - nb);
}

// This thread's share (items t0, t0 + stride, ...), kNormLoads loads in flight; items past the end count as
// zeros, which change nothing.  A layer has about ten items per thread, so its time is the number of round trips: a
// batch of four and single loads for the rest, array by array, made seven of them, this makes two (the
// optimizer step of a 13B decoder layer on fresh gradients, seven such launches: 142.5 -> 132.4 us).
constexpr int kNormLoads = 8;
__device__ __forceinline__ void norm_share(const NormRange& r, int64_t t0, int64_t stride, NormAcc& a) {
  for (int64_t i = t0; i < r.n; i += kNormLoads * stride) {
    float4 v[kNormLoads];
#pragma unroll
    for (int u = 0; u < kNormLoads; ++u) {
      v[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (i + u * stride < r.n) v[u] = load_item(r, i + u * stride);
    }
#pragma unroll
    for (int u = 0; u < kNormLoads; ++u) {
      add_square(v[u].x, a.hi[0], a.lo[0]);
      add_square(v[u].y, a.hi[1], a.lo[1]);
      add_square(v[u].z, a.hi[2], a.lo[2]);
      add_square(v[u].w, a.hi[3], a.lo[3]);
      a.amax = fmaxf(a.amax, fmaxf(fmaxf(fabsf(v[u].x), fabsf(v[u].y)), fmaxf(fabsf(v[u].z), fabsf(v[u].w))));
    }
  }
}

// The same share summed in doubles, for values whose squares leave the range of the pairs.
__device__ __noinline__ double norm_share_wide(const NormRange& r, int64_t t0, int64_t stride) {
  double acc = 0.0;
  for (int64_t i = t0; i < r.n; i += stride) {
    const float4 v = load_item(r, i);
    acc += static_cast<double>(v.x) * v.x;
    acc += static_cast<double>(v.y) * v.y;
    acc += static_cast<double>(v.z) * v.z;
    acc += static_cast<double>(v.w) * v.w;
  }
  return acc;
}

// Sum of squares of dA, dB and ds, added into *sqnorm: every thread adds a fixed subset in a
// fixed order, then fixed trees add the threads and the CTAs, so the result does not depend on
// scheduling.
__global__ void __launch_bounds__(kNormThreads) grad_sqnorm_kernel(const NormRange r,
                                                                   float* __restrict__ sqnorm) {
  cg::cluster_group cluster = cg::this_cluster();
  // Every CTA has to have started before another writes its shared memory: arrive here, wait before
  // that write (the loads lie between, so the wait costs nothing).
  auto started = cluster.barrier_arrive();
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kNormThreads;
  const int64_t t0 = static_cast<int64_t>(blockIdx.x) * kNormThreads + threadIdx.x;
  __shared__ double part[kNormThreads / 32];
  __shared__ double cta_sum[kNormCluster];   // CTA 0's copy collects every CTA's sum
  NormAcc n{};
  norm_share(r, t0, stride, n);
  // A thread whose values are all tiny, or one of them huge or infinite, sums them in doubles,
  // which neither overflow nor lose them; its warp then adds doubles.
  const bool wide = n.amax > kNormBig || (n.amax < kNormSmall && n.amax > 0.0f);
  double acc;
  if (__any_sync(0xffffffffu, wide)) {
    acc = 0.0;
    if (wide) {
      acc = norm_share_wide(r, t0, stride);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) acc += static_cast<double>(n.hi[i]) + n.lo[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  } else {
    float hi = n.hi[0], lo = n.lo[0];
#pragma unroll
    for (int i = 1; i < 4; ++i) add_pair(n.hi[i], n.lo[i], hi, lo);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h = __shfl_xor_sync(0xffffffffu, hi, o), l = __shfl_xor_sync(0xffffffffu, lo, o);
      add_pair(h, l, hi, lo);
    }
    acc = static_cast<double>(hi) + lo;
  }
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc = part[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  }
  cluster.barrier_wait(std::move(started));
  if (threadIdx.x == 0) cluster.map_shared_rank(cta_sum, 0)[blockIdx.x] = acc;
  cluster.sync();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    double total = 0.0;
    for (unsigned i = 0; i < gridDim.x; ++i) total += cta_sum[i];
    *sqnorm = static_cast<float>(static_cast<double>(*sqnorm) + total);
  }
}

// ---- AdamW -----------------------------------------------------------------------------------
struct AdamSeg {
  const float* g;     // gradient
  float* p;           // fp32 parameter (master copy)
  float* m;
  float* v;
  uint16_t* p_bf16;   // bf16 copy written after the update, or nullptr
  int64_t n;
  float lr, wd;
};

// One AdamW step per element of three segments (A, B, s) in one launch:
//   g <- coef g;  m <- b1 m + (1 - b1) g;  v <- b2 v + (1 - b2) g^2;
//   p <- p (1 - lr wd) - lr (m / bc1) / (sqrt(v / bc2) + eps)
// with coef = min(1, max_norm / (sqrt(sqnorm) + 1e-6)) (1 when max_norm <= 0).
struct AdamHyper {
  float beta1, beta2, eps, bc1, bc2;
};
__device__ __forceinline__ void adam_element(float grad, float coef, float lr, float wd, const AdamHyper& h, float& p,
                                             float& m, float& v) {
  const float g = coef * grad;
  m = h.beta1 * m + (1.0f - h.beta1) * g;
  v = h.beta2 * v + (1.0f - h.beta2) * g * g;
  p = p * (1.0f - lr * wd) - lr * (m / h.bc1) / (sqrtf(v / h.bc2) + h.eps);
}
__device__ __forceinline__ float clip_coef(const float* sqnorm, float max_norm) {
  return max_norm > 0.0f ? fminf(1.0f, max_norm / (sqrtf(*sqnorm) + 1e-6f)) : 1.0f;
}

// Four elements per thread, each array one 16-byte access (HBM bound: 30 bytes per element).
// Measured on a 13824 x 5120 layer at r = 32: one element per thread 13.1 us, four 5.9 us.
__global__ void __launch_bounds__(256) adamw4_kernel(AdamSeg s0, AdamSeg s1, AdamSeg s2,
                                                     const float* __restrict__ sqnorm, float max_norm, AdamHyper h) {
  const int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;   // float4 index
  const int64_t n0 = s0.n / 4, n1 = s1.n / 4, n2 = s2.n / 4;
  if (e >= n0 + n1 + n2) return;
  const AdamSeg& S = e < n0 ? s0 : (e < n0 + n1 ? s1 : s2);
  const int64_t i = e < n0 ? e : (e < n0 + n1 ? e - n0 : e - n0 - n1);
  const float4 g = __ldg(reinterpret_cast<const float4*>(S.g) + i);
  float4 m = reinterpret_cast<const float4*>(S.m)[i];
  float4 v = reinterpret_cast<const float4*>(S.v)[i];
  float4 p = reinterpret_cast<const float4*>(S.p)[i];
  const float coef = clip_coef(sqnorm, max_norm);
  adam_element(g.x, coef, S.lr, S.wd, h, p.x, m.x, v.x);
  adam_element(g.y, coef, S.lr, S.wd, h, p.y, m.y, v.y);
  adam_element(g.z, coef, S.lr, S.wd, h, p.z, m.z, v.z);
  adam_element(g.w, coef, S.lr, S.wd, h, p.w, m.w, v.w);
  reinterpret_cast<float4*>(S.m)[i] = m;
  reinterpret_cast<float4*>(S.v)[i] = v;
  reinterpret_cast<float4*>(S.p)[i] = p;
  if (S.p_bf16) reinterpret_cast<uint2*>(S.p_bf16)[i] = make_uint2(pack_rn_bf16x2(p.x, p.y), pack_rn_bf16x2(p.z, p.w));
}

// Arrays that are not 16-byte aligned (bf16 copies: 8-byte): one element per thread.
__global__ void adamw_kernel(AdamSeg s0, AdamSeg s1, AdamSeg s2, const float* __restrict__ sqnorm, float max_norm,
                             AdamHyper h) {
  const float coef = clip_coef(sqnorm, max_norm);
  const int64_t total = s0.n + s1.n + s2.n;
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < total;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const AdamSeg& S = e < s0.n ? s0 : (e < s0.n + s1.n ? s1 : s2);
    const int64_t i = e < s0.n ? e : (e < s0.n + s1.n ? e - s0.n : e - s0.n - s1.n);
    float p = S.p[i], m = S.m[i], v = S.v[i];
    adam_element(S.g[i], coef, S.lr, S.wd, h, p, m, v);
    S.m[i] = m;
    S.v[i] = v;
    S.p[i] = p;
    if (S.p_bf16) S.p_bf16[i] = static_cast<uint16_t>(pack_rn_bf16x2(p, 0.0f) & 0xFFFFu);
  }
}

}  // namespace

namespace {

bool aligned(const void* p, uintptr_t bytes) { return (reinterpret_cast<uintptr_t>(p) & (bytes - 1)) == 0; }

// CTAs of the norm's cluster on the current device: 16 where such a cluster can be resident.
cudaError_t norm_cluster_size(int* size) {
  static std::atomic<int> cache[kMaxDevices];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (cache[dev].load(std::memory_order_acquire) == 0) {
    e = cudaFuncSetAttribute(grad_sqnorm_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kNormCluster, 1, 1);
    cfg.blockDim = dim3(kNormThreads, 1, 1);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kNormCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, grad_sqnorm_kernel, &cfg);
    if (e != cudaSuccess) {
      (void)cudaGetLastError();   // not launchable at this size
      n = 0;
    }
    cache[dev].store(n > 0 ? kNormCluster : 8, std::memory_order_release);
  }
  *size = cache[dev].load(std::memory_order_acquire);
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_grad_sqnorm(const float* dA, int64_t na, const float* dB, int64_t nb, const float* ds, int64_t nc,
                               float* sqnorm, cudaStream_t stream) {
  int size = 0;
  cudaError_t e = norm_cluster_size(&size);
  if (e != cudaSuccess) return e;
  const NormRange r{{dA, na, aligned(dA, 16)}, {dB, nb, aligned(dB, 16)}, {ds, nc, aligned(ds, 16)}, (na + nb + nc) / 4};
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(size), 1, 1);
  cfg.blockDim = dim3(kNormThreads, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(size);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, grad_sqnorm_kernel, r, sqnorm);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

cudaError_t launch_adamw(const AdamwArgs& a, cudaStream_t stream) {
  const AdamSeg s0{a.dA, a.A32, a.mA, a.vA, a.A, a.nA, a.lr_ab, a.wd_ab};
  const AdamSeg s1{a.dB, a.B32, a.mB, a.vB, a.B, a.nB, a.lr_ab, a.wd_ab};
  const AdamSeg s2{a.ds, a.s, a.ms, a.vs, nullptr, a.ns, a.lr_s, a.wd_s};
  const AdamHyper h{a.beta1, a.beta2, a.eps, a.bc1, a.bc2};
  const int64_t total = a.nA + a.nB + a.ns;
  bool vec = true;   // the segments' sizes are multiples of 4 (m and k are multiples of 128)
  for (const AdamSeg* s : {&s0, &s1, &s2})
    vec = vec && aligned(s->g, 16) && aligned(s->p, 16) && aligned(s->m, 16) && aligned(s->v, 16) &&
          aligned(s->p_bf16, 8);
  if (vec) {
    adamw4_kernel<<<static_cast<unsigned>((total / 4 + 255) / 256), 256, 0, stream>>>(s0, s1, s2, a.sqnorm, a.max_norm,
                                                                                      h);
  } else {
    const int64_t want = (total + 255) / 256;
    adamw_kernel<<<static_cast<unsigned>(want < 2048 ? want : 2048), 256, 0, stream>>>(s0, s1, s2, a.sqnorm, a.max_norm,
                                                                                       h);
  }
  return cudaGetLastError();
}

}  // namespace lrqat
