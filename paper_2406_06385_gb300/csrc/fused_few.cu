// Fused LR-QAT forward (Y = X W_hat^T) for a few tokens (up to 16) and ranks up to 64: a serving call.
// Nothing is worth a pass of its own here: the stored base is read once (the floor, 2.5 us for a
// 4096 x 4096 8-bit base), and the products are small.
//
// The pair GEMM has 16 tiles of 256 rows for such a call on a 4096 x 4096 layer, and each walks the
// contraction in 64 stages paced by barrier and MMA-issue latencies (57 us, 27 us with two pairs per
// tile).  Here a CTA takes 32 rows and its sixteen warps split the contraction, so every SM has
// work, and W_hat never leaves registers: with mma.sync (m16n8k16) the accumulator of the low-rank
// product L = A B has the register layout that the A operand of the main product wants, so a
// warp turns L and the stored base into bf16 codes and multiplies them at once.  The tcgen05 path
// would need the codes in shared or tensor memory and 128 rows per MMA; the tensor work is 1.6 GFLOP at
// T = 16, r = 32, far below either rate.
// Measured, 4096 x 4096, T = 16, r = 32 (adapter layouts included): 57 + 2 us before,
// 13.1 + 2.1 us.
//
// Columns and ranks are taken in an order that makes a thread's loads contiguous (a contraction may
// be summed in any order, the same on both operands): in a block of 64 columns, thread c of a
// quad owns the 16 columns 16 c .. 16 c + 15, four of them (4 s ..) in K step s at the positions
// 2 c, 2 c + 1, 2 c + 8, 2 c + 9 that the fragment layout gives it; ranks likewise, r16 / 4 per thread.
#include <cuda_runtime.h>
#include <cstdint>

#include "kernels.h"
#include "ptx.cuh"
#include "quant.cuh"

namespace lrqat {
namespace {

constexpr int kRows = 32;       // weight rows per CTA (two m16 tiles)
constexpr int kWarps = 16;      // parts of the contraction
constexpr int kThreads = 32 * kWarps;

// D += A B, m16n8k16, bf16 inputs and fp32 sums.
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The 16 stored values of a row that a thread owns in a block: 16, 8 (packed) or 32 (16-bit) bytes.
template <int FMT>
struct Raw {
  static constexpr int kWords = FMT == FMT_I4 ? 2 : fmt_16bit(FMT) ? 8 : 4;
  uint32_t w[kWords];
};
template <int FMT>
__device__ __forceinline__ void load_raw(const void* phi, int64_t row, int64_t k, int64_t col, Raw<FMT>& r) {
  if constexpr (FMT == FMT_I4) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(static_cast<const uint8_t*>(phi) + (row * k + col) / 2));
    r.w[0] = v.x, r.w[1] = v.y;
  } else {
    const uint4* src = reinterpret_cast<const uint4*>(static_cast<const uint8_t*>(phi) +
                                                      (row * k + col) * (fmt_16bit(FMT) ? 2 : 1));
#pragma unroll
    for (int i = 0; i < Raw<FMT>::kWords / 4; ++i) {
      const uint4 v = __ldg(src + i);
      r.w[4 * i] = v.x, r.w[4 * i + 1] = v.y, r.w[4 * i + 2] = v.z, r.w[4 * i + 3] = v.w;
    }
  }
}

// NT8: token tiles of 8.  KS: rank steps of 16.
template <int FMT, int NT8, int KS>
__global__ void __launch_bounds__(kThreads, 1) fused_few_kernel(const FewArgs args) {
  __shared__ float part[kWarps / 2][8 * NT8][kRows + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, c = lane & 3;   // fragment row (or column n) and quad position
  const int64_t row0 = static_cast<int64_t>(blockIdx.x) * kRows, k = args.k;
  const QuantParams qp = args.q;
  const uint32_t lr2 = pack_rn_bf16x2(qp.lr_scale, qp.lr_scale);   // exact: a power of two with u_bf16
  const bool ub = args.u_bf16, zp = args.zero != nullptr, grouped = args.group_size != 0;

  const int nblocks = static_cast<int>(k / 64);
  Raw<FMT> raw[2][2], nxt[2][2];
  auto load_block = [&](int b, Raw<FMT> (&r)[2][2]) {
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        load_raw<FMT>(args.phi, row0 + 16 * mt + 8 * h + g, k, static_cast<int64_t>(b) * 64 + 16 * c, r[mt][h]);
  };
  if (warp < nblocks) load_block(warp, nxt);
  // The base is the caller's, complete before the call's first kernel began; X and the factors may come
  // from the call's kernels before this one and are read with plain loads after the wait.
  griddep_wait();

  // A [32 rows, r16] as fragments: rows g, g + 8 of each m16 tile, this thread's r16 / 4 ranks
  uint32_t af[2][KS][4];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint2* src = reinterpret_cast<const uint2*>(args.a_pad + (row0 + 16 * mt + 8 * h + g) * 64 + c * (4 * KS));
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const uint2 v = src[ks];   // ranks at positions 2 c, 2 c + 1 | 2 c + 8, 2 c + 9
        af[mt][ks][h] = v.x;
        af[mt][ks][2 + h] = v.y;
      }
    }
  uint32_t z2[2][2] = {}, s2[2][2] = {};   // the rows' zero offsets and group scales as bf16x2
  if (zp && !grouped) {
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float z = args.zero[row0 + 16 * mt + 8 * h + g];
        z2[mt][h] = pack_rn_bf16x2(z, z);
      }
  }
  float acc[2][NT8][4] = {};
  for (int b = warp; b < nblocks; b += kWarps) {
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int h = 0; h < 2; ++h) raw[mt][h] = nxt[mt][h];
    if (b + kWarps < nblocks) load_block(b + kWarps, nxt);   // the next block's base comes meanwhile
    const int64_t col0 = static_cast<int64_t>(b) * 64;
    if (grouped) {
      const int64_t gi = col0 / args.group_size;
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int64_t e = (row0 + 16 * mt + 8 * h + g) * args.s_ld + gi;
          s2[mt][h] = pack_rn_bf16x2(args.s[e], args.s[e]);
          if (zp) z2[mt][h] = pack_rn_bf16x2(args.zero[e], args.zero[e]);
        }
    }
    // X: token 8 n + g, this thread's 16 columns (tokens past T read as zeros)
    uint4 x[NT8][2];
#pragma unroll
    for (int n = 0; n < NT8; ++n) {
      const int t = 8 * n + g;
      const uint4* src = reinterpret_cast<const uint4*>(args.X + static_cast<int64_t>(t) * k + col0 + 16 * c);
#pragma unroll
      for (int h = 0; h < 2; ++h) x[n][h] = t < args.T ? src[h] : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      // L of the step's 16 columns: column n of half hf is physical column 16 (n / 2) + 4 s + 2 hf + n % 2
      float L[2][2][4] = {};   // [m tile][half]: (row g: 2 columns | row g + 8: 2 columns)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int64_t col = col0 + 16 * (g >> 1) + 4 * s + 2 * hf + (g & 1);
        const uint2* src = reinterpret_cast<const uint2*>(args.bt_pad + col * 64 + c * (4 * KS));
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          const uint2 v = src[ks];
#pragma unroll
          for (int mt = 0; mt < 2; ++mt) mma16816(L[mt][hf], af[mt][ks], v.x, v.y);
        }
      }
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        uint32_t w[4];   // the main product's A fragment: (g | g + 8) x (first | second column pair)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float v[16];
          decode16<FMT>(raw[mt][h].w, v);   // (the four values of step s; the rest is dead code)
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            const float l0 = L[mt][hf][2 * h], l1 = L[mt][hf][2 * h + 1];
            const float v0 = v[4 * s + 2 * hf], v1 = v[4 * s + 2 * hf + 1];
            const float2 u = ub ? u_bf16x2(l0, l1, v0, v1, lr2)
                                : __ffma2_rn(make_float2(l0, l1), make_float2(qp.lr_scale, qp.lr_scale),
                                             make_float2(v0, v1));
            uint32_t cw = codes_bf16x2(__fadd2_rn(u, make_float2(qp.magic, qp.magic)), qp);
            if (zp) cw = sub_bf16x2(cw, z2[mt][h]);
            if (grouped) cw = mul_bf16x2(cw, s2[mt][h]);
            w[2 * hf + h] = cw;
          }
        }
#pragma unroll
        for (int n = 0; n < NT8; ++n) {
          const uint4& xv = x[n][s >> 1];   // columns 4 s .. 4 s + 3: two words
          mma16816(acc[mt][n], w, (s & 1) ? xv.z : xv.x, (s & 1) ? xv.w : xv.y);
        }
      }
    }
  }
  // The warps' sums: the upper half of the warps hands its sums to the lower, then every output adds
  // the eight in order.
  auto put = [&](int slot, bool add) {
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int n = 0; n < NT8; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float& p = part[slot][8 * n + 2 * c + (e & 1)][16 * mt + g + 8 * (e >> 1)];
          p = add ? p + acc[mt][n][e] : acc[mt][n][e];
        }
  };
  if (warp >= kWarps / 2) put(warp - kWarps / 2, false);
  __syncthreads();
  if (warp < kWarps / 2) put(warp, true);
  __syncthreads();
  const float sx = args.s_x != nullptr ? *args.s_x : 1.0f;
  for (int o = threadIdx.x; o < 8 * NT8 * (kRows / 2); o += kThreads) {
    const int t = o / (kRows / 2), r = 2 * (o % (kRows / 2));
    if (t >= args.T) break;
    float y0 = 0.0f, y1 = 0.0f;
#pragma unroll
    for (int p = 0; p < kWarps / 2; ++p) {
      y0 += part[p][t][r];
      y1 += part[p][t][r + 1];
    }
    const float f0 = (grouped ? 1.0f : args.s[row0 + r]) * sx, f1 = (grouped ? 1.0f : args.s[row0 + r + 1]) * sx;
    *reinterpret_cast<uint32_t*>(args.Y + static_cast<int64_t>(t) * args.m + row0 + r) = pack_rn_bf16x2(y0 * f0, y1 * f1);
  }
}

template <int FMT, int NT8>
cudaError_t launch_ks(const FewArgs& a, cudaStream_t stream) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(a.m / kRows), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1] = {follows_in_call()};
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e;
  switch (a.r16) {
    case 16: e = cudaLaunchKernelEx(&cfg, fused_few_kernel<FMT, NT8, 1>, a); break;
    case 32: e = cudaLaunchKernelEx(&cfg, fused_few_kernel<FMT, NT8, 2>, a); break;
    case 48: e = cudaLaunchKernelEx(&cfg, fused_few_kernel<FMT, NT8, 3>, a); break;
    case 64: e = cudaLaunchKernelEx(&cfg, fused_few_kernel<FMT, NT8, 4>, a); break;
    default: return cudaErrorInvalidValue;
  }
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int FMT>
cudaError_t launch_nt(const FewArgs& a, cudaStream_t stream) {
  return a.T <= 8 ? launch_ks<FMT, 1>(a, stream) : launch_ks<FMT, 2>(a, stream);
}

}  // namespace

cudaError_t launch_fused_few(int fmt, const FewArgs& a, cudaStream_t stream) {
  if (a.T < 1 || a.T > kFewTokens || a.m % kRows || a.k % 64) return cudaErrorInvalidValue;
  switch (fmt) {
    case FMT_Q8: return launch_nt<FMT_Q8>(a, stream);
    case FMT_I4: return launch_nt<FMT_I4>(a, stream);
    case FMT_BF16: return launch_nt<FMT_BF16>(a, stream);
    case FMT_F16: return a.u_bf16 ? cudaErrorInvalidValue : launch_nt<FMT_F16>(a, stream);
    case FMT_E4M3: return launch_nt<FMT_E4M3>(a, stream);
    case FMT_E5M2: return launch_nt<FMT_E5M2>(a, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lrqat
