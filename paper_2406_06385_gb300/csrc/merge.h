// Launcher of the tensor-core low-rank code pass (merge.cu).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "quant.cuh"

namespace lrqat {

// Codes c = clip(round(phi^{-1}(Phi0) + (alpha/r) A B), n, p) of every element on the tensor cores:
// the merge W_Z of Sec. 3 (int8), or the one-byte codes c + bias that the GEMMs read as their
// base, row-major and / or transposed.
//   a_mn == 0: tm_a over A [m, r] (r % 8 == 0, 16-byte aligned), K-major boxes of 128 rows x 64
//     columns (16 or 32 columns for r16 = 16 or 32, with the swizzle of their row length);
//   a_mn == 1: tm_a over the zero-padded A^T [r16, m], 64 x r16 boxes, MN-major.
//   tm_b over B [r, k] or the zero-padded B [r16, k], 64 x r16 boxes.  All 128-byte swizzled;
//   tm_phi over the stored base in 128-column chunks: 8-bit values 128 x 128 boxes (SW128),
//   packed nibbles 64-byte x 128-row boxes (SW64), 16-bit values 64 x 128 boxes (SW128);
//   wz and wt 16-byte aligned.
struct MergeArgs {
  int8_t* wz;            // codes [m, k], or nullptr
  int8_t* wt;            // codes transposed [k, m] (without mask bits), or nullptr
  int64_t m, k;
  int32_t r16;           // adapter rank rounded up to 16 (<= 256)
  QuantParams q;         // q.lo / q.hi: n and p in the magic domain
  int* status;
  uint64_t timeout_ns;
  uint32_t code_bias;    // added to every stored code: 0 (two's complement), 64 or 128 (c + bias, unsigned)
  int32_t bits;          // b; code_bias 0 or 64 up to 7, 0 or 128 for 8
  int32_t mask_bit;      // wz: bit 7 = 1[n <= round(u) <= p], the STE mask (needs code_bias 64)
  // The scales (and zero offsets, or nullptr) as bf16 rows [s_groups][m] for the GEMM producers,
  // from s [m, s_groups]; s_out == nullptr: not written.
  const float* s;
  const float* z;
  uint16_t* s_out;
  uint16_t* z_out;
  int32_t s_groups;
  // A^T [r16, m] (rows past r zero) from A [m, r] for the weight-gradient kernel; at_out == nullptr:
  // not written.
  const uint16_t* A;
  uint16_t* at_out;
  int32_t r;
};
// fmt: a PhiFmt value (quant.cuh); u_bf16: the bf16 pre-round value (not with FP16 bases)
cudaError_t launch_merge_tc(int fmt, int u_bf16, int a_mn, const CUtensorMap& tm_a, const CUtensorMap& tm_b,
                            const CUtensorMap& tm_phi, const MergeArgs& args, cudaStream_t stream);

}  // namespace lrqat
