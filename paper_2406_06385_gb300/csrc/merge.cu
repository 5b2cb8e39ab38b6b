// Merge on the tensor cores (Sec. 3: after training the integer weight is
// W_Z = clip(round(phi^{-1}(Phi0) + (alpha/r) A B), n, p), and W_hat = s W_Z), and the
// same pass writing the one-byte codes that the fused GEMMs read as their base (the codes
// path): the code plus a bias (64, or 128 for 8-bit weights), row-major for the forward,
// transposed for dX, and for dW row-major with the clip mask in the byte's top bit.
//
// Tiles of 128 x 128: the tile's rows of A and columns of B land by TMA, r16 / 16 tcgen05
// MMAs write the low-rank tile L = A B into TMEM, and warps q and q + 4 turn rows 32q .. 32q + 31
// into codes (TMEM lane = row): they read L 32 columns at a time, take the stored base of the same
// 32 columns (staged by TMA into the operand slot), round, clip, add the bias and store 32
// one-byte codes as one 32-byte word.  The CTAs are persistent and overlap one tile's codes with
// the next tile's copies and MMAs (two TMEM buffers).  The pass moves the base and the codes once (the
// product costs 2 m k r flops on the tensor cores instead of the CUDA cores).
//   A operand: K-major boxes of 64 rank columns read from A [m, r] (r % 8 == 0; columns
//   past r read as zeros), or (AMN) two MN-major boxes of r16 rank rows x 64 rows read
//   from the zero-padded A^T [r16, m].
//   B operand: two MN-major boxes of r16 rank rows x 64 columns read from B [r, k] (rows
//   past r read as zeros) or from the zero-padded B [r16, k].
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "kernels.h"
#include "merge.h"
#include "ptx.cuh"
#include "quant.cuh"

namespace lrqat {
namespace {

// Operand slot: A (up to 64 KB at r16 = 256), then B (two boxes of r16 rows x 128 bytes).
// Two slots when they fit (ranks up to 128), else one.  Every CTA asks for at least 80 KB of
// shared memory so that no more than two CTAs share an SM: two 256-column TMEM allocations
// fill its 512 columns, and a third CTA would wait inside tcgen05.alloc.
constexpr uint32_t MIN_SMEM_BYTES = 80 * 1024;
constexpr uint32_t MAX_SMEM_BYTES = 232448 - 1024;   // the per-CTA limit, less the static barriers
constexpr uint32_t TMEM_COLS = 256;   // two 128-column low-rank tiles
constexpr int NUM_EPI_WARPS = 8;
constexpr int TMA_WARP = NUM_EPI_WARPS, MMA_WARP = NUM_EPI_WARPS + 1;
constexpr int NUM_THREADS = 32 * (MMA_WARP + 1);
// Transposed output: each epilogue warp turns blocks of 32 rows x 32 codes through a staging
// buffer of 32 rows of eight words, nine words apart (conflict-free both ways).
constexpr int STG_ROW = 9;
constexpr uint32_t STG_BYTES = NUM_EPI_WARPS * 32 * STG_ROW * 4;

// Rank columns of a K-major A box: 16 or 32 (rows of 32 or 64 bytes) for those ranks, else 64.
__host__ __device__ constexpr int a_box_cols(int r16) { return r16 <= 32 ? r16 : 64; }
__host__ __device__ constexpr uint32_t a_tile_bytes(int r16, bool amn) {
  return amn           ? 2u * 128u * static_cast<uint32_t>(r16)
         : r16 <= 32   ? 256u * static_cast<uint32_t>(r16)
                       : 16384u * static_cast<uint32_t>((r16 + 63) / 64);
}
// Bytes of the stored base of a 128 x 128 tile: 8-bit values, packed nibbles, 16-bit values.
__host__ __device__ constexpr uint32_t phi_tile_bytes(int fmt) {
  return fmt == FMT_I4 ? 8192u : fmt_16bit(fmt) ? 32768u : 16384u;
}
// Operand slot: A, then B, then the stored base of the tile.
__host__ __device__ constexpr uint32_t slot_bytes(int r16, bool amn, int fmt) {
  return a_tile_bytes(r16, amn) + 2u * 128u * static_cast<uint32_t>(r16) + phi_tile_bytes(fmt);
}
// Slots: as many (up to four) as fit while two CTAs share an SM; when not even two fit, as
// many as fit in one CTA per SM.
constexpr uint32_t MAX_SLOTS = 4;
constexpr uint32_t TWO_PER_SM_BYTES = 232448u / 2u - 1024u;
__host__ __device__ constexpr uint32_t min_u(uint32_t a, uint32_t b) { return a < b ? a : b; }
__host__ __device__ constexpr int num_slots(int r16, bool amn, int fmt) {
  return (TWO_PER_SM_BYTES - 1024u - STG_BYTES) / slot_bytes(r16, amn, fmt) >= 2
             ? static_cast<int>(min_u(MAX_SLOTS, (TWO_PER_SM_BYTES - 1024u - STG_BYTES) / slot_bytes(r16, amn, fmt)))
             : static_cast<int>(min_u(MAX_SLOTS, (MAX_SMEM_BYTES - 1024u - STG_BYTES) / slot_bytes(r16, amn, fmt)));
}
__host__ __device__ constexpr uint32_t smem_bytes(int r16, bool amn, int fmt) {
  return num_slots(r16, amn, fmt) * slot_bytes(r16, amn, fmt) + 1024u + STG_BYTES < MIN_SMEM_BYTES
             ? MIN_SMEM_BYTES
             : num_slots(r16, amn, fmt) * slot_bytes(r16, amn, fmt) + 1024u + STG_BYTES;
}

__device__ __forceinline__ void drain_wait(uint32_t bar, uint32_t parity, uint64_t timeout_ns) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > timeout_ns) break;
  }
}

// Raw words of the stored base per 32 columns of a row: 16 bytes (packed nibbles),
// 32 bytes (one byte per value) or 64 bytes (16-bit values).
template <int FMT>
__host__ __device__ constexpr int raw_words() { return FMT == FMT_I4 ? 4 : fmt_16bit(FMT) ? 16 : 8; }

// Raw words of columns 32 cc .. 32 cc + 31 of row `row` of the base tile in shared memory, as
// TMA wrote it: 128-byte rows (SW128) of 8-bit values, 64-byte rows (SW64) of nibbles, or two
// 64-column boxes of 128-byte rows (SW128) of 16-bit values.
template <int FMT>
__device__ __forceinline__ void lds_raw32(uint32_t tile, uint32_t row, int cc, uint32_t* w) {
  constexpr int NV = raw_words<FMT>() / 4;
#pragma unroll
  for (int e = 0; e < NV; ++e) {
    uint32_t addr;
    if (FMT == FMT_I4) addr = tile + swz_offset(row, cc, 64);
    else if (fmt_16bit(FMT)) addr = tile + 16384u * (cc >> 1) + swz_offset(row, 4 * (cc & 1) + e, 128);
    else addr = tile + swz_offset(row, 2 * cc + e, 128);
    const uint4 a = ld_shared_v4(addr);
    w[4 * e] = a.x, w[4 * e + 1] = a.y, w[4 * e + 2] = a.z, w[4 * e + 3] = a.w;
  }
}

// The raw words of 32 columns -> v[32] in the units of u_f.
template <int FMT>
__device__ __forceinline__ void decode32(const uint32_t* w, float (&v)[32]) {
  decode16<FMT>(w, v);
  decode16<FMT>(w + raw_words<FMT>() / 2, v + 16);
}

// Four rounded values t (u + magic) -> the bytes clip(round(u), n, p) + 64 (b <= 7), with MASK bit 7
// = 1[n <= round(u) <= p].  c + 192 lies in [128, 255] on the grid, where a bf16 is 0x43 : byte with
// byte = c + 64, so the code is formed as the exact float c + 192, cut to bf16 (exact up to 256,
// beyond the clip limits further out), clipped two at a time, and its low byte is the result: 13
// instructions per four codes where fp32 clips with an integer bias took 19 (11.3 instructions per
// weight in all; 4096 x 4096 with whole-sector stores 11.6 -> 10.8 us, with the transposed copy and masks
// 19.0 -> 16.2 us, where the separate transpose made it 20.3).  A NaN clips to n and is masked, as the fp32 clip did.
template <bool MASK>
__device__ __forceinline__ uint32_t code_bytes(const float2 (&tt)[2], const QuantParams& q, uint32_t lo, uint32_t hi) {
  uint32_t w[2], m[2];
  const float off = 192.0f - q.magic_c;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float2 c = __ffma2_rn(tt[h], make_float2(q.inv2f, q.inv2f), make_float2(off, off));
    const uint32_t x = __byte_perm(__float_as_uint(c.x), __float_as_uint(c.y), 0x7632u);
    w[h] = x;
    asm("max.bf16x2 %0, %0, %1;" : "+r"(w[h]) : "r"(lo));
    asm("min.bf16x2 %0, %0, %1;" : "+r"(w[h]) : "r"(hi));
    if (MASK) asm("set.eq.u32.bf16x2 %0, %1, %2;" : "=r"(m[h]) : "r"(w[h]), "r"(x));
  }
  uint32_t r = __byte_perm(w[0], w[1], 0x6420u);
  if (MASK) r |= __byte_perm(m[0], m[1], 0x6420u) & 0x80808080u;
  return r;
}
// 8-bit weights (codes up to 127 + bias): clipped in fp32; the bits of t are those of magic (low
// byte zero) plus the integer code, whose low byte with the bias added is the result.
__device__ __forceinline__ uint32_t code_bytes_wide(const float2 (&tt)[2], const QuantParams& q, uint32_t bias) {
  uint32_t tb[4];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    tb[2 * h] = __float_as_uint(fminf(fmaxf(tt[h].x, q.lo), q.hi)) + bias;
    tb[2 * h + 1] = __float_as_uint(fminf(fmaxf(tt[h].y, q.lo), q.hi)) + bias;
  }
  return __byte_perm(__byte_perm(tb[0], tb[1], 0x0040u), __byte_perm(tb[2], tb[3], 0x0040u), 0x5410u);
}
// Bytes b = c + 64 (0 .. 127) -> the two's complement c: bit 6 inverted, then copied into bit 7.
__device__ __forceinline__ uint32_t unbias64(uint32_t w) {
  const uint32_t x = w ^ 0x40404040u;
  return x | ((x & 0x40404040u) << 1);
}
// One 32-byte store (a whole sector; two 16-byte ones write half sectors twice).
__device__ __forceinline__ void st_global_v8(void* p, const uint32_t (&o)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(o[0]), "r"(o[1]), "r"(o[2]),
               "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7])
               : "memory");
}

// Rows r0 .. r3 of four bytes -> the four columns of four bytes.
__device__ __forceinline__ void transpose_bytes4(uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3, uint32_t (&c)[4]) {
  const uint32_t a = __byte_perm(r0, r1, 0x5140), b = __byte_perm(r0, r1, 0x7362);
  const uint32_t d = __byte_perm(r2, r3, 0x5140), e = __byte_perm(r2, r3, 0x7362);
  c[0] = __byte_perm(a, d, 0x5410);
  c[1] = __byte_perm(a, d, 0x7632);
  c[2] = __byte_perm(b, e, 0x5410);
  c[3] = __byte_perm(b, e, 0x7632);
}

// The GEMM producers' scales (and zero offsets) as bf16 rows [groups][m], spread over the
// epilogue threads of the whole grid: a launch of its own took 2-7 us.
__device__ __forceinline__ void write_scale_rows(const MergeArgs& a) {
  const int64_t n = a.m * a.s_groups, nthr = static_cast<int64_t>(gridDim.x) * (32 * NUM_EPI_WARPS);
  for (int64_t e = static_cast<int64_t>(blockIdx.x) * (32 * NUM_EPI_WARPS) + threadIdx.x; e < n; e += nthr) {
    const int64_t g = e / a.m, i = e % a.m;
    const int64_t src = i * a.s_groups + g;   // one group: s [m]
    a.s_out[e] = static_cast<uint16_t>(pack_rn_bf16x2(a.s[src], 0.0f) & 0xffffu);
    if (a.z_out) a.z_out[e] = static_cast<uint16_t>(pack_rn_bf16x2(a.z[src], 0.0f) & 0xffffu);
  }
}

__device__ __forceinline__ void write_a_transposed(const MergeArgs& a) {
  const int64_t m8 = a.m / 8, n = a.r16 * m8, nthr = static_cast<int64_t>(gridDim.x) * (32 * NUM_EPI_WARPS);
  for (int64_t e = static_cast<int64_t>(blockIdx.x) * (32 * NUM_EPI_WARPS) + threadIdx.x; e < n; e += nthr) {
    const int c = static_cast<int>(e / m8);
    const int64_t i0 = (e % m8) * 8;
    uint32_t w[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const uint32_t lo = c < a.r ? a.A[(i0 + 2 * x) * a.r + c] : 0u, hi = c < a.r ? a.A[(i0 + 2 * x + 1) * a.r + c] : 0u;
      w[x] = lo | (hi << 16);
    }
    reinterpret_cast<uint4*>(a.at_out)[e] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// Persistent: CTA b takes the 128 x 128 tiles b, b + gridDim.x, ... (column tile fastest).
// The TMA warp brings tile i's A rows, B columns and stored base into operand slot i % NSLOT, as
// many tiles ahead as there are slots; the MMA warp issues its r16 / 16 MMAs into TMEM buffer
// i % 2 (128 columns) (one thread that loaded, waited and multiplied tile by tile exposed the load
// latency of every tile: 4096 x 4096, r = 32, 12.6 -> 11.6 us); warps 0-7 turn tile i - 1's buffer into codes
// meanwhile, warp e rows 32 (e % 4) .. + 31 (TMEM lane = row) of columns 64 (e / 4) .. + 63.  A slot
// is refilled once the epilogue has read the tile's base (which is after the tile's MMAs completed).
// WIDE: 8-bit weights (floating-point bases only).
template <int FMT, bool UB, bool AMN, bool MASK, bool WIDE>
__global__ void __launch_bounds__(NUM_THREADS, 2) merge_tc_kernel(const __grid_constant__ CUtensorMap tm_a,
                                                               const __grid_constant__ CUtensorMap tm_b,
                                                               const __grid_constant__ CUtensorMap tm_phi,
                                                               const MergeArgs args) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * MAX_SLOTS + 5];   // FULL[4], SEMPTY[4], LFULL[2], LEMPTY[2], DRAIN
  __shared__ uint32_t tmem_base_s;
  __shared__ volatile int abort_s;
  const uint32_t smem = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto bar = [&](int i) { return smem_u32(&bars[i]); };
  constexpr int B_FULL = 0, B_SEMPTY = MAX_SLOTS, B_LFULL = 2 * MAX_SLOTS, B_LEMPTY = B_LFULL + 2,
                B_DRAIN = B_LEMPTY + 2;
  const int r16 = args.r16;
  const int nslot = num_slots(r16, AMN, FMT);
  const int64_t nkb = args.k / 128;
  const int64_t num_tiles = (args.m / 128) * nkb;
  if (threadIdx.x == 0) {
    abort_s = 0;
    for (uint32_t i = 0; i < MAX_SLOTS; ++i) {
      mbar_init(bar(B_FULL + i), 1);
      mbar_init(bar(B_SEMPTY + i), NUM_EPI_WARPS);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(B_LFULL + i), 1);
      mbar_init(bar(B_LEMPTY + i), NUM_EPI_WARPS);
    }
    mbar_init(bar(B_DRAIN), 1);
    mbar_fence_init();
  }
  if (warp == MMA_WARP) tmem_alloc(smem_u32(&tmem_base_s), TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_launch();
  const uint32_t tmem = tmem_base_s;
  const WaitCtl ctl{&abort_s, args.status, args.timeout_ns};

  const uint32_t rbox = 128u * static_cast<uint32_t>(r16);   // one r16-row x 64-column box
  const uint32_t off_b = a_tile_bytes(r16, AMN), sbytes = slot_bytes(r16, AMN, FMT);
  const uint32_t off_phi = off_b + 2u * rbox;
  if (warp == TMA_WARP) {
    // ------------------------------------------------------------ TMA
    if (lane == 0) {
      prefetch_tensormap(&tm_a);
      prefetch_tensormap(&tm_b);
      prefetch_tensormap(&tm_phi);
      uint32_t i = 0;
      for (int64_t t = blockIdx.x; t < num_tiles; t += gridDim.x, ++i) {
        const int64_t rb = t / nkb, cb = t % nkb;
        const uint32_t sl = i % nslot, su = i / nslot;
        const uint32_t sa = smem + sl * sbytes;
        if (!wait_spin_bounded(bar(B_SEMPTY + sl), (su & 1u) ^ 1u, ctl, 1)) break;
        mbar_arrive_expect_tx(bar(B_FULL + sl), sbytes);
        // the base first: the longest way to come
        if (fmt_16bit(FMT)) {
          tma_load_2d(sa + off_phi, &tm_phi, static_cast<int32_t>(cb * 128), static_cast<int32_t>(rb * 128),
                      bar(B_FULL + sl));
          tma_load_2d(sa + off_phi + 16384u, &tm_phi, static_cast<int32_t>(cb * 128 + 64),
                      static_cast<int32_t>(rb * 128), bar(B_FULL + sl));
        } else {
          tma_load_2d(sa + off_phi, &tm_phi, static_cast<int32_t>(FMT == FMT_I4 ? cb * 64 : cb * 128),
                      static_cast<int32_t>(rb * 128), bar(B_FULL + sl));
        }
        if (AMN) {
          tma_load_2d(sa, &tm_a, static_cast<int32_t>(rb * 128), 0, bar(B_FULL + sl));
          tma_load_2d(sa + rbox, &tm_a, static_cast<int32_t>(rb * 128 + 64), 0, bar(B_FULL + sl));
        } else {
          for (int kb = 0; kb < (r16 + 63) / 64; ++kb)
            tma_load_2d(sa + 16384u * kb, &tm_a, 64 * kb, static_cast<int32_t>(rb * 128), bar(B_FULL + sl));
        }
        tma_load_2d(sa + off_b, &tm_b, static_cast<int32_t>(cb * 128), 0, bar(B_FULL + sl));
        tma_load_2d(sa + off_b + rbox, &tm_b, static_cast<int32_t>(cb * 128 + 64), 0, bar(B_FULL + sl));
      }
      // every issued copy lands before the shared memory is released (already so unless a wait
      // gave up): the last use of each slot
      for (uint32_t x = i > static_cast<uint32_t>(nslot) ? i - nslot : 0; x < i; ++x)
        drain_wait(bar(B_FULL + x % nslot), (x / nslot) & 1u, args.timeout_ns);
    }
  } else if (warp == MMA_WARP) {
    // ------------------------------------------------------------ MMA
    if (lane == 0) {
      // A K-major: 32 bytes per 16-element K step inside a box of a_box_cols rank columns, one box
      // (16 KB) per 64 ranks; A and B MN-major: two 64-wide atoms (LBO = one box), 16 rank rows =
      // 2048 bytes per K step.
      const uint32_t idesc = make_idesc_bf16(128, 128, AMN ? 1 : 0, 1);
      const uint32_t acols = static_cast<uint32_t>(a_box_cols(r16));
      const uint32_t a_swz = acols == 64 ? SWZ_128B : acols == 32 ? SWZ_64B : SWZ_32B;
      uint32_t i = 0;
      for (int64_t t = blockIdx.x; t < num_tiles; t += gridDim.x, ++i) {
        const uint32_t sl = i % nslot, su = i / nslot, b = i & 1u, bu = i >> 1;
        const uint32_t sa = smem + sl * sbytes;
        if (!wait_spin_bounded(bar(B_FULL + sl), su & 1u, ctl, 2)) break;
        if (!wait_spin_bounded(bar(B_LEMPTY + b), (bu & 1u) ^ 1u, ctl, 3)) break;
        tc_fence_after();
        const uint64_t db = make_sdesc(sa + off_b, rbox, 1024, SWZ_128B);
        for (int ks = 0; ks < r16 / 16; ++ks) {
          const uint64_t da = AMN ? make_sdesc(sa + 2048u * ks, rbox, 1024, SWZ_128B)
                                  : make_sdesc(sa + 16384u * (ks >> 2) + 32u * (ks & 3), 16, 16u * acols, a_swz);
          mma_bf16(tmem + 128u * b, da, db + 128 * ks, idesc, ks > 0 ? 1u : 0u);
        }
        mma_commit(bar(B_LFULL + b));     // the low-rank tile is ready
      }
      // every MMA has completed before the shared memory and TMEM are released
      mma_commit(bar(B_DRAIN));
      drain_wait(bar(B_DRAIN), 0, args.timeout_ns);
    }
  } else {
    // ------------------------------------------------------------ epilogue
    if (args.s_out != nullptr) write_scale_rows(args);
    if (args.at_out != nullptr) write_a_transposed(args);
    constexpr int NW = raw_words<FMT>();
    const QuantParams q = args.q;
    const uint32_t lr2 = pack_rn_bf16x2(q.lr_scale, q.lr_scale);   // exact: a power of two when UB
    // bf16(n + 192) and bf16(p + 192) in both halves: 0x43 : n + 64 and 0x43 : p + 64
    const int half_range = 1 << (args.bits - 1);
    const uint32_t clip_lo = (0x4300u | static_cast<uint32_t>((64 - half_range) & 0x7f)) * 0x10001u;
    const uint32_t clip_hi = (0x4300u | static_cast<uint32_t>((63 + half_range) & 0x7f)) * 0x10001u;
    const bool wz32 = (reinterpret_cast<uintptr_t>(args.wz) & 31u) == 0;
    const int quarter = warp & 3, half = warp >> 2;                // TMEM lanes, 64-column half
    const uint32_t lane_off = static_cast<uint32_t>(32 * quarter) << 16;
    const uint32_t r_in = 32 * quarter + lane;   // this thread's row inside a tile
    const uint32_t stage = smem + nslot * sbytes + warp * (32u * STG_ROW * 4u);
    bool ok = true;
    uint32_t i = 0;
    for (int64_t t = blockIdx.x; t < num_tiles; t += gridDim.x, ++i) {
      const int64_t row0 = (t / nkb) * 128, row = row0 + r_in;
      const int64_t colt = (t % nkb) * 128;
      const uint32_t b = i & 1u, bu = i >> 1, sl = i % nslot;
      const uint32_t phi_tile = smem + sl * sbytes + off_phi;
      // the tile's MMAs completed, so its operands (and base) are in the slot
      ok = wait_bounded(bar(B_LFULL + b), bu & 1u, ctl, 4);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
#pragma unroll
      for (int c2 = 0; c2 < 2; ++c2) {
        const int cc = 2 * half + c2;
        float v[32], L[32];
        uint32_t raw[NW];
        lds_raw32<FMT>(phi_tile, r_in, cc, raw);
        tmem_ld32(tmem + lane_off + 128u * b + 32u * cc, L);
        decode32<FMT>(raw, v);
        tmem_ld_wait();
        if (c2 == 1) {
          // the tile's last reads of the TMEM buffer
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(B_LEMPTY + b));
        }
        uint32_t o[8];
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          float2 tt[2];   // u + magic: u rounded half to even in units of 2^f
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int j = 4 * g + 2 * h;
            const float2 u = UB ? u_bf16x2(L[j], L[j + 1], v[j], v[j + 1], lr2)
                                : __ffma2_rn(make_float2(L[j], L[j + 1]), make_float2(q.lr_scale, q.lr_scale),
                                             make_float2(v[j], v[j + 1]));
            tt[h] = __fadd2_rn(u, make_float2(q.magic, q.magic));
          }
          o[g] = WIDE ? code_bytes_wide(tt, q, args.code_bias) : code_bytes<MASK>(tt, q, clip_lo, clip_hi);
        }
        if (args.wz != nullptr) {
          if (!WIDE && args.code_bias == 0) {
#pragma unroll
            for (int g = 0; g < 8; ++g) o[g] = unbias64(o[g]);
          }
          int8_t* dst = args.wz + row * args.k + colt + 32 * cc;
          if (wz32) {
            st_global_v8(dst, o);
          } else {
            reinterpret_cast<uint4*>(dst)[0] = make_uint4(o[0], o[1], o[2], o[3]);
            reinterpret_cast<uint4*>(dst)[1] = make_uint4(o[4], o[5], o[6], o[7]);
          }
        }
        if (args.wt != nullptr) {
          // lane (w, ib) takes the words w (columns 4 w .. 4 w + 3) of rows 8 ib .. 8 ib + 7 and
          // writes them as four 8-byte pieces of transposed rows (4 lanes cover 32 bytes of one)
          __syncwarp();   // the previous block's reads are done
#pragma unroll
          for (int w = 0; w < 8; ++w)
            st_shared_u32(stage + (lane * STG_ROW + w) * 4u, MASK ? o[w] & 0x7f7f7f7fu : o[w]);
          __syncwarp();
          const int w = lane >> 2, ib = lane & 3;
          uint32_t x[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) x[e] = ld_shared_u32(stage + ((8 * ib + e) * STG_ROW + w) * 4u);
          uint32_t lo[4], hi[4];
          transpose_bytes4(x[0], x[1], x[2], x[3], lo);
          transpose_bytes4(x[4], x[5], x[6], x[7], hi);
          int8_t* dst = args.wt + (colt + 32 * cc + 4 * w) * args.m + row0 + 32 * quarter + 8 * ib;
#pragma unroll
          for (int e = 0; e < 4; ++e) *reinterpret_cast<uint2*>(dst + e * args.m) = make_uint2(lo[e], hi[e]);
        }
      }
      // The slot may be refilled.  Reported after the stores of what was read from it: an arrive
      // issued right after the reads overtook them while they queued behind the previous block's
      // global stores, and the next copy then landed under them.
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(B_SEMPTY + sl));
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == MMA_WARP) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

template <int FMT, bool UB, bool AMN, bool MASK, bool WIDE = false>
cudaError_t launch_merge_one(const CUtensorMap& tm_a, const CUtensorMap& tm_b, const CUtensorMap& tm_phi,
                             const MergeArgs& args, cudaStream_t stream) {
  static bool configured[kMaxDevices] = {};
  const cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(merge_tc_kernel<FMT, UB, AMN, MASK, WIDE>),
                                         static_cast<int>(MAX_SMEM_BYTES), configured);
  if (e != cudaSuccess) return e;
  static int sms[kMaxDevices] = {};
  int dev = 0;
  cudaError_t e2 = cudaGetDevice(&dev);
  if (e2 != cudaSuccess) return e2;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (sms[dev] == 0) {
    e2 = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e2 != cudaSuccess) return e2;
  }
  const int64_t tiles = (args.m / 128) * (args.k / 128);
  const uint32_t smem = smem_bytes(args.r16, AMN, FMT);
  const int64_t per_sm = 232448 / smem >= 2 ? 2 : 1;
  const int64_t grid = tiles < per_sm * sms[dev] ? tiles : per_sm * sms[dev];
  merge_tc_kernel<FMT, UB, AMN, MASK, WIDE><<<static_cast<unsigned>(grid), NUM_THREADS, smem, stream>>>(tm_a, tm_b, tm_phi, args);
  return cudaGetLastError();
}

template <int FMT, bool UB>
cudaError_t launch_merge_fmt(int a_mn, const CUtensorMap& tm_a, const CUtensorMap& tm_b, const CUtensorMap& tm_phi,
                             const MergeArgs& args, cudaStream_t stream) {
  if (args.bits > 7) {
    if constexpr (fmt_float(FMT))
      return a_mn ? launch_merge_one<FMT, UB, true, false, true>(tm_a, tm_b, tm_phi, args, stream)
                  : launch_merge_one<FMT, UB, false, false, true>(tm_a, tm_b, tm_phi, args, stream);
    return cudaErrorInvalidValue;
  }
  if (args.mask_bit)
    return a_mn ? launch_merge_one<FMT, UB, true, true>(tm_a, tm_b, tm_phi, args, stream)
                : launch_merge_one<FMT, UB, false, true>(tm_a, tm_b, tm_phi, args, stream);
  return a_mn ? launch_merge_one<FMT, UB, true, false>(tm_a, tm_b, tm_phi, args, stream)
              : launch_merge_one<FMT, UB, false, false>(tm_a, tm_b, tm_phi, args, stream);
}

template <bool UB>
cudaError_t launch_merge_ub(int fmt, int a_mn, const CUtensorMap& tm_a, const CUtensorMap& tm_b,
                            const CUtensorMap& tm_phi, const MergeArgs& args, cudaStream_t stream) {
  switch (fmt) {
    case FMT_Q8: return launch_merge_fmt<FMT_Q8, UB>(a_mn, tm_a, tm_b, tm_phi, args, stream);
    case FMT_I4: return launch_merge_fmt<FMT_I4, UB>(a_mn, tm_a, tm_b, tm_phi, args, stream);
    case FMT_BF16: return launch_merge_fmt<FMT_BF16, UB>(a_mn, tm_a, tm_b, tm_phi, args, stream);
    case FMT_F16:
      return UB ? cudaErrorInvalidValue : launch_merge_fmt<FMT_F16, false>(a_mn, tm_a, tm_b, tm_phi, args, stream);
    case FMT_E4M3: return launch_merge_fmt<FMT_E4M3, UB>(a_mn, tm_a, tm_b, tm_phi, args, stream);
    case FMT_E5M2: return launch_merge_fmt<FMT_E5M2, UB>(a_mn, tm_a, tm_b, tm_phi, args, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

static_assert(smem_bytes(256, true, FMT_BF16) <= MAX_SMEM_BYTES && smem_bytes(256, false, FMT_BF16) <= MAX_SMEM_BYTES,
              "smem budget");
static_assert(num_slots(32, true, FMT_Q8) == 3 && num_slots(32, false, FMT_Q8) == 3 && num_slots(256, true, FMT_BF16) == 1, "operand slots");

cudaError_t launch_merge_tc(int fmt, int u_bf16, int a_mn, const CUtensorMap& tm_a, const CUtensorMap& tm_b,
                            const CUtensorMap& tm_phi, const MergeArgs& args, cudaStream_t stream) {
  if (args.m % 128 || args.k % 128 || args.r16 < 16 || args.r16 > 256 || (args.r16 & 15)) return cudaErrorInvalidValue;
  // the byte's top bit must be free; codes of 7 bits are stored plus 64 or plain
  if (args.mask_bit && args.code_bias != 64) return cudaErrorInvalidValue;
  if (args.bits <= 7 && args.code_bias != 64 && args.code_bias != 0) return cudaErrorInvalidValue;
  return u_bf16 ? launch_merge_ub<true>(fmt, a_mn, tm_a, tm_b, tm_phi, args, stream)
                : launch_merge_ub<false>(fmt, a_mn, tm_a, tm_b, tm_phi, args, stream);
}

}  // namespace lrqat
