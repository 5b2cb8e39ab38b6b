// Fused weight-gradient kernel on CTA pairs over the codes of the codes pass (any rank, m and k
// multiples of 256).  For a tile of 256 weight rows i x 256 columns j and a range of tokens
//   G = dY^T X_hat                 (tcgen05, fp32 accumulator in TMEM, never stored)
// and, in the epilogue, the straight-through gradients of Eq. 8 from the code byte of every weight
// (c + 64, bit 7 = the clip mask M):
//   dU = G * s * M,  dA_partial = dU B^T,  dB^T_partial = dU^T A,  ds_partial = sum_j G * c.
//
// Against the kernel that recomputes the low-rank tile (dw_pair.cu): a unit's epilogue there is
// a chain per 128-column chunk (load operands, low-rank MMA, dU, contractions, the next chunk's
// dU into the same buffer), and G, which the next unit's main loop waits for, is held through it:
// about 16,000 cycles per unit.  The codes need no low-rank tile: their bytes go from global
// memory to registers before G is complete, so the shared memory of its operands holds dU of both
// chunks, the element work of the whole tile runs in one go and G is free after it; the
// contractions then run beside the next unit's main loop.
// Measured, dW of a 4096 x 4096 layer at T = 8192, r = 32: 185.8 us with the low-rank tile -> 168.5;
// 13824 x 5120 at T = 16384 (under the power cap) 1421 -> 1350 us; 4096 x 14336 g128 590 -> 538 us.
//
// Every MMA is a pair MMA (a kernel may not mix one-SM and pair MMAs):
//   G:    M = 256 rows i, N = 256 columns j (each CTA holds 128 of the X columns), K = tokens
//         (4 K steps of 16 per 64-token stage);
//   dB^T: of a 128-column chunk and a round of R ranks (R = r16 up to 64, then 64): M = 256 with
//         rows = the chunk's columns j of each CTA's dU^T, N = 2 R with each CTA supplying the
//         A^T rows of its own 128 weight rows, K = 128 weight rows; a CTA's partial over its own rows
//         is in columns R * rank .. of its lanes (the other R mix rows of both CTAs);
//   dA:   of a round: M = 256 rows i, N = R (each CTA holds half of the ranks of B), K = 256 columns j.
// These three jobs per round take turns in two 128-column TMEM buffers, so the epilogue warps write
// one job's partials out while the next job's MMAs run.  The partials are laid out as in
// dw_pair.cu (dB per 128-row block), so the same reduction sums them, and every G has its tokens in
// the same order as there (ranks above 64: as in dw.cu), so dU is the same bit for bit.
//
// Roles (480 threads per CTA): warp 0 loads the factors of the rounds, warp 1 owns TMEM and (in
// the leader, rank 0) issues the main loop's MMAs, warps 2..9 run the epilogue, warps 10..13
// fill the stages (one box of every stage each), warp 14 (in the leader) issues the jobs' MMAs.
// Loads that the MMAs read complete on the leader's barriers (both CTAs' bytes); the leader waits
// for the peer's "dU written", "G read" and "buffer drained" events, which each peer warp reports
// with a 16-byte copy into the leader's shared memory.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "kernels.h"
#include "ptx.cuh"
#include "quant.cuh"

namespace lrqat {
namespace {

constexpr int NS = 4;
constexpr int BKT = 64;                        // tokens per pipeline stage
constexpr int NUM_EPI_WARPS = 8;
constexpr int NUM_LOADERS = 4;                 // one per box of a stage
constexpr int FIRST_LOADER = 2 + NUM_EPI_WARPS;
constexpr int JOB_MMA_WARP = FIRST_LOADER + NUM_LOADERS;   // the leader's contraction MMAs
constexpr int NUM_THREADS = 32 * (JOB_MMA_WARP + 1);
constexpr uint32_t SIG_TX = 16u * NUM_EPI_WARPS;   // bytes of the peer's per-warp signals

constexpr uint32_t BOX_BYTES = 64 * BKT * 2;   // one 64-column x 64-token bf16 box (SW128)
constexpr uint32_t STAGE_DY = 2 * BOX_BYTES;   // this CTA's 128 rows i
constexpr uint32_t STAGE_BYTES = STAGE_DY + 2 * BOX_BYTES;   // + its 128 of the 256 columns j
constexpr uint32_t OFF_STAGES = 0;
// A^T [R rank rows, this CTA's 128 rows i] (2 boxes of 64 i): this CTA's half of the N = 2 R rows of
// the dB^T jobs' B operand (K-major).
constexpr uint32_t OFF_AT = OFF_STAGES + NS * STAGE_BYTES;
// B [this CTA's R / 2 ranks, the tile's 256 columns] (4 boxes of 64 columns): B operand of the dA
// job (K-major).
constexpr uint32_t OFF_B = OFF_AT + 16384;
constexpr uint32_t OFF_DU = OFF_B + 16384;     // dU: 2 chunks x 2 atom columns of 128 rows x 128 B
constexpr uint32_t SMEM_TILES = OFF_DU + 65536;
constexpr uint32_t SMEM_BYTES = SMEM_TILES + 1024;
static_assert(SMEM_BYTES + 1024 <= 232448, "shared memory budget");
static_assert(OFF_AT % 1024 == 0 && OFF_B % 1024 == 0 && OFF_DU % 1024 == 0,
              "swizzled tiles start on 1024-byte boundaries");

constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t COL_G = 0;      // 256 columns
constexpr uint32_t COL_JOB = 256;  // two job buffers of 128 columns

constexpr int BAR_FULL = 0;                    // leader: both CTAs' stage landed
constexpr int BAR_EMPTY = BAR_FULL + NS;       // both: the stage's MMAs finished
constexpr int BAR_EFFULL = BAR_EMPTY + NS;     // leader: both CTAs' factors of the round landed
constexpr int BAR_EFEMPTY = BAR_EFFULL + 1;    // both: the round's MMAs finished
constexpr int BAR_ACCFULL = BAR_EFEMPTY + 1;   // both: G complete
constexpr int BAR_ACCEMPTY = BAR_ACCFULL + 1;  // leader: both CTAs read G
constexpr int BAR_DUFULL = BAR_ACCEMPTY + 1;   // leader: both CTAs wrote dU of the unit
constexpr int BAR_DUEMPTY = BAR_DUFULL + 1;    // both: the unit's jobs finished
constexpr int BAR_JFULL = BAR_DUEMPTY + 1;     // both: the job of the buffer finished (2)
constexpr int BAR_JEMPTY = BAR_JFULL + 2;      // leader: both CTAs wrote the buffer out (2)
constexpr int BAR_DRAIN = BAR_JEMPTY + 2;      // the main-loop MMAs' last completion
constexpr int BAR_DRAIN_J = BAR_DRAIN + 1;     // the jobs' last completion
constexpr int NUM_BARS = BAR_DRAIN_J + 1;

__device__ __forceinline__ void drain_wait(uint32_t bar, uint32_t parity, uint64_t timeout_ns) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > timeout_ns) break;
  }
}

struct Unit {
  int ib, jt, sp, t0, nsteps;   // ib: 256-row block of the pair
  int rev;                      // stages in descending token order
  int half_last;                // the last stage holds 32 tokens of the unit (an odd multiple of 32)
  uint32_t keep;                // the 128 x 128 tiles that the unit writes (bit 2 r + c; wide plan)
};

__device__ __forceinline__ Unit decode_unit(int u, const DwArgs& a) {
  Unit x;
  x.ib = u % a.ni;
  x.jt = (u / a.ni) % a.nj;
  x.sp = u / (a.ni * a.nj);
  x.t0 = x.sp * a.tchunk;
  int t1 = x.t0 + a.tchunk;
  if (t1 > a.T) t1 = a.T;
  x.nsteps = (t1 - x.t0 + BKT - 1) / BKT;
  // the splits of ranks above 64 are multiples of 32 tokens: what follows in the stage's box
  // belongs to the next split
  x.half_last = (t1 - x.t0 + 31) / 32 & 1;
  x.keep = 15u;
  x.rev = 0;
  return x;
}

// Whole pair tile number u in processing order: groups of kColGroup column tiles with the
// column tile varying fastest (as in dw.cu).
constexpr int64_t kColGroup = 8;
__device__ __forceinline__ void dw_whole_tile(int64_t u, int ni, int64_t full_tiles, int& ib, int& jt) {
  const int64_t grouped = full_tiles / ni / kColGroup * kColGroup * ni;
  if (u < grouped) {
    const int64_t grp = u / (kColGroup * ni), r = u % (kColGroup * ni);
    jt = static_cast<int>(grp * kColGroup + r % kColGroup);
    ib = static_cast<int>(r / kColGroup);
  } else {
    ib = static_cast<int>(u % ni);
    jt = static_cast<int>(u / ni);
  }
}

// This pair's units (equal token splits, round robin over the pairs), or (tail schedule) its
// whole tiles of the full waves followed by its one part of a tail tile.
struct WorkIter {
  int64_t u;
  bool tail;
  int64_t st, st_u;   // wide plan: the tile that holds unit u or one before it, and its first unit
};

__device__ __forceinline__ WorkIter work_begin(const DwArgs& a, int pair) {
  return {static_cast<int64_t>(pair), a.sched.tail != 0 && pair < a.sched.tail_grid, a.sched.full_tiles,
          a.sched.full_tiles};
}

template <bool WIDE>
__device__ __forceinline__ bool work_next(WorkIter& it, const DwArgs& a, int pair, int npairs, Unit& x) {
  // Odd waves run their stages in descending token order: a wave shares its column (or row) blocks
  // with the wave before it, whose last stages are then still in L2 when it starts.
  if (!a.sched.tail) {
    if (it.u >= a.num_units) return false;
    x = decode_unit(static_cast<int>(it.u), a);
    x.rev = WIDE || a.r16 > 64 ? 0 : static_cast<int>((it.u / npairs) & 1);
    it.u += npairs;
    return true;
  }
  if (it.u < a.sched.full_tiles) {
    dw_whole_tile(it.u, a.ni, a.sched.full_tiles, x.ib, x.jt);
    x.sp = 0;
    x.t0 = 0;
    x.nsteps = static_cast<int>(a.sched.tsteps);
    x.half_last = 0;
    x.keep = 15u;
    x.rev = WIDE || a.r16 > 64 ? 0 : static_cast<int>((it.u / npairs) & 1);
    it.u += npairs;
    return true;
  }
  if (WIDE) {
    // the tiles past the leading whole column tiles, in order, each with its passes
    const int64_t tiles = static_cast<int64_t>(a.ni) * a.nj;
    for (; it.st < tiles; ++it.st) {
      int q[3];
      uint32_t keep[3];
      x.ib = static_cast<int>(it.st % a.ni);
      x.jt = static_cast<int>(it.st / a.ni);
      const int n = wide_passes(x.ib, x.jt, 2 * a.ni, a.base, q, keep);
      int64_t p = it.u - it.st_u;   // which pass of this tile, if it is one
      x.sp = static_cast<int>(p);
      for (int y = 0; y < n; ++y) {
        if (p < q[y]) {
          const int64_t s0 = p * a.base.tsteps / q[y], s1 = (p + 1) * a.base.tsteps / q[y];   // 32-token stages
          x.t0 = static_cast<int>(s0 * 32);
          x.nsteps = static_cast<int>((s1 - s0 + 1) / 2);
          x.half_last = static_cast<int>((s1 - s0) & 1);
          x.rev = 0;
          x.keep = keep[y];
          it.u += npairs;
          return true;
        }
        p -= q[y];
      }
      it.st_u = it.u - p;
    }
    return false;
  }
  if (!it.tail) return false;
  it.tail = false;
  int64_t t;
  int j, q;
  dw_tail_part(pair, a.sched, t, j, q);
  const int64_t tile = a.sched.full_tiles + t;
  const int64_t s0 = j * a.sched.tsteps / q, s1 = (j + 1) * a.sched.tsteps / q;
  x.ib = static_cast<int>(tile % a.ni);
  x.jt = static_cast<int>(tile / a.ni);
  x.sp = j;
  x.t0 = static_cast<int>(s0 * BKT);
  x.nsteps = static_cast<int>(s1 - s0);
  x.half_last = 0;
  x.keep = 15u;
  x.rev = 0;
  return true;
}

// WIDE: the wide plan of ranks above 64 (its pass bookkeeping costs registers: 169 -> 178 us where it
// was compiled into every launch).
template <bool ZP, bool WIDE>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    dw_codes_kernel(const __grid_constant__ CUtensorMap tm_dy, const __grid_constant__ CUtensorMap tm_x,
                    const __grid_constant__ CUtensorMap tm_at, const __grid_constant__ CUtensorMap tm_b,
                    const DwArgs args) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[NUM_BARS];
  __shared__ __align__(16) uint32_t sig_buf[8];   // [0, 4): source of the peer's signals, [4, 8): their target
  __shared__ uint32_t tmem_base_s;
  __shared__ volatile int abort_s;

  const uint32_t smem = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_cta_rank();
  const bool leader = rank == 0;
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  auto bar = [&](int i) { return smem_u32(&bars[i]); };
  auto lbar = [&](int i) { return map_shared_rank(smem_u32(&bars[i]), 0); };   // the leader's copy
  constexpr int BN = 256;
  const int R = args.r16 < 64 ? args.r16 : 64;       // ranks per round
  const int rounds = (args.r16 + 63) / 64;
  const uint32_t abox = static_cast<uint32_t>(R) * 128u;   // bytes of one R-row x 64-column box
  const uint32_t bbox = abox / 2;                          // bytes of one R/2-row x 64-column box
  const int ni128 = 2 * args.ni;                           // 128-row blocks

  if (threadIdx.x == 0) {
    abort_s = 0;
    for (int s = 0; s < NS; ++s) {
      mbar_init(bar(BAR_FULL + s), 1);
      mbar_init(bar(BAR_EMPTY + s), 1);
    }
    mbar_init(bar(BAR_EFFULL), 1);
    mbar_init(bar(BAR_EFEMPTY), 1);
    mbar_init(bar(BAR_ACCFULL), 1);
    mbar_init(bar(BAR_ACCEMPTY), NUM_EPI_WARPS);
    mbar_init(bar(BAR_DUFULL), NUM_EPI_WARPS);
    mbar_init(bar(BAR_DUEMPTY), 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar(BAR_JFULL + b), 1);
      mbar_init(bar(BAR_JEMPTY + b), NUM_EPI_WARPS);
    }
    mbar_init(bar(BAR_DRAIN), 1);
    mbar_init(bar(BAR_DRAIN_J), 1);
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc_pair(smem_u32(&tmem_base_s), TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // both CTAs' barriers exist before either signals the other
  tc_fence_after();
  griddep_launch();
  griddep_wait();   // no global memory is touched above
  const uint32_t tmem = tmem_base_s;
  const WaitCtl ctl{&abort_s, args.status, args.timeout_ns};
  const uint32_t sig_src = smem_u32(&sig_buf[0]);
  const uint32_t sig_dst_leader = map_shared_rank(smem_u32(&sig_buf[4]), 0);

  if (warp == 0) {
    // ------------------------------------------------- factors of the rank rounds
    if (lane == 0) {
      prefetch_tensormap(&tm_at);
      prefetch_tensormap(&tm_b);
      uint32_t n = 0;   // rounds so far
      bool ok = true;
      WorkIter wi = work_begin(args, pair);
      Unit w;
      while (ok && work_next<WIDE>(wi, args, pair, npairs, w)) {
        if (args.sched.tail && w.sp == 0) {   // the reduction reads which slots hold data
          const int64_t tile2 = w.ib + static_cast<int64_t>(args.ni) * w.jt;
          int segs;
          if (WIDE) {
            int q[3];
            uint32_t keep[3];
            const int n = wide_passes(w.ib, w.jt, ni128, args.base, q, keep);
            segs = q[0] + (n > 1 ? q[1] : 0) + (n > 2 ? q[2] : 0);
          } else {
            segs = dw_tile_segments(tile2, args.sched);
          }
          args.tile_segs[(2 * w.ib + static_cast<int>(rank)) + static_cast<int64_t>(ni128) * w.jt] = segs;
        }
        const int i_own = w.ib * 256 + static_cast<int>(rank) * 128, j0 = w.jt * BN;
        for (int rc = 0; rc < rounds; ++rc, ++n) {
          if (!(ok = wait_spin_bounded(bar(BAR_EFEMPTY), (n & 1u) ^ 1u, ctl, 2))) break;
          if (leader) mbar_arrive_expect_tx(bar(BAR_EFFULL), 2u * (2u * abox + 4u * bbox));
          const int ra = 64 * rc, rb = 64 * rc + static_cast<int>(rank) * (R / 2);
          tma_load_2d_pair(smem + OFF_AT, &tm_at, i_own, ra, lbar(BAR_EFFULL));
          tma_load_2d_pair(smem + OFF_AT + abox, &tm_at, i_own + 64, ra, lbar(BAR_EFFULL));
#pragma unroll
          for (int x = 0; x < 4; ++x)
            tma_load_2d_pair(smem + OFF_B + x * bbox, &tm_b, j0 + 64 * x, rb, lbar(BAR_EFFULL));
        }
      }
    }
  } else if (warp >= FIRST_LOADER && warp < FIRST_LOADER + NUM_LOADERS) {
    // ------------------------------------------------ pipeline stage loaders
    // Loader b issues box b of every stage (boxes 0-1: this CTA's dY columns i, boxes 2-3: its X
    // columns j): one warp's copies are handled one after another.  Loader 0 of the leader announces
    // the stage's bytes.
    const int b = warp - FIRST_LOADER;
    if (lane == 0) {
      if (b < 2) prefetch_tensormap(&tm_dy);
      else prefetch_tensormap(&tm_x);
      uint32_t g = 0;
      bool ok = true;
      WorkIter wi = work_begin(args, pair);
      Unit w;
      while (ok && work_next<WIDE>(wi, args, pair, npairs, w)) {
        const int i_own = w.ib * 256 + static_cast<int>(rank) * 128;
        const int j_own = w.jt * BN + static_cast<int>(rank) * 128;
        for (int step = 0; step < w.nsteps; ++step, ++g) {
          const uint32_t s = g % NS, ph = (g / NS) & 1u;
          if (!(ok = wait_spin_bounded(bar(BAR_EMPTY + s), ph ^ 1u, ctl, 1))) break;
          const uint32_t st = smem + OFF_STAGES + s * STAGE_BYTES;
          const uint32_t fb = lbar(BAR_FULL + s);
          if (b == 0 && leader) mbar_arrive_expect_tx(bar(BAR_FULL + s), 2u * STAGE_BYTES);
          const int tok = w.t0 + (w.rev ? w.nsteps - 1 - step : step) * BKT;
          if (b < 2) tma_load_2d_pair(st + b * BOX_BYTES, &tm_dy, i_own + 64 * b, tok, fb);
          else tma_load_2d_pair(st + STAGE_DY + (b - 2) * BOX_BYTES, &tm_x, j_own + 64 * (b - 2), tok, fb);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------ MMA issuer (the leader's)
    if (lane == 0 && leader) {
      const uint32_t idesc_g = make_idesc_bf16(256, BN, 1, 1);
      const uint64_t d_dy0 = make_sdesc(smem + OFF_STAGES, BOX_BYTES, 1024, SWZ_128B);
      const uint64_t d_x0 = make_sdesc(smem + OFF_STAGES + STAGE_DY, BOX_BYTES, 1024, SWZ_128B);
      const uint32_t b_full = bar(BAR_FULL);
      uint32_t it = 0;
      uint32_t s = 0, ph = 0;   // stage and phase of the global step
      bool ok = true;
      WorkIter wi = work_begin(args, pair);
      Unit w;
      while (ok && work_next<WIDE>(wi, args, pair, npairs, w)) {
        if (!(ok = wait_spin_bounded(bar(BAR_ACCEMPTY), (it & 1u) ^ 1u, ctl, 4))) break;
        tc_fence_after();
        for (int step = 0; step < w.nsteps; ++step) {
          if (!(ok = wait_spin_bounded(b_full + 8u * s, ph, ctl, 5))) break;
          tc_fence_after();
          const uint64_t a = d_dy0 + s * (STAGE_BYTES >> 4), b = d_x0 + s * (STAGE_BYTES >> 4);
          const bool whole = !w.half_last || (w.rev ? step > 0 : step + 1 < w.nsteps);
          // 16-token K steps: 16 rows of 128 bytes
          mma_bf16_pair(tmem + COL_G, a, b, idesc_g, step > 0 ? 1u : 0u);
          mma_bf16_pair(tmem + COL_G, a + 128, b + 128, idesc_g, 1u);
          if (whole) {
            mma_bf16_pair(tmem + COL_G, a + 256, b + 256, idesc_g, 1u);
            mma_bf16_pair(tmem + COL_G, a + 384, b + 384, idesc_g, 1u);
          }
          mma_commit_pair(bar(BAR_EMPTY + s));
          if (++s == NS) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!ok) break;
        mma_commit_pair(bar(BAR_ACCFULL));
        ++it;
      }
      // the peer's last drain report lands before the CTAs end
      if (ok) ok = wait_spin_bounded(bar(BAR_ACCEMPTY), (it & 1u) ^ 1u, ctl, 14);
      mma_commit_pair_self(bar(BAR_DRAIN));
      drain_wait(bar(BAR_DRAIN), 0, args.timeout_ns);
    }
  } else if (warp == JOB_MMA_WARP) {
    // -------------------------------------------- contraction MMAs (the leader's)
    if (lane == 0 && leader) {
      const uint32_t idesc_da = make_idesc_bf16(256, R, 0, 0);
      const uint32_t idesc_db = make_idesc_bf16(256, 2 * R, 1, 0);
      uint32_t it = 0, n = 0, job = 0;
      bool ok = true;
      WorkIter wi = work_begin(args, pair);
      Unit w;
      while (ok && work_next<WIDE>(wi, args, pair, npairs, w)) {
        if (!(ok = wait_spin_bounded(bar(BAR_DUFULL), it & 1u, ctl, 8))) break;
        for (int rc = 0; rc < rounds && ok; ++rc, ++n) {
          if (!(ok = wait_spin_bounded(bar(BAR_EFFULL), n & 1u, ctl, 6))) break;
          for (int x = 0; x < 3; ++x, ++job) {   // dB^T of chunk 0, of chunk 1, dA
            const uint32_t b = job & 1u;
            if (!(ok = wait_spin_bounded(bar(BAR_JEMPTY + b), ((job >> 1) & 1u) ^ 1u, ctl, 7))) break;
            tc_fence_after();
            const uint32_t d = tmem + COL_JOB + 128u * b;
            if (x < 2) {
#pragma unroll
              for (int ks = 0; ks < 8; ++ks) {
                const uint64_t ad = make_sdesc(smem + OFF_DU + 32768u * x + 2048u * ks, 16384, 1024, SWZ_128B);
                const uint64_t bd = make_sdesc(smem + OFF_AT + abox * (ks >> 2) + 32u * (ks & 3), 16, 1024, SWZ_128B);
                mma_bf16_pair(d, ad, bd, idesc_db, ks > 0 ? 1u : 0u);
              }
            } else {
#pragma unroll
              for (int ks = 0; ks < 16; ++ks) {
                const uint64_t ad = make_sdesc(smem + OFF_DU + 16384u * (ks >> 2) + 32u * (ks & 3), 16, 1024, SWZ_128B);
                const uint64_t bd = make_sdesc(smem + OFF_B + bbox * (ks >> 2) + 32u * (ks & 3), 16, 1024, SWZ_128B);
                mma_bf16_pair(d, ad, bd, idesc_da, ks > 0 ? 1u : 0u);
              }
            }
            mma_commit_pair(bar(BAR_JFULL + b));
          }
          if (!ok) break;
          mma_commit_pair(bar(BAR_EFEMPTY));
        }
        if (!ok) break;
        mma_commit_pair(bar(BAR_DUEMPTY));
        ++it;
      }
      // the peer's reports of the last two jobs land before the CTAs end
      for (uint32_t x = job >= 2 ? job - 2 : 0; ok && x < job; ++x)
        ok = wait_spin_bounded(bar(BAR_JEMPTY + (x & 1u)), (x >> 1) & 1u, ctl, 13);
      mma_commit_pair_self(bar(BAR_DRAIN_J));
      drain_wait(bar(BAR_DRAIN_J), 0, args.timeout_ns);
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int pw = warp - 2;
    const int q = warp & 3;
    const int h = pw >> 2;
    const int row = q * 32 + lane;
    const uint32_t lane_off = static_cast<uint32_t>(q * 32) << 16;
    const int nb = args.k / 128;
    const float gscale = args.s_x != nullptr ? *args.s_x : 1.0f;
    const int hr = R / 2;   // ranks of a job that this warp half writes out
    const bool vec = (args.r & 3) == 0;
    // A warp's event on a leader barrier: the leader's warps arrive (warp 0 also announces
    // the peer's signal bytes), the peer's warps send their signal.
    auto report = [&](int b) {
      if (leader) {
        if (pw == 0) mbar_arrive_expect_tx(bar(b), SIG_TX);
        else mbar_arrive(bar(b));
      } else {
        signal_remote16(sig_dst_leader, sig_src, lbar(b));
      }
    };
    uint32_t it = 0, job = 0;
    bool ok = true;
    WorkIter wi = work_begin(args, pair);
    Unit w;
    while (ok && work_next<WIDE>(wi, args, pair, npairs, w)) {
      const int ib128 = 2 * w.ib + static_cast<int>(rank);
      const int i_g = ib128 * 128 + row;
      // this thread's code bytes (columns 64 h .. 64 h + 63 of both chunks of row i_g) and scales,
      // in flight while the unit's main loop runs
      const uint8_t* cp = static_cast<const uint8_t*>(args.phi) + static_cast<int64_t>(i_g) * args.k + w.jt * BN + 64 * h;
      uint4 raw[8];
      float s_i[2], z_i[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int e = 0; e < 4; ++e) raw[4 * c + e] = reinterpret_cast<const uint4*>(cp + 128 * c)[e];
        const int64_t si = args.s_ld ? static_cast<int64_t>(i_g) * args.s_ld + (w.jt * BN + 128 * c) / args.group_size : i_g;
        s_i[c] = args.s[si];
        z_i[c] = ZP ? args.zero[si] : 0.0f;
      }
      ok = wait_bounded(bar(BAR_DUEMPTY), (it & 1u) ^ 1u, ctl, 3);
      ok = ok && wait_bounded(bar(BAR_ACCFULL), it & 1u, ctl, 9);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const float gs_i = gscale * s_i[c];
        // a 128 x 128 tile that this unit does not write: no mask bits (dU = 0) and no ds
        const bool keep = !WIDE || (w.keep >> (2 * rank + c)) & 1u;
        const uint32_t kept = keep ? 0xffffffffu : 0x7f7f7f7fu;
        float2 ds2 = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          const int jl = 64 * h + 32 * p;   // column within the chunk
          float G[32];
          tmem_ld32(tmem + lane_off + COL_G + 128 * c + jl, G);
          tmem_ld_wait();
          if (c == 1 && p == 1) {
            // the last read of G for this unit: it is free for the next unit's main loop
            tc_fence_before();
            __syncwarp();
            if (lane == 0) report(BAR_ACCEMPTY);
          }
          uint32_t du[16];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const uint4& r4 = raw[4 * c + 2 * p + (e >> 2)];
            const uint32_t wd = ((e & 3) == 0 ? r4.x : (e & 3) == 1 ? r4.y : (e & 3) == 2 ? r4.z : r4.w) & kept;
            float2 cv[2];
            decode_codes4(wd, cv[0], cv[1]);
#pragma unroll
            for (int v = 0; v < 2; ++v) {
              const float2 g2 = make_float2(G[4 * e + 2 * v], G[4 * e + 2 * v + 1]);
              ds2 = __ffma2_rn(g2, ZP ? __fadd2_rn(cv[v], make_float2(-z_i[c], -z_i[c])) : cv[v], ds2);
              const float2 gs = __fmul2_rn(g2, make_float2(gs_i, gs_i));
              du[2 * e + v] = pack_rn_bf16x2(gs.x, gs.y) & (v == 0 ? code_masks2<0>(wd) : code_masks2<1>(wd));
            }
          }
          const uint32_t dub = smem + OFF_DU + 32768u * c + 16384u * h;
#pragma unroll
          for (int wq = 0; wq < 4; ++wq)
            st_shared_v4(dub + swz_offset(row, 4 * p + wq, 128), du[4 * wq], du[4 * wq + 1], du[4 * wq + 2],
                         du[4 * wq + 3]);
        }
        args.ds_part[(static_cast<int64_t>(w.sp * 2 + h) * args.m + i_g) * nb + w.jt * 2 + c] = keep ? (ds2.x + ds2.y) * gscale : 0.0f;
      }
      tc_fence_before();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) report(BAR_DUFULL);
      // the jobs' partials: dB^T (lanes = columns j of the chunk) and dA (lanes = rows i)
      float* dst_b = args.dB_part + static_cast<int64_t>(ib128 * args.nsplit + w.sp) * args.r * args.k + w.jt * BN + row;
      float* dst_a = args.dA_part + (static_cast<int64_t>(w.jt * args.nsplit + w.sp) * args.m + i_g) * args.r;
      for (int rc = 0; rc < rounds && ok; ++rc) {
        for (int x = 0; x < 3; ++x, ++job) {
          const uint32_t b = job & 1u;
          ok = wait_bounded(bar(BAR_JFULL + b), (job >> 1) & 1u, ctl, 12);
          if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
          tc_fence_after();
          const uint32_t col = tmem + lane_off + COL_JOB + 128u * b + (x < 2 ? rank * R : 0u) + h * hr;
          const int t0 = 64 * rc + h * hr;
          for (int c8 = 0; c8 < hr; c8 += 8) {
            float vv[8];
            tmem_ld8(col + c8, vv);
            tmem_ld_wait();
            if (x < 2) {
              float* dst = dst_b + 128 * x;
#pragma unroll
              for (int e = 0; e < 8; ++e)
                if (t0 + c8 + e < args.r) dst[static_cast<int64_t>(t0 + c8 + e) * args.k] = vv[e];
            } else if (vec) {
#pragma unroll
              for (int e = 0; e < 8; e += 4)
                if (t0 + c8 + e < args.r)
                  *reinterpret_cast<float4*>(dst_a + t0 + c8 + e) = make_float4(vv[e], vv[e + 1], vv[e + 2], vv[e + 3]);
            } else {
#pragma unroll
              for (int e = 0; e < 8; ++e)
                if (t0 + c8 + e < args.r) dst_a[t0 + c8 + e] = vv[e];
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) report(BAR_JEMPTY + b);
        }
      }
      if (!ok) break;
      ++it;
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // neither CTA leaves while the other may still read its shared memory
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem, TMEM_COLS);
  }
}

template <bool ZP, bool WIDE>
cudaError_t launch_codes_one(const CUtensorMap& dy, const CUtensorMap& x, const CUtensorMap& at, const CUtensorMap& b,
                             const DwArgs& args, int npairs, cudaStream_t stream) {
  static bool configured[kMaxDevices] = {};
  const void* fn = reinterpret_cast<const void*>(dw_codes_kernel<ZP, WIDE>);
  cudaError_t e = ensure_smem_attr(fn, static_cast<int>(SMEM_BYTES), configured);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(2 * npairs), 1, 1);
  cfg.blockDim = dim3(NUM_THREADS, 1, 1);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[1] = follows_in_call();
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, dw_codes_kernel<ZP, WIDE>, dy, x, at, b, args);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_dw_codes(const CUtensorMap& tm_dy, const CUtensorMap& tm_x, const CUtensorMap& tm_at,
                            const CUtensorMap& tm_b, const DwArgs& args, int npairs, cudaStream_t stream) {
  if (npairs < 1 || args.nchunks != 2 || args.r16 < 16 || args.r16 > 256 || (args.r16 & 15) || args.m % 256 ||
      args.k % 256 || args.ni != args.m / 256 || args.nj != args.k / 256 || args.u_bf16 || args.phi == nullptr ||
      (args.sched.tail && args.r16 > 64 && !args.wide))
    return cudaErrorInvalidValue;
  if (args.wide)
    return args.zero != nullptr ? launch_codes_one<true, true>(tm_dy, tm_x, tm_at, tm_b, args, npairs, stream)
                                : launch_codes_one<false, true>(tm_dy, tm_x, tm_at, tm_b, args, npairs, stream);
  return args.zero != nullptr ? launch_codes_one<true, false>(tm_dy, tm_x, tm_at, tm_b, args, npairs, stream)
                              : launch_codes_one<false, false>(tm_dy, tm_x, tm_at, tm_b, args, npairs, stream);
}

}  // namespace lrqat
