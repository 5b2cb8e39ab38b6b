// Fused LR-QAT GEMM for the forward (Y = X W_hat^T) and the input gradient
// (dX = dY W_hat) on CTA pairs: the same on-chip recompute of W_hat as the one-SM
// kernel (Eq. 8; the recompute replaces the checkpointing of Sec. 3), with the main
// product issued as tcgen05 MMAs of M = 256 rows across the two SMs of a cluster.
//
// Why pairs: the one-SM kernel (128 x 448 tiles) moves its whole 448-token operand through
// each SM's shared memory every stage; in a pair each CTA holds its own 128 weight rows and only
// half of every accumulator's tokens, and the tensor cores of the pair exchange the token halves
// (measured on a 4096 x 4096 layer at T = 8192 on the codes: forward 276 -> 181 us).
//
// A pair processes tiles of 256 weight rows (CTA rank c: rows 128 c .. 128 c + 127; an odd last
// 128-row block leaves CTA 1's half of its tiles empty) x up to 448 tokens (one accumulator of up to 256
// tokens or two of up to 224; CTA c holds half of each one's; the host picks smaller token tiles where
// 448 leave pairs idle, and two or four pairs per tile where those do too: pair_tile in
// lrqat_api.cu), one 64-wide slice of the contraction per stage:
//   * token ring (four to eight slots per CTA; three with the low-rank tile in 448-token tiles): loader
//     warps bring this CTA's token halves (SW128) with TMA whose completion lands on the leader's
//     barrier; each slot also holds this CTA's W_hat tile of the stage;
//   * factor ring (four or eight slots; two for 16-bit bases with the low-rank tile in 448-token tiles):
//     the stored base of this CTA's rows (completion on its own barrier; only its own producers read
//     it), with it the stage's scales (and zero offsets) where the producers apply them (dX, group-wise
//     forward), and with the low-rank tile this CTA's half (32 rows) of the second factor's slice
//     (completion on the leader's barrier: the low-rank MMA reads both halves);
//   * in the leader, one thread per accumulator issues its main product (M = 256, 4 MMAs per stage)
//     and, with the low-rank tile in the stage, another the tile L = RF SF^T (M = 256, N = 64) into one of
//     four TMEM buffers after one accumulator or the one buffer after two (which one thread issues
//     then), so that neither waits behind the other's barriers; every commit is multicast to both CTAs;
//   * sixteen producer warps per CTA, in four groups that take every fourth stage each (one group with
//     the low-rank tile in 448-token tiles), build this CTA's W_hat tile exactly as the one-SM kernel
//     does, and drain this CTA's 128 rows of the accumulators in the epilogue.
// One barrier per slot in the leader counts the stage's token bytes and both CTAs' "W_hat
// written" events, so the MMA thread tests one barrier per stage; the peer's events ("W_hat
// written", "L read", "accumulators drained") travel as 16-byte copies into the leader's shared
// memory whose completion counts on the leader's barrier (a thread-issued remote arrive is
// several times slower under the pair's operand traffic), after fence.proxy.async has ordered
// the peer's writes.
// On the codes (NL: every backward, and the forwards for which prefer_codes_fwd in lrqat_api.cu says
// so, unless set otherwise) the base holds the one-byte codes of the codes pass; no factors, no L.
#include <cuda.h>
#include <cuda_runtime.h>
#include <atomic>
#include <cstdint>

#include "kernels.h"
#include "ptx.cuh"
#include "quant.cuh"

namespace lrqat {
namespace {

constexpr int BM = 128;                          // weight rows per CTA (256 per pair)
constexpr int BK = 64;
constexpr int BNP = 224;                         // most tokens per accumulator of two (N of the pair MMA)
constexpr int NACC = 2;                          // accumulators (one for tiles of up to 256 tokens)
constexpr int NT_MAX = 8;                        // token ring slots
constexpr int NLB_MAX = 4;                       // low-rank TMEM buffers (one per producer group)
constexpr int MAX_TILE_L = 256;                  // most tokens of a tile beside four of them
constexpr int NF_MAX = 8;                        // factor ring slots
constexpr int NUM_PROD_WARPS = 16;
constexpr int FIRST_TMA_WARP = 2 + NUM_PROD_WARPS;
constexpr int NUM_TOK_LOADERS = 4;               // token loaders (every fourth stage each)
constexpr int NUM_TMA_WARPS = NUM_TOK_LOADERS + 1;   // and the factor loader
constexpr int NUM_THREADS = 32 * (FIRST_TMA_WARP + NUM_TMA_WARPS);
// G, the producer groups: 4 = group g takes the stages gg % 4 == g and a warp turns 32 rows x 64 columns
// of each; 1 = all sixteen warps share every stage, 16 columns each.  Four groups need four token slots
// and a low-rank buffer each, so beside the low-rank tile they take tiles of up to 256 tokens; one
// group gets by with three slots (two accumulators of 224 tokens) and one buffer.  Its stage is a
// chain of barriers, longer than four groups' (1455 cycles against 1050), but serves 448 tokens: the
// better one where calls are long (allocation-free 4096 x 4096 forward, T = 8192: 256-token tiles
// 270 us, 448-token tiles 217; FP16 base 395 and 250), the worse one below (T = 1024: 45 and 58 us).

constexpr uint32_t RF_BYTES = 128 * 128;         // 128 rows x 64 rank columns (bf16)
constexpr uint32_t W_BYTES = 128 * 128;          // 128 rows x 64 bf16
constexpr uint32_t SFH_BYTES = 32 * 128;         // 32 slice rows x up to 64 rank columns (bf16)

// Shared-memory rings.  A token slot holds this CTA's half of the stage's tokens (a tile of btp
// tokens: 64 btp bytes) and its W_hat tile, a factor slot the stored base and, with the low-rank tile
// (which also has the row factor resident), this CTA's half of the second factor's slice.  On the codes
// eight factor slots where they leave room for five token slots (tiles up to 256 tokens; dX 224) or, with codes
// that come from HBM (deep), four, then as many token slots as fit (up to eight); else, and with the low-rank
// tile, whose stages are twice as long, four factor slots first.  Four slots of a short stage do not
// cover a fetch from HBM: tiles of 64 to 320 tokens took 1.2 to 1.45 times their stages' cycles (14336 x 4096
// forward at T = 2048: 256-token tiles 183 us with four factor slots, 134 with eight; 288 190, 150).  Where the
// codes stay in L2 eight slots beside five token slots are up to 25% faster and at most 3% slower, beside four up
// to 12% slower (1024 x 14336 at T = 1024, 288 tokens).
// XS: each factor slot also holds the stage's scales (and zero offsets) as bf16, copied by the
// factor loader, so that the producers read them from shared memory with the base instead of
// from global memory: for dX the 64 scales of the stage's contraction indices in the CTA's row
// group, for the group-wise forward the 128 scales of the CTA's rows in the stage's group.
constexpr uint32_t RING_BYTES = 232448 - 1024 - 1024;   // less the static barriers and the alignment
template <int FMT, bool NL, bool XS, int G>
struct PairRing {
  static_assert(G == 4 || (G == 1 && !NL), "producer groups");
  static constexpr uint32_t RF = NL ? 0u : RF_BYTES;
  static constexpr uint32_t PHI_BYTES = fmt_16bit(FMT) ? 128 * 128 : 128 * 64;
  static constexpr uint32_t PHI_TX = FMT == FMT_I4 ? PHI_BYTES / 2 : PHI_BYTES;
  static constexpr uint32_t FS_SF = PHI_BYTES;
  // scales at +0, zero offsets at +512 (dX: 128 bytes each, group-wise forward: 256)
  static constexpr uint32_t FS_X = PHI_BYTES + (NL ? 0u : SFH_BYTES);
  static constexpr uint32_t FSLOT_BYTES = FS_X + (XS ? 1024u : 0u);
  static constexpr uint32_t OFF_RF = 0;
  static constexpr uint32_t OFF_TSLOTS = RF;
  static_assert(FSLOT_BYTES % 1024 == 0 && FS_SF % 1024 == 0, "swizzled tiles must start on 1024-byte boundaries");
  __host__ __device__ static constexpr uint32_t tslot(int btp) { return 64u * btp + W_BYTES; }
  __host__ __device__ static constexpr int nt(int btp, bool deep) {
    if (G == 1) return 3;
    const int n8 = static_cast<int>((RING_BYTES - RF - 8u * FSLOT_BYTES) / tslot(btp));
    const int n = NL && n8 >= (deep ? 4 : 5) ? n8 : static_cast<int>((RING_BYTES - RF - 4u * FSLOT_BYTES) / tslot(btp));
    return n < NT_MAX ? n : NT_MAX;
  }
  // four or eight, multiples of G: a group then knows that the previous use of a slot it waits for has
  // landed (it was its own), so barrier phases cannot alias; one group: four, or two of 16-bit bases
  __host__ __device__ static constexpr int nf(int btp, bool deep) {
    if (G == 1) return fmt_16bit(FMT) ? 2 : 4;
    return (RING_BYTES - RF - nt(btp, deep) * tslot(btp)) / FSLOT_BYTES >= 8 ? 8 : 4;
  }
  // the largest token tile: 448 on the codes and of one group; beside four low-rank buffers 256
  // (16-bit bases: 192)
  static constexpr int MAX_TILE = NL || G == 1 ? 448 : fmt_16bit(FMT) ? 192 : MAX_TILE_L;
  __host__ __device__ static constexpr uint32_t smem(int btp, bool deep) {
    return RF + nt(btp, deep) * tslot(btp) + nf(btp, deep) * FSLOT_BYTES + 1024u;
  }
  static_assert(nt(MAX_TILE, true) >= (G == 4 ? 4 : 1) && smem(MAX_TILE, true) <= RING_BYTES + 1024 &&
                    smem(32, true) <= RING_BYTES + 1024,
                "shared memory budget");
};

constexpr uint32_t TMEM_COLS = 512;
// the 64-column low-rank buffers: four after one accumulator, or one after two
__host__ __device__ constexpr uint32_t col_l(int groups) { return groups == 1 ? NACC * BNP : MAX_TILE_L; }
static_assert(col_l(4) + NLB_MAX * BK <= TMEM_COLS && col_l(1) + BK <= TMEM_COLS, "TMEM budget");

// leader: the stage's operands are in place, i.e. both token halves of the slot landed and both
// CTAs' producers wrote their W_hat tiles (one barrier, so that the MMA thread tests one per stage)
constexpr int BAR_TFULL = 0;
constexpr int BAR_TEMPTY = BAR_TFULL + NT_MAX;   // both: main product of the slot finished
constexpr int BAR_PFULL = BAR_TEMPTY + NT_MAX;   // both: this CTA's base tile landed

constexpr int BAR_FFULL = BAR_PFULL + NF_MAX;    // leader: both factor-slice halves landed
constexpr int BAR_FEMPTY = BAR_FFULL + NF_MAX;   // both: slot read by this CTA's producers (after L)
constexpr int BAR_LFULL = BAR_FEMPTY + NF_MAX;   // both: low-rank tile of the buffer computed
constexpr int BAR_LEMPTY = BAR_LFULL + NLB_MAX;  // leader: both CTAs read the buffer
constexpr int BAR_RFFULL = BAR_LEMPTY + NLB_MAX; // leader: both row-factor halves landed
constexpr int BAR_RFEMPTY = BAR_RFFULL + 1;      // both: last low-rank MMA of the tile finished
constexpr int BAR_ACCFULL = BAR_RFEMPTY + 1;     // both: accumulators of the tile complete
constexpr int BAR_ACCEMPTY = BAR_ACCFULL + 1;    // leader: both CTAs drained them
constexpr int BAR_DRAIN = BAR_ACCEMPTY + 1;
constexpr int BAR_DRAIN_B = BAR_DRAIN + 1;       // the second issuer's
constexpr int NUM_BARS = BAR_DRAIN_B + 1;

__device__ __forceinline__ void drain_wait(uint32_t bar, uint32_t parity, uint64_t timeout_ns) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > timeout_ns) break;
  }
}

// Stages are numbered globally over the pair's tiles (gg), identically in both CTAs: token
// slot gg % NT, factor slot gg % NF, low-rank buffer gg % NLB.  A cursor follows a ring's slot and
// the parity of its use.
struct Cursor {
  uint32_t s = 0, ph = 0;
  __device__ __forceinline__ void next(uint32_t n) {
    if (++s == n) {
      s = 0;
      ph ^= 1u;
    }
  }
  __device__ __forceinline__ void skip(uint32_t k, uint32_t n) {
    for (s += k; s >= n; s -= n) ph ^= 1u;
  }
};
template <int MODE, int FMT, bool ZP, bool UB, bool NL, int G>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    fused_pair_kernel(const __grid_constant__ CUtensorMap tm_tok, const __grid_constant__ CUtensorMap tm_phi,
                      const __grid_constant__ CUtensorMap tm_rf, const __grid_constant__ CUtensorMap tm_sf,
                      const FusedArgs args) {
  using PR = PairRing<FMT, NL, MODE == FUSED_DX || MODE == FUSED_FWD_GROUP, G>;
  constexpr int NLB = G, GROUP_WARPS = NUM_PROD_WARPS / G;
  constexpr uint32_t COL_L = col_l(G);
  constexpr uint32_t OFF_RF = PR::OFF_RF, OFF_TSLOTS = PR::OFF_TSLOTS;
  constexpr bool PACKED = FMT == FMT_I4;
  constexpr uint32_t FSLOT_BYTES = PR::FSLOT_BYTES;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[NUM_BARS];
  __shared__ __align__(16) uint32_t sig_buf[8];   // [0, 4): source of the peer's signals, [4, 8): their target
  __shared__ uint32_t tmem_base_s;
  __shared__ volatile int abort_s;

  const uint32_t smem = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  // A cluster holds `ksplit` pairs that share a tile: pair `slice` takes that part of the contraction
  // (1: one pair per cluster, persistent over its tiles).  rank: this CTA's place in its pair.
  const int ksplit = G == 1 ? 1 : args.ksplit;
  const uint32_t crank = cluster_cta_rank(), rank = crank & 1u, lead = G == 1 ? 0u : crank & ~1u;
  const int slice = static_cast<int>(crank >> 1);
  const bool leader = rank == 0;
  const uint32_t pair_mask = 3u << lead;   // the pair's CTAs, for multicast commits
  const int pair = blockIdx.x / (2 * ksplit), npairs = gridDim.x / (2 * ksplit);
  auto bar = [&](int i) { return smem_u32(&bars[i]); };
  auto lbar = [&](int i) { return map_shared_rank(smem_u32(&bars[i]), lead); };   // the leader's copy

  // the token tile: one accumulator of bnp <= 256 tokens or two of bnp <= 224, half of each per CTA
  const int bnp = G == 1 ? BNP : args.bnp, bnh = bnp / 2, nacc = G == 1 ? NACC : args.nacc, btp = bnp * nacc;
  const int NT = PR::nt(btp, args.deep), NF = PR::nf(btp, args.deep);
  const uint32_t TSLOT_BYTES = PR::tslot(btp), TOK_BOX = 128u * bnh, TS_W = 64u * btp;
  const uint32_t OFF_FSLOTS = OFF_TSLOTS + NT * TSLOT_BYTES;
  // one thread issues both accumulators where the other issuer's warp has the low-rank tiles
  constexpr bool BOTH = !NL && G == 1;
  const uint32_t issuers = BOTH ? 1 : nacc;   // threads that issue (and commit) the main product
  if (threadIdx.x == 0) {
    abort_s = 0;
    for (int s = 0; s < NT; ++s) {
      mbar_init(bar(BAR_TFULL + s), 1 + GROUP_WARPS);   // the leader's token loader and producer warps
      mbar_init(bar(BAR_TEMPTY + s), issuers);
    }
    for (int s = 0; s < NF; ++s) {
      mbar_init(bar(BAR_PFULL + s), 1);
      mbar_init(bar(BAR_FFULL + s), 1);
      // freed by this CTA's producers after they built W_hat: by then they have waited for the
      // low-rank tile, so the low-rank MMA that read the slot's factor half has completed
      mbar_init(bar(BAR_FEMPTY + s), GROUP_WARPS);
    }
    for (int b = 0; b < NLB; ++b) {
      mbar_init(bar(BAR_LFULL + b), 1);
      mbar_init(bar(BAR_LEMPTY + b), GROUP_WARPS);
    }
    mbar_init(bar(BAR_RFFULL), 1);
    mbar_init(bar(BAR_RFEMPTY), 1);
    mbar_init(bar(BAR_ACCFULL), issuers);
    mbar_init(bar(BAR_ACCEMPTY), NUM_PROD_WARPS);
    mbar_init(bar(BAR_DRAIN), 1);
    mbar_init(bar(BAR_DRAIN_B), 1);
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
  // this pair's stages k0 .. k0 + nk - 1 (kdim is a multiple of 128, ksplit at most kdim / 64)
  const int nk_all = args.kdim / BK, k0 = nk_all * slice / ksplit, nk = nk_all * (slice + 1) / ksplit - k0;
  const int num_rb2 = (args.num_rb + 1) / 2;   // 256-row blocks
  // This CTA's first row in row block rb2.  With an odd number of 128-row blocks the last pair's
  // CTA 1 has none: it takes part with zero-filled loads (and the last block's scales) and stores
  // nothing.
  auto row_block = [&](int rb2) {
    const int r0 = rb2 * 2 * BM + static_cast<int>(rank) * BM;
    return r0 < args.rows ? r0 : args.rows - BM;
  };
  const int num_tiles = num_rb2 * ((args.T + btp - 1) / btp);
  const uint32_t sig_src = smem_u32(&sig_buf[0]);
  const uint32_t sig_dst_leader = map_shared_rank(smem_u32(&sig_buf[4]), lead);
  // A producer warp's event on a leader barrier: the leader's warps arrive (warp 0 also
  // announces the peer's 16 signal bytes of each of the n warps), the peer's warps send their signal.
  auto report = [&](int b, int pw, int n) {
    if (leader) {
      if (pw == 0) mbar_arrive_expect_tx(bar(b), 16u * n);
      else mbar_arrive(bar(b));
    } else {
      signal_remote16(sig_dst_leader, sig_src, lbar(b));
    }
  };

  // The main product of the pair's tiles into accumulator a (BOTH: into both), by one thread of the leader.  Two
  // accumulators have a thread each: a thread's barrier test and commit (~110
  // and ~70 cycles a stage, with the tensor pipe queueing about one MMA ahead) then run beside the
  // other's MMAs (4096 x 4096, 288-token tiles 906 -> 739 cycles a stage, 320 925 -> 801; at 448 the
  // operands' shared-memory traffic sets the pace either way, 1101 -> 1106).
  auto issue_main = [&](int a, int drain) {
    const uint32_t idesc_main = make_idesc_bf16(256, bnp, 0, 0);
    const uint32_t TSLOT_D = TSLOT_BYTES >> 4, d = tmem + a * BNP;
    const uint64_t d_w0 = make_sdesc(smem + OFF_TSLOTS + TS_W, 16, 1024, SWZ_128B);
    const uint64_t d_tok = make_sdesc(smem + OFF_TSLOTS + a * TOK_BOX, 16, 1024, SWZ_128B);
    uint32_t it = 0;
    Cursor cur;
    bool ok = true;
    for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
      if (!(ok = wait_spin_bounded(bar(BAR_ACCEMPTY), (it & 1u) ^ 1u, ctl, 7))) break;
      tc_fence_after();
      // unrolled: the loop's own overhead between two stages' MMAs was ~120 cycles of idle tensor pipe
#pragma unroll 4
      for (int kk = 0; kk < nk; ++kk) {
        const uint32_t s = cur.s;
        if (!(ok = wait_spin_bounded(bar(BAR_TFULL + s), cur.ph, ctl, 9))) break;
        cur.next(NT);
        tc_fence_after();
        const uint64_t w = d_w0 + s * TSLOT_D, t = d_tok + s * TSLOT_D;
        const uint32_t acc = kk > 0 ? 1u : 0u;
        static_assert(BK == 64, "four K steps below");
        mma_bf16_pair(d, w, t, idesc_main, acc);
        mma_bf16_pair(d, w + 2, t + 2, idesc_main, 1u);
        mma_bf16_pair(d, w + 4, t + 4, idesc_main, 1u);
        mma_bf16_pair(d, w + 6, t + 6, idesc_main, 1u);
        if (BOTH) {
          const uint64_t t2 = t + (TOK_BOX >> 4);
          mma_bf16_pair(d + BNP, w, t2, idesc_main, acc);
          mma_bf16_pair(d + BNP, w + 2, t2 + 2, idesc_main, 1u);
          mma_bf16_pair(d + BNP, w + 4, t2 + 4, idesc_main, 1u);
          mma_bf16_pair(d + BNP, w + 6, t2 + 6, idesc_main, 1u);
        }
        mma_commit_pair(bar(BAR_TEMPTY + s), pair_mask);
      }
      if (!ok) break;
      mma_commit_pair(bar(BAR_ACCFULL), pair_mask);
      ++it;
    }
    // the peer's last drain report lands before the CTAs end
    if (ok) ok = wait_spin_bounded(bar(BAR_ACCEMPTY), (it & 1u) ^ 1u, ctl, 10);
    mma_commit_pair_self(bar(drain));
    drain_wait(bar(drain), 0, args.timeout_ns);
  };

  // Epilogue: the factor of an output row, and 16 tokens of it scaled, masked and stored.
  auto out_scale = [&](int row_g) {
    float scale = 1.0f;
    if (MODE == FUSED_FWD_PC) scale = args.s[row_g];
    if (MODE != FUSED_DX && args.s_x != nullptr) scale *= *args.s_x;
    return scale;
  };
  auto store_tokens = [&](float (&acc)[16], float scale, int row_g, int tok0) {
    uint32_t mword = 0xffffffffu;
    if (MODE == FUSED_DX && args.xmask != nullptr && tok0 < args.T)
      mword = args.xmask[static_cast<int64_t>(row_g) * args.xmask_ld + tok0 / 32] >> (tok0 & 31);
#pragma unroll
    for (int e = 0; e < 16; ++e) acc[e] = ((mword >> e) & 1u) ? acc[e] * scale : 0.0f;
    store_row_pairs_bf16(acc, lane & 1, args.out, args.out_ld, row_g, tok0, args.T);
  };

  if (warp == 0) {
    // ------------------- row factor (per tile) and, in the leader, the low-rank MMAs
    // A thread of its own issues the low-rank tiles, so that the main product never waits
    // behind their barriers; each thread's commits track only its own MMAs.  On the codes it is the
    // second accumulator's issuer.
    if (NL) {
      if (leader && lane == 0 && nacc == 2) issue_main(1, BAR_DRAIN_B);
    } else if (lane == 0) {
      prefetch_tensormap(&tm_rf);
      const uint32_t idesc_l = make_idesc_bf16(256, BK, 0, 0);
      const int lsteps = args.r16 / 16;
      const uint64_t d_rf = make_sdesc(smem + OFF_RF, 16, 1024, SWZ_128B);
      // the K-major half slice: 32 rows of sf_cols bf16 (32, 64 or 128 bytes, swizzled to match)
      const uint32_t sf_swz = args.sf_cols == 64 ? SWZ_128B : args.sf_cols == 32 ? SWZ_64B : SWZ_32B;
      const uint64_t d_sf0 = make_sdesc(smem + OFF_FSLOTS + PR::FS_SF, 16, 16u * args.sf_cols, sf_swz);
      constexpr uint32_t FSLOT_D = FSLOT_BYTES >> 4;
      uint32_t it = 0, g = 0;
      Cursor f;
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
        const int rb2 = tile % num_rb2;
        if (!(ok = wait_spin_bounded(bar(BAR_RFEMPTY), (it & 1u) ^ 1u, ctl, 1))) break;
        if (leader) mbar_arrive_expect_tx(bar(BAR_RFFULL), 2u * RF_BYTES);
        tma_load_2d_pair(smem + OFF_RF, &tm_rf, 0, rb2 * 2 * BM + static_cast<int>(rank) * BM, lbar(BAR_RFFULL));
        if (leader) {
          if (!(ok = wait_spin_bounded(bar(BAR_RFFULL), it & 1u, ctl, 6))) break;
          for (int kk = 0; kk < nk && ok; ++kk) {
            // L(gg) into buffer gg % NLB once both factor halves landed and both CTAs read L(gg - NLB)
            const uint32_t gg = g + kk, s = f.s, b = gg % NLB;
            if (!(ok = wait_spin_bounded(bar(BAR_FFULL + s), f.ph, ctl, 4))) break;
            f.next(NF);
            if (!(ok = wait_spin_bounded(bar(BAR_LEMPTY + b), ((gg / NLB) & 1u) ^ 1u, ctl, 5))) break;
            tc_fence_after();
            const uint64_t sf = d_sf0 + s * FSLOT_D;
            const uint32_t dl = tmem + COL_L + BK * b;
            for (int ks = 0; ks < lsteps; ++ks) mma_bf16_pair(dl, d_rf + 2 * ks, sf + 2 * ks, idesc_l, ks > 0 ? 1u : 0u);
            mma_commit_pair(bar(BAR_LFULL + b), pair_mask);
          }
          if (!ok) break;
          mma_commit_pair(bar(BAR_RFEMPTY), pair_mask);   // last read of the row factor issued
        }
        g += nk;
        ++it;
      }
      if (leader && ok) {
        // the peer's reports of the last low-rank tiles land before the CTAs end
        for (uint32_t gg = g >= NLB ? g - NLB : 0; ok && gg < g; ++gg)
          ok = wait_spin_bounded(bar(BAR_LEMPTY + gg % NLB), (gg / NLB) & 1u, ctl, 11);
      }
    }
  } else if (warp >= FIRST_TMA_WARP && warp < FIRST_TMA_WARP + NUM_TOK_LOADERS) {
    // ------------------------------------ token loaders (one warp's copies come one after another)
    // Loader t takes the stages t, t + NL4, ...  A loader waits for the product of stage gg - NT in
    // a barrier phase that the next but one use of the slot would alias: it must know that stage
    // gg - 2 NT has finished, which its previous wait (stage gg - NL4 - NT) tells it for NL4 <= NT.
    const int NL4 = NT < NUM_TOK_LOADERS ? NT : NUM_TOK_LOADERS;
    if (lane == 0 && warp - FIRST_TMA_WARP < NL4) {
      prefetch_tensormap(&tm_tok);
      int kk = warp - FIRST_TMA_WARP;   // this loader's next stage of the tile
      Cursor c;
      c.skip(kk, NT);
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
        const int tok = tile / num_rb2 * btp + static_cast<int>(rank) * bnh;
        for (; kk < nk; kk += NL4) {
          if (!(ok = wait_spin_bounded(bar(BAR_TEMPTY + c.s), c.ph ^ 1u, ctl, 2))) break;
          if (leader) mbar_arrive_expect_tx(bar(BAR_TFULL + c.s), 128u * btp);
          const uint32_t st = smem + OFF_TSLOTS + c.s * TSLOT_BYTES, fb = lbar(BAR_TFULL + c.s);
          tma_load_2d_pair(st, &tm_tok, (k0 + kk) * BK, tok, fb);
          if (nacc == 2) tma_load_2d_pair(st + TOK_BOX, &tm_tok, (k0 + kk) * BK, tok + bnp, fb);
          c.skip(NL4, NT);
        }
        kk -= nk;
      }
    }
  } else if (warp == FIRST_TMA_WARP + NUM_TOK_LOADERS) {
    // ------------------------------------------------- factor-ring loader
    if (lane == 0) {
      prefetch_tensormap(&tm_phi);
      if (!NL) prefetch_tensormap(&tm_sf);
      const uint32_t sf_tx = static_cast<uint32_t>(32 * 2 * args.sf_cols);   // one CTA's half slice
      Cursor f;
      uint32_t last = 0, last_ph = 0;   // the last copy's slot and parity
      bool any = false, ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
        const int rb2 = tile % num_rb2;
        for (int kk = k0; kk < k0 + nk; ++kk) {
          const uint32_t s = f.s;
          if (!(ok = wait_spin_bounded(bar(BAR_FEMPTY + s), f.ph ^ 1u, ctl, 3))) break;
          any = true;
          last = s;
          last_ph = f.ph;
          f.next(NF);
          const uint32_t fs = smem + OFF_FSLOTS + s * FSLOT_BYTES;
          constexpr uint32_t XTX = MODE == FUSED_DX        ? (ZP ? 256u : 128u)
                                   : MODE == FUSED_FWD_GROUP ? (ZP ? 512u : 256u)
                                                             : 0u;
          mbar_arrive_expect_tx(bar(BAR_PFULL + s), PR::PHI_TX + XTX);
          tma_load_2d(fs, &tm_phi, PACKED ? kk * (BK / 2) : kk * BK, rb2 * 2 * BM + static_cast<int>(rank) * BM,
                      bar(BAR_PFULL + s));
          if (MODE == FUSED_DX) {
            // the stage's 64 scales (and zero offsets) of this CTA's row group (group sizes are
            // multiples of 128, so a CTA's 128 rows lie in one group)
            const int64_t xoff = (args.s_ld ? static_cast<int64_t>(row_block(rb2) / args.group_size) * args.kdim : 0) +
                                 kk * BK;
            bulk_load(fs + PR::FS_X, args.s_bf16 + xoff, 128u, bar(BAR_PFULL + s));
            if (ZP) bulk_load(fs + PR::FS_X + 512u, args.z_bf16 + xoff, 128u, bar(BAR_PFULL + s));
          } else if (MODE == FUSED_FWD_GROUP) {
            // the 128 scales (and zero offsets) of this CTA's rows in the stage's group, from the
            // bf16 rows [groups][m] (a group holds a multiple of 128 contraction indices, so two
            // stages never straddle it)
            const int64_t xoff = static_cast<int64_t>((kk * BK) / args.group_size) * args.rows + row_block(rb2);
            bulk_load(fs + PR::FS_X, args.s_bf16 + xoff, 256u, bar(BAR_PFULL + s));
            if (ZP) bulk_load(fs + PR::FS_X + 512u, args.z_bf16 + xoff, 256u, bar(BAR_PFULL + s));
          }
          if (!NL) {
            if (leader) mbar_arrive_expect_tx(bar(BAR_FFULL + s), 2u * sf_tx);
            tma_load_2d_pair(fs + PR::FS_SF, &tm_sf, 0, kk * BK + static_cast<int>(rank) * 32, lbar(BAR_FFULL + s));
          }
        }
      }
      if (any) drain_wait(bar(BAR_PFULL + last), last_ph, args.timeout_ns);
    }
  } else if (warp == 1) {
    // ------------------------------------ main-product MMA issuer (the leader's)
    if (leader && lane == 0) issue_main(0, BAR_DRAIN);
  } else {
    // ------------------------------------------- W_hat producers + epilogue
    const int pw = warp - 2;              // 0..15
    const int q = warp & 3;               // TMEM lane quarter this warp may access
    const int c = pw >> 2;                // group (one group: 16-column chunk of the slice); epilogue block
    const int gw = G == 4 ? q : pw;       // this warp in its group
    const int lb = G == 4 ? c : 0;        // the group's low-rank buffer
    const int y0 = G == 4 ? 0 : 2 * c;    // the first eight of the slice's columns that this warp turns
    const int row = q * 32 + lane;        // row of this CTA's tile handled by this thread
    const uint32_t lane_off = static_cast<uint32_t>(q * 32) << 16;
    const QuantParams qp = args.q;
    const uint32_t lr2 = pack_rn_bf16x2(qp.lr_scale, qp.lr_scale);
    uint32_t g = 0;
    uint32_t it = 0;
    Cursor fc, tc;   // factor and token slots
    if (G == 4) {
      fc.skip(c, NF);
      tc.skip(c, NT);
    }
    bool ok = true;
    for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
      const int rb2 = tile % num_rb2;
      const int tb = tile / num_rb2;
      const int row_g = row_block(rb2) + row;
      const bool has_rows = rb2 * 2 * BM + static_cast<int>(rank) * BM < args.rows;
      const uint32_t z_row = MODE == FUSED_FWD_PC && ZP ? pack_rn_bf16x2(args.zero[row_g], args.zero[row_g]) : 0u;
      // Group c's stages of the tile (gg % 4 == c; one group: every stage).  A ready barrier costs a test of
      // ~110 cycles and the proxy fence and reports ~100 more, whatever the warp does between them: with all sixteen warps in
      // every stage these made a stage on the codes 770 cycles (4096 x 4096, 32-token tiles), four groups
      // in flight pay them side by side (596 cycles; 256-token tiles 863 -> 700).  With the low-rank tile
      // a group has a TMEM buffer of its own, so four low-rank tiles are in flight instead of one
      // (1700 -> 1030 cycles a stage; T = 1024 forward 58 -> 45 us).
      for (int kk = G == 4 ? static_cast<int>((static_cast<uint32_t>(c) - g) & 3u) : 0; kk < nk; kk += G) {
        ok = wait_bounded(bar(BAR_PFULL + fc.s), fc.ph, ctl, 12);
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        const uint32_t fs = smem + OFF_FSLOTS + fc.s * FSLOT_BYTES;
        constexpr int RAW = PACKED ? 2 : fmt_16bit(FMT) ? 8 : 4;   // words of 16 stored values
        constexpr int ROW_BYTES = 16 * RAW;
        uint32_t raw[RAW * G];                                     // this warp's 16 G columns of the row
        if (PACKED && G == 1) {
          const uint2 r = ld_shared_v2(fs + swz_offset(row, c >> 1, ROW_BYTES) + 8 * (c & 1));
          raw[0] = r.x, raw[1] = r.y;
        } else {
#pragma unroll
          for (int x = 0; x < RAW * G / 4; ++x) {
            const uint4 r = ld_shared_v4(fs + swz_offset(row, y0 * RAW / 8 + x, ROW_BYTES));
            raw[4 * x] = r.x, raw[4 * x + 1] = r.y, raw[4 * x + 2] = r.z, raw[4 * x + 3] = r.w;
          }
        }
        uint32_t sg = 0, zg = z_row;   // forward: the row's scale and zero offset in the stage, as bf16x2
        if (MODE == FUSED_FWD_GROUP) {
          sg = ld_shared_u16(fs + PR::FS_X + 2u * row);
          sg |= sg << 16;
          if (ZP) {
            zg = ld_shared_u16(fs + PR::FS_X + 512u + 2u * row);
            zg |= zg << 16;
          }
        }
        uint32_t w[8 * G];
        if constexpr (NL) {
#pragma unroll
          for (int x = 0; x < G; ++x) {
            const uint32_t in[4] = {raw[4 * x], raw[4 * x + 1], raw[4 * x + 2], raw[4 * x + 3]};
            if (args.codes_bias == 64) {
#pragma unroll
              for (int i = 0; i < 4; ++i) decode_b64_bf16x4(in[i], w[8 * x + 2 * i], w[8 * x + 2 * i + 1]);
            } else {
              float v[16];
              decode_ob16(in, v);
#pragma unroll
              for (int e = 0; e < 8; ++e) w[8 * x + e] = pack_int_bf16x2(v[2 * e], v[2 * e + 1]);
            }
          }
        } else {
          float v[16];
          if (G == 1) decode16<FMT>(raw, v);   // before the wait: the one buffer is to be read and reported at once
          // the group's low-rank buffer (gg % NLB)
          ok = wait_bounded(bar(BAR_LFULL + lb), ((g + kk) / NLB) & 1u, ctl, 13);
          if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int x = 0; x < G; ++x) {
            float Lv[16];
            tmem_ld16(tmem + lane_off + COL_L + BK * lb + 8 * y0 + 16 * x, Lv);
            if (G == 4) {
              uint32_t in[RAW];
#pragma unroll
              for (int e = 0; e < RAW; ++e) in[e] = raw[RAW * x + e];
              decode16<FMT>(in, v);
            }
            tmem_ld_wait();
            if (x == G - 1) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) report(BAR_LEMPTY + lb, gw, GROUP_WARPS);
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const float2 u = UB ? u_bf16x2(Lv[2 * e], Lv[2 * e + 1], v[2 * e], v[2 * e + 1], lr2)
                                  : __ffma2_rn(make_float2(Lv[2 * e], Lv[2 * e + 1]),
                                               make_float2(qp.lr_scale, qp.lr_scale),
                                               make_float2(v[2 * e], v[2 * e + 1]));
              w[8 * x + e] = codes_bf16x2(__fadd2_rn(u, make_float2(qp.magic, qp.magic)), qp);
            }
          }
        }
#pragma unroll
        for (int x = 0; x < 2 * G; ++x) {
          if (MODE == FUSED_DX) {
            // the bf16 scales (zero offsets) of eight contraction indices, as bf16x2 words
            const uint4 s4 = ld_shared_v4(fs + PR::FS_X + 16u * (y0 + x));
            if (ZP) {
              const uint4 z4 = ld_shared_v4(fs + PR::FS_X + 512u + 16u * (y0 + x));
              w[4 * x] = sub_bf16x2(w[4 * x], z4.x), w[4 * x + 1] = sub_bf16x2(w[4 * x + 1], z4.y);
              w[4 * x + 2] = sub_bf16x2(w[4 * x + 2], z4.z), w[4 * x + 3] = sub_bf16x2(w[4 * x + 3], z4.w);
            }
            w[4 * x] = mul_bf16x2(w[4 * x], s4.x), w[4 * x + 1] = mul_bf16x2(w[4 * x + 1], s4.y);
            w[4 * x + 2] = mul_bf16x2(w[4 * x + 2], s4.z), w[4 * x + 3] = mul_bf16x2(w[4 * x + 3], s4.w);
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              if (ZP) w[4 * x + e] = sub_bf16x2(w[4 * x + e], zg);
              if (MODE == FUSED_FWD_GROUP) w[4 * x + e] = mul_bf16x2(w[4 * x + e], sg);
            }
          }
        }
        // the slot's W_hat buffer was last read by the product of the stage NT before
        ok = wait_bounded(bar(BAR_TEMPTY + tc.s), tc.ph ^ 1u, ctl, 14);
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        const uint32_t wt = smem + OFF_TSLOTS + tc.s * TSLOT_BYTES + TS_W;
#pragma unroll
        for (int x = 0; x < 2 * G; ++x)
          st_shared_v4(wt + swz_offset(row, y0 + x, 128), w[4 * x], w[4 * x + 1], w[4 * x + 2], w[4 * x + 3]);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          report(BAR_TFULL + tc.s, gw, GROUP_WARPS);
          mbar_arrive(bar(BAR_FEMPTY + fc.s));
        }
        if (G == 1) {   // (skip's loop made a stage of the one group 7% longer)
          fc.next(NF);
          tc.next(NT);
        } else {
          fc.skip(G, NF);
          tc.skip(G, NT);
        }
      }
      if (!ok) break;
      // ------------------------------------------------------------ epilogue
      ok = wait_spin_bounded(bar(BAR_ACCFULL), it & 1u, ctl, 15);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      tc_fence_after();
      if (G == 1 || ksplit == 1) {
        const float scale = out_scale(row_g);
#pragma unroll 1
        for (int col = has_rows ? 16 * c : btp; col < btp; col += 64) {   // token offset in the tile
          float acc[16];
          tmem_ld16(tmem + lane_off + (col < bnp ? col : BNP + col - bnp), acc);
          tmem_ld_wait();
          store_tokens(acc, scale, row_g, tb * btp + col);
        }
      } else {
        // the other slices' token columns of this CTA's partial sums go to its ring (idle: the tile's
        // copies, W_hat tiles and products are all done), [token][row]
#pragma unroll 1
        for (int col = 16 * c; col < btp; col += 64) {
          if (col / (btp / ksplit) == slice) continue;
          float acc[16];
          tmem_ld16(tmem + lane_off + col, acc);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 16; ++e) st_shared_f32(smem + ((col + e) * BM + row) * 4u, acc[e]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) report(BAR_ACCEMPTY, pw, NUM_PROD_WARPS);
      g += nk;
      ++it;
    }
  }

  if (G == 4 && ksplit > 1) {
    // One tile per cluster: its pairs' partial sums meet.  Pair p owns the p-th part of the tile's
    // tokens and adds the slices' sums in order through distributed shared memory.
    __syncwarp();
    cluster_sync_all();
    if (warp >= 2 && warp < FIRST_TMA_WARP && pair < num_tiles && !abort_s) {
      tc_fence_after();
      const int q = warp & 3, c = (warp - 2) >> 2, row = q * 32 + lane;
      const int rb2 = pair % num_rb2, tb = pair / num_rb2, own = btp / ksplit;
      const int row_g = row_block(rb2) + row;
      const bool has_rows = rb2 * 2 * BM + static_cast<int>(rank) * BM < args.rows;
      const float scale = out_scale(row_g);
#pragma unroll 1
      for (int col = slice * own + 16 * c; col < (slice + 1) * own; col += 64) {
        float mine[16], acc[16];
        tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) + col, mine);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = 0.0f;
        for (int p = 0; p < ksplit; ++p) {
          const uint32_t src = map_shared_rank(smem + (col * BM + row) * 4u, 2u * p + rank);
#pragma unroll
          for (int e = 0; e < 16; ++e) acc[e] += p == slice ? mine[e] : ld_cluster_f32(src + e * BM * 4u);
        }
        if (has_rows) store_tokens(acc, scale, row_g, tb * btp + col);
      }
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

template <int MODE, int FMT, bool ZP, bool UB, bool NL, int G = 4>
cudaError_t launch_pair_one(const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& c, const CUtensorMap& d,
                            const FusedArgs& args, int npairs, cudaStream_t stream) {
  if constexpr (!NL && G == 4)   // beside the low-rank tile, two accumulators take one producer group
    if (args.nacc == 2) return launch_pair_one<MODE, FMT, ZP, UB, NL, 1>(a, b, c, d, args, npairs, stream);
  using PR = PairRing<FMT, NL, MODE == FUSED_DX || MODE == FUSED_FWD_GROUP, G>;
  if (args.bnp * args.nacc > PR::MAX_TILE) return cudaErrorInvalidValue;
  if (G == 1 && (args.bnp != BNP || args.ksplit != 1)) return cudaErrorInvalidValue;
  if (args.ksplit > 1 && (args.nacc != 1 || args.bnp % (16 * args.ksplit))) return cudaErrorInvalidValue;
  const uint32_t smem = PR::smem(args.bnp * args.nacc, args.deep);
  static bool configured[kMaxDevices] = {};
  const void* fn = reinterpret_cast<const void*>(fused_pair_kernel<MODE, FMT, ZP, UB, NL, G>);
  cudaError_t e = ensure_smem_attr(fn, 232448 - 1024, configured);   // the most any tile asks for
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(2 * args.ksplit * npairs), 1, 1);
  cfg.blockDim = dim3(NUM_THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[1] = follows_in_call();
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(2 * args.ksplit);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (args.ksplit > 1) {   // one tile per cluster, however many are resident at once
    cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, fused_pair_kernel<MODE, FMT, ZP, UB, NL, G>, a, b, c, d, args);
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  // The persistent grid holds no more pairs than can be resident at once (an SM that has no
  // partner in its GPC cannot host half of a pair), looked up once per device.
  static int max_pairs[kMaxDevices] = {};
  int dev = 0;
  e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (max_pairs[dev] == 0) {
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, fused_pair_kernel<MODE, FMT, ZP, UB, NL, G>, &cfg);
    if (e != cudaSuccess) return e;
    if (n < 1) return cudaErrorInvalidConfiguration;
    max_pairs[dev] = n;
  }
  if (npairs > max_pairs[dev]) {
    npairs = max_pairs[dev];
    cfg.gridDim = dim3(static_cast<unsigned>(2 * npairs), 1, 1);
  }
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, fused_pair_kernel<MODE, FMT, ZP, UB, NL, G>, a, b, c, d, args);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <int MODE, int FMT>
cudaError_t launch_pair_fmt(const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& c, const CUtensorMap& d,
                            const FusedArgs& args, int npairs, cudaStream_t stream) {
  if (args.r16 == 0) {
    if (FMT != FMT_Q8 || args.u_bf16) return cudaErrorInvalidValue;
    return args.zero != nullptr ? launch_pair_one<MODE, FMT_Q8, true, false, true>(a, b, c, d, args, npairs, stream)
                                : launch_pair_one<MODE, FMT_Q8, false, false, true>(a, b, c, d, args, npairs, stream);
  }
  if (args.u_bf16) {
    if (FMT == FMT_F16 || args.zero != nullptr) return cudaErrorInvalidValue;
    return launch_pair_one<MODE, FMT == FMT_F16 ? FMT_Q8 : FMT, false, true, false>(a, b, c, d, args, npairs, stream);
  }
  if (fmt_float(FMT)) {
    if (args.zero != nullptr) return cudaErrorInvalidValue;
    return launch_pair_one<MODE, FMT, false, false, false>(a, b, c, d, args, npairs, stream);
  }
  return args.zero != nullptr ? launch_pair_one<MODE, FMT, true, false, false>(a, b, c, d, args, npairs, stream)
                              : launch_pair_one<MODE, FMT, false, false, false>(a, b, c, d, args, npairs, stream);
}

template <int MODE>
cudaError_t launch_pair_mode(int fmt, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& c,
                             const CUtensorMap& d, const FusedArgs& args, int npairs, cudaStream_t stream) {
  switch (fmt) {
    case FMT_Q8: return launch_pair_fmt<MODE, FMT_Q8>(a, b, c, d, args, npairs, stream);
    case FMT_I4:
      if (MODE == FUSED_DX) return cudaErrorInvalidValue;
      return launch_pair_fmt<MODE, MODE == FUSED_DX ? FMT_Q8 : FMT_I4>(a, b, c, d, args, npairs, stream);
    case FMT_BF16: return launch_pair_fmt<MODE, FMT_BF16>(a, b, c, d, args, npairs, stream);
    case FMT_F16: return launch_pair_fmt<MODE, FMT_F16>(a, b, c, d, args, npairs, stream);
    case FMT_E4M3: return launch_pair_fmt<MODE, FMT_E4M3>(a, b, c, d, args, npairs, stream);
    case FMT_E5M2: return launch_pair_fmt<MODE, FMT_E5M2>(a, b, c, d, args, npairs, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

int fused_pair_max_clusters(int ksplit) {
  static std::atomic<int> cache[kMaxDevices][5];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices || ksplit < 1 || ksplit > 4) return 0;
  int n = cache[dev][ksplit].load(std::memory_order_acquire);
  if (n > 0) return n;
  using PR = PairRing<FMT_Q8, true, false, 4>;
  static bool configured[kMaxDevices] = {};
  const void* fn = reinterpret_cast<const void*>(fused_pair_kernel<FUSED_FWD_PC, FMT_Q8, false, false, true, 4>);
  if (ensure_smem_attr(fn, 232448 - 1024, configured) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(2 * ksplit), 1, 1);
  cfg.blockDim = dim3(NUM_THREADS, 1, 1);
  cfg.dynamicSmemBytes = PR::smem(256, true);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(2 * ksplit);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&n, fused_pair_kernel<FUSED_FWD_PC, FMT_Q8, false, false, true, 4>, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  cache[dev][ksplit].store(n, std::memory_order_release);
  return n;
}

cudaError_t launch_fused_pair(int mode, int fmt, const CUtensorMap& tm_tok, const CUtensorMap& tm_phi,
                              const CUtensorMap& tm_rf, const CUtensorMap& tm_sf, const FusedArgs& args, int npairs,
                              cudaStream_t stream) {
  if (npairs < 1 || (args.kdim % 128) != 0 || args.kdim < 128 || (args.rows % BM) != 0 || args.sf_mn ||
      args.num_rb != args.rows / 128 || args.bnp < 16 || (args.bnp & 15) ||
      !(args.nacc == 1 ? args.bnp <= 256 : args.nacc == 2 && args.bnp <= BNP) || args.ksplit < 1 || args.ksplit > 4 ||
      args.ksplit > args.kdim / BK)
    return cudaErrorInvalidValue;
  switch (mode) {
    case FUSED_FWD_PC: return launch_pair_mode<FUSED_FWD_PC>(fmt, tm_tok, tm_phi, tm_rf, tm_sf, args, npairs, stream);
    case FUSED_FWD_GROUP:
      return launch_pair_mode<FUSED_FWD_GROUP>(fmt, tm_tok, tm_phi, tm_rf, tm_sf, args, npairs, stream);
    case FUSED_DX: return launch_pair_mode<FUSED_DX>(fmt, tm_tok, tm_phi, tm_rf, tm_sf, args, npairs, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lrqat
