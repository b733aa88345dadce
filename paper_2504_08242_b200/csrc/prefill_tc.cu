// Chunked-prefill attention on the 5th-generation tensor cores (paper Sec. IV-A, Fig. 5(b)):
// chunk rows at positions pos..pos+n-1 attend causally to cache rows 0..pos+i.
//
// Two kernels (see choose_form).  A query tile is 128 rows: tokens of the chunk x heads that share a kv head.
//  - prefill_tc_kernel (this file): one CTA owns TWO query tiles of the same kv head and walks the KV cache in tiles of
//    128 keys, every K/V tile serving both query tiles:
//      loader warp : TMA (tiled, 128-byte swizzle) Q once, then K/V tiles into 2-stage rings
//      MMA warps   : one thread issues the tcgen05.mma of S = Q K^T, another those of O += P V, accumulators in TMEM
//      softmax WGs : one warpgroup per query tile, one thread per row holding the row's 128 scores in registers:
//                    row maximum, P = exp2(...) with fp32-pair arithmetic written to TMEM as bf16 and released to the
//                    MMA issuer in two parts; lazy rescale of O only when the maximum grew by > 2^8
//    TMEM (512 columns): O_A | O_B (128 each) | S (128) | P_A | P_B (64 each).  The one S buffer goes back and forth
//    between the query tiles: a softmax holds it only while it reads its scores into registers, so the next tile's
//    scores are computed during the softmax and not after O += P V has read P.  What bounds it: the softmax warps (two
//    per scheduler, 2720 cycles per pair of tiles for 2048 of the special-function unit and as many of the tensor pipe), and the
//    clock, which falls with the tensor pipe's use (about 1.5 GHz here).  Measured on four 8192-token prompts with 32 / 8
//    heads in chunks of 512 (us a prompt set, in a burst / back to back), from P written over S and one issuing thread:
//    2188 / 2390; P in its own columns and S shared, one issuer 2460 / 2613; two issuers 2024 / 2277; the PV
//    issuer standing back for the scores 1963 / 2225; named barriers 1986 / 2223 (2720 against 3140 cycles per pair of
//    tiles).
//  - prefill_frag_kernel (prefill_tc_frag.cuh): one query tile per CTA, both warpgroups on it; on small grids a cluster of
//    2, 4 or 8 CTAs shares a query tile and splits its KV walk.
// head_dim 64 runs the same kernels with half as many operand slices and accumulator columns.  Measured against the
// mma.sync kernel that took it before (us a call, append included, 32 / 8 heads): 16 rows at position 0 4.9 : 6.6, 448
// rows at position 0 8.1 : 14.8, at position 2048 23 : 60, four prompts at once 65 : 171 -- never slower, so that kernel
// is left with the non-positive scales.
// All mbarrier waits are bounded; on expiry the CTA sets the status word, drains its own copies and MMAs, frees
// TMEM and returns.
#include "host_checks.h"
#include <algorithm>

#include "kernels.h"
#include "tc_common.cuh"
#include "tc_softmax.cuh"
#include "tmap.h"

namespace jup {

constexpr int TC_BM = 128;              // query rows per tile
constexpr int TC_BN = 128;              // keys per KV tile
constexpr int TC_PANEL_BYTES = 16384;   // 128 rows x 64 elements of bf16: a Q, K or V tile is D / 64 of them

struct TcParams {
  int q_heads, q_len, pos;
  int prefix_len;  // rows of a shared prefix cache attended before the sequence's own cache (0: none)
  // A query tile is `tokens` tokens x `pack` heads that share a kv head, tokens * pack <= 128 rows, the heads running
  // fastest.
  int tokens;
  FastDiv pack, head_blocks, blocks_per_kv, batch_blocks;  // head_blocks = q_heads / pack, batch_blocks = batch x head_blocks
  int q_blocks;  // query tiles (fragment form) or pairs of query tiles per (sequence, block of heads)
  float scale_log2;
  float* out;
  float* lse;
  int* status;
  float* scratch;  // fragment form with several CTAs per query tile: their partial results
  int prefix_batched;  // 1: the front segment has one cache per sequence (fused form), 0: one cache shared by all
  // Fused KVCache write (fused_write != 0).  The chunk's K/V rows, token-major [batch][q_len][kv_heads][D], are
  // the attention's own segment; the CTAs of each group's first query head also write them, bit-exactly, into rows
  // copy_pos + r of the cache, with tiled stores straight from the K/V slots the tiles were loaded into (tensor
  // maps tm_ck / tm_cv over the destination cache).
  int fused_write;
  int copy_pos;
};

// One past the last of the chunk's K/V tiles that the query tile(s) of tokens [t0, t1) write to the cache: the tiles whose
// last token they hold.  (The first is t0 / TC_BN.)
__device__ __forceinline__ int own_tiles_end(int t1, int q_len) { return t1 == q_len ? (q_len + TC_BN - 1) / TC_BN : t1 / TC_BN; }

constexpr int TC_NQ = 2;  // query tiles per CTA
template <int D>
struct TcCfg {
  static constexpr int TILE_BYTES = TC_BM * D * 2;
  static constexpr int PANELS = D / 64;
  static constexpr int KV_STAGES = 2;
  static constexpr int SOFTMAX_WARPS = 4 * TC_NQ;
  static constexpr int LOADER_WARP = SOFTMAX_WARPS;
  static constexpr int QK_WARP = SOFTMAX_WARPS + 1, PV_WARP = SOFTMAX_WARPS + 2;
  // Three full warpgroups (the third: loader, two MMA issuers, an idle warp) so that the register file can be
  // re-divided: a softmax thread holds a whole score row (REGS_SOFTMAX), the third warpgroup gives its share back
  // (REGS_OTHER); 2 x 128 x 208 + 128 x 88 = 384 x 168, the registers the CTA starts with.
  static constexpr int THREADS = 384;
  static constexpr int REGS_SOFTMAX = 208, REGS_OTHER = 88;
  // TMEM columns: O_0 | O_1 | S | P_0 | P_1
  static constexpr int O_COL0 = 0, S_COL = 256, P_COL0 = 384;
  // shared memory: [Q tiles][K ring][V ring][barriers]
  static constexpr int SMEM_Q = 0;
  static constexpr int SMEM_K = TC_NQ * TILE_BYTES;
  static constexpr int SMEM_V = SMEM_K + KV_STAGES * TILE_BYTES;
  static constexpr int SMEM_BAR = SMEM_V + KV_STAGES * TILE_BYTES;
  static constexpr int SMEM_BYTES = SMEM_BAR + 256 + 1024;  // + slack for 1024-byte alignment
  static_assert(SMEM_BYTES <= 227 * 1024, "shared memory per CTA");
};

// barrier indices (8 bytes each) inside the barrier block
enum {
  BAR_Q_FULL = 0,    // [2]
  BAR_K_FULL = 2,    // [2]
  BAR_K_EMPTY = 4,   // [2]
  BAR_V_FULL = 6,    // [2]
  BAR_V_EMPTY = 8,   // [2]
  BAR_S_FULL = 10,   // [2] one per query tile
  BAR_O_READY = 12,  // [2]
  BAR_DRAIN = 14,    // [2] one per issuing thread
  BAR_COUNT = 16
};
constexpr int TC_BOX_FLOATS = TC_BM * 32;  // 16 KB
constexpr int NQ = TC_NQ;

template <int D>
__global__ void __launch_bounds__(TcCfg<D>::THREADS, 1)
prefill_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                  const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_pk,
                  const __grid_constant__ CUtensorMap tm_pv, const __grid_constant__ CUtensorMap tm_o,
                  const __grid_constant__ CUtensorMap tm_ck, const __grid_constant__ CUtensorMap tm_cv, TcParams p) {
  using Cfg = TcCfg<D>;
  constexpr int TILE_BYTES = Cfg::TILE_BYTES;
  constexpr int KV_STAGES = Cfg::KV_STAGES;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t sQ = smem_base + Cfg::SMEM_Q, sK = smem_base + Cfg::SMEM_K, sV = smem_base + Cfg::SMEM_V;
  const uint32_t sBar = smem_base + Cfg::SMEM_BAR;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_gen + Cfg::SMEM_BAR + 8 * BAR_COUNT);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + Cfg::SMEM_BAR + 8 * BAR_COUNT + 8);
  const uint32_t qk_turn = sBar + 8u * BAR_COUNT + 16u;  // odd while a batch of scores is being issued
  static_assert(8 * BAR_COUNT + 20 <= 256, "barrier block");
  auto bar = [&](int i) { return sBar + 8u * i; };

  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;

  // ---- work assignment: heaviest query blocks first
  int bh, hb, hr;
  const int qblk = p.q_blocks - 1 - p.batch_blocks.divmod(blockIdx.x, bh);
  const int b = p.head_blocks.divmod(bh, hb), hk = p.blocks_per_kv.divmod(hb, hr);  // hr: 0 for a group's first heads
  const int pack = p.pack.d, h0 = hb * pack;
  // KV tiles 0..Tp-1 come from the shared prefix (every row sees them, no causal limit), the rest from
  // the sequence's own cache
  const int Tp = (p.prefix_len + TC_BN - 1) / TC_BN;
  // T[x]: KV tiles of query tile x; Tall: KV tiles the CTA loads
  int T[2] = {0, 0};
#pragma unroll
  for (int x = 0; x < NQ; ++x) {
    const int t0 = (qblk * NQ + x) * p.tokens;
    if (t0 < p.q_len) T[x] = Tp + (p.pos + min(p.q_len, t0 + p.tokens) + TC_BN - 1) / TC_BN;
  }
  const int Tall = max(T[0], T[1]);

  // ---- set-up
  if (threadIdx.x == 0) {
    for (int i = 0; i < BAR_COUNT; ++i) mbar_init(bar(i), 1u);
    *abort_flag = 0;
    count_publish(qk_turn, 0);
    mbar_fence_init();
  }
  if (warp == Cfg::QK_WARP) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
    tmem_relinquish();
  } else if (warp == Cfg::LOADER_WARP && lane == 0) {
    // the tensor maps are kernel parameters: fetching them does not depend on the previous kernel
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_k);
    tma_prefetch_desc(&tm_v);
    tma_prefetch_desc(&tm_o);
    if (Tp > 0) {
      tma_prefetch_desc(&tm_pk);
      tma_prefetch_desc(&tm_pv);
    }
    if (p.fused_write != 0) {
      tma_prefetch_desc(&tm_ck);
      tma_prefetch_desc(&tm_cv);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = warp_uniform(*tmem_slot);
  pdl_wait();  // everything above overlapped the previous kernel's tail; global memory is touched from here on

  if (warp == Cfg::LOADER_WARP) {
    // =============================================================== loader
    reg_dec<Cfg::REGS_OTHER>();
    if (lane == 0) {
#pragma unroll
      for (int x = 0; x < NQ; ++x) {
        if (T[x] == 0) continue;
        // (rows of a Q tile beyond its pack x tokens are never written: they belong to no query, and whatever the
        // tensor cores make of them is never used)
        mbar_expect_tx(bar(BAR_Q_FULL + x), static_cast<uint32_t>(pack * p.tokens) * (D * 2u));
#pragma unroll
        for (int c = 0; c < Cfg::PANELS; ++c)
          tma_load_4d(sQ + x * TILE_BYTES + c * TC_PANEL_BYTES, &tm_q, bar(BAR_Q_FULL + x), c * 64, h0, (qblk * NQ + x) * p.tokens, b);
      }
      int issued = 0;
      bool ok = true;
      // Fused KVCache write: the chunk's own K/V tiles are loaded for the attention anyway; the tiles whose last token
      // is in this CTA's query tiles (of each group's first heads) go from their slots to the cache with tiled stores,
      // as soon as they have landed.  A slot is refilled only after its store has read it.
      const bool writer = p.fused_write != 0 && hr == 0;
      const int own0 = qblk * NQ * p.tokens / TC_BN;
      const int own1 = own_tiles_end(min((qblk + 1) * NQ * p.tokens, p.q_len), p.q_len);
      auto store_own_tile = [&](int j) {
        const int t = j - Tp;  // tile of the chunk
        if (!writer || t < own0 || t >= own1) return;
        const int s = j % KV_STAGES, u = j / KV_STAGES;
        ok = ok && mbar_wait(bar(BAR_K_FULL + s), u & 1, abort_flag, p.status);
        ok = ok && mbar_wait(bar(BAR_V_FULL + s), u & 1, abort_flag, p.status);
        if (!ok) return;
        const int row = p.copy_pos + t * TC_BN;  // rows beyond copy_pos + q_len are clipped by the tensor maps
#pragma unroll
        for (int c = 0; c < Cfg::PANELS; ++c) {
          tma_store_4d(&tm_ck, sK + s * TILE_BYTES + c * TC_PANEL_BYTES, c * 64, row, hk, b);
          tma_store_4d(&tm_cv, sV + s * TILE_BYTES + c * TC_PANEL_BYTES, c * 64, row, hk, b);
        }
        tma_store_commit();
        tma_store_wait_read();
      };
      for (int j = 0; j < Tall && ok; ++j) {
        const int s = j % KV_STAGES, u = j / KV_STAGES;
        if (u > 0) store_own_tile(j - KV_STAGES);
        if (!ok) break;
        if (u > 0) ok = mbar_wait(bar(BAR_K_EMPTY + s), (u - 1) & 1, abort_flag, p.status);
        if (!ok) break;
        mbar_expect_tx(bar(BAR_K_FULL + s), TILE_BYTES);
        const CUtensorMap* mk = j < Tp ? &tm_pk : &tm_k;
        const int krow = (j < Tp ? j : j - Tp) * TC_BN, kb = (j < Tp && !p.prefix_batched) ? 0 : b;
#pragma unroll
        for (int c = 0; c < Cfg::PANELS; ++c)
          tma_load_4d(sK + s * TILE_BYTES + c * TC_PANEL_BYTES, mk, bar(BAR_K_FULL + s), c * 64, krow, hk, kb);
        if (u > 0) ok = mbar_wait(bar(BAR_V_EMPTY + s), (u - 1) & 1, abort_flag, p.status);
        if (!ok) {
          issued = 2 * j + 1;
          break;
        }
        mbar_expect_tx(bar(BAR_V_FULL + s), TILE_BYTES);
        const CUtensorMap* mv = j < Tp ? &tm_pv : &tm_v;
#pragma unroll
        for (int c = 0; c < Cfg::PANELS; ++c)
          tma_load_4d(sV + s * TILE_BYTES + c * TC_PANEL_BYTES, mv, bar(BAR_V_FULL + s), c * 64, krow, hk, kb);
        issued = 2 * j + 2;
      }
      for (int j = max(0, Tall - KV_STAGES); j < Tall && ok; ++j) store_own_tile(j);
      if (*abort_flag) {
        // wait (bounded) until every copy this thread started has landed before shared memory is released
        int dummy = 0;
        volatile int* none = &dummy;
        const int nk = (issued + 1) / 2, nv = issued / 2;
        for (int j = max(0, nk - KV_STAGES); j < nk; ++j)
          mbar_wait(bar(BAR_K_FULL + j % KV_STAGES), (j / KV_STAGES) & 1, none, nullptr);
        for (int j = max(0, nv - KV_STAGES); j < nv; ++j)
          mbar_wait(bar(BAR_V_FULL + j % KV_STAGES), (j / KV_STAGES) & 1, none, nullptr);
        for (int x = 0; x < NQ; ++x)
          if (T[x] > 0) mbar_wait(bar(BAR_Q_FULL + x), 0, none, nullptr);
      }
    }
    __syncwarp();
  } else if (warp == Cfg::QK_WARP) {
    // =============================================================== issuer of S = Q K^T
    // Two threads issue the MMAs, one the scores and one the products with V: an issuing thread is held up while the
    // tensor pipe works through what it has queued, so the barrier tests and commits between two batches of a single
    // thread leave the pipe idle; with two threads the pipe works on one batch while the other thread prepares its
    // next.  The issue loops are kept to an integer addition or two per MMA (descriptor halves, see tc_desc_lo).
    reg_dec<Cfg::REGS_OTHER>();
    constexpr uint32_t idesc_qk = tc_idesc_bf16(TC_BM, TC_BN, false, false);
    const uint32_t s_col = tmem + Cfg::S_COL;
    const bool leader = elect_one();
    bool ok = true;
    // One S buffer serves both query tiles: it may be written once the softmax that got the previous scores has
    // read them (a fraction of a tile's time), long before that tile's P V is due, so the scores are complete when
    // the softmax comes for them and only its own work is on a tile's critical path.
    int prev_x = -1;  // owner of the scores written last
    int turn = 0;
    for (int j = 0; j < Tall; ++j) {
      const uint32_t k_lo = tc_desc_lo(sK + (j % KV_STAGES) * TILE_BYTES, 16);
      ok = ok && mbar_wait(bar(BAR_K_FULL + j % KV_STAGES), (j / KV_STAGES) & 1, abort_flag, p.status);
#pragma unroll
      for (int x = 0; x < NQ; ++x) {
        if (j >= T[x]) continue;
        if (j == 0) ok = ok && mbar_wait(bar(BAR_Q_FULL + x), 0, abort_flag, p.status);
        if (prev_x >= 0) named_sync(NB_S_FREE + prev_x, 160);
        prev_x = x;
        ok = __all_sync(0xffffffffu, ok);
        if (leader && ok) {
          flag_write(qk_turn, ++turn);  // odd: a batch of scores is being issued
          tc_fence_after();
          const uint32_t q_lo = tc_desc_lo(sQ + x * TILE_BYTES, 16);
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const uint32_t off = ((ks >> 2) * TC_PANEL_BYTES + (ks & 3) * 32) >> 4;
            tc_mma_ss_lo(s_col, q_lo + off, k_lo + off, idesc_qk, ks > 0);
          }
          tc_commit(bar(BAR_S_FULL + x));
          flag_write(qk_turn, ++turn);
        }
        __syncwarp();
      }
      if (leader && ok) tc_commit(bar(BAR_K_EMPTY + j % KV_STAGES));
    }
    if (prev_x >= 0) named_sync(NB_S_FREE + prev_x, 160);
    if (leader && !ok) {  // make sure no MMA of this thread is still running before TMEM and smem go away
      int dummy = 0;
      tc_commit(bar(BAR_DRAIN));
      mbar_wait(bar(BAR_DRAIN), 0, &dummy, nullptr);
    }
    __syncwarp();
  } else if (warp == Cfg::PV_WARP) {
    // =============================================================== issuer of O += P V
    // The pipe serves the two threads' MMAs in turn, which would double the time to the next scores, and those are
    // what everybody waits for: this thread stands back while a batch of scores is being issued.  (Looked at once per
    // batch: the shared-memory read takes longer than an MMA.)
    reg_dec<Cfg::REGS_OTHER>();
    constexpr uint32_t idesc_pv = tc_idesc_bf16(TC_BM, D, false, true);
    const bool leader = elect_one();
    bool ok = true;
    for (int j = 0; j < Tall; ++j) {
      const uint32_t v_lo = tc_desc_lo(sV + (j % KV_STAGES) * TILE_BYTES, TC_PANEL_BYTES);
      ok = ok && mbar_wait(bar(BAR_V_FULL + j % KV_STAGES), (j / KV_STAGES) & 1, abort_flag, p.status);
#pragma unroll
      for (int x = 0; x < NQ; ++x) {
        if (j >= T[x]) continue;
        const uint32_t o_col = tmem + Cfg::O_COL0 + x * 128, p_col = tmem + Cfg::P_COL0 + x * 64;
        named_sync(NB_P_EARLY + x, 160);  // the first 96 keys while the softmax finishes the last 32
        ok = __all_sync(0xffffffffu, ok);
        if (leader && ok) {
          for (int it = 0; it < 4096 && (flag_read(qk_turn) & 1); ++it) {}
          tc_fence_after();
#pragma unroll
          for (int ks = 0; ks < 6; ++ks)
            tc_mma_ts_lo(o_col, p_col + ks * 8, v_lo + ks * (2048 >> 4), idesc_pv, (j > 0 || ks > 0));
        }
        __syncwarp();
        named_sync(NB_P_FULL + x, 160);
        if (leader && ok) {
          tc_fence_after();
#pragma unroll
          for (int ks = 6; ks < 8; ++ks) tc_mma_ts_lo(o_col, p_col + ks * 8, v_lo + ks * (2048 >> 4), idesc_pv, 1);
          tc_commit(bar(BAR_O_READY + x));
        }
        __syncwarp();
      }
      if (leader && ok) tc_commit(bar(BAR_V_EMPTY + j % KV_STAGES));
    }
    if (leader && !ok) {
      int dummy = 0;
      tc_commit(bar(BAR_DRAIN + 1));
      mbar_wait(bar(BAR_DRAIN + 1), 0, &dummy, nullptr);
    }
    __syncwarp();
  } else if (warp < Cfg::SOFTMAX_WARPS) {
    // =============================================================== softmax warpgroups
    reg_inc<Cfg::REGS_SOFTMAX>();
    const int x = warp >> 2;                      // query tile of this warpgroup
    const int row_in_tile = (warp & 3) * 32 + lane;
    const int t0 = (qblk * NQ + x) * p.tokens;
    const int lim = p.pos + min(t0 + p.pack.div(row_in_tile), p.q_len - 1) + 1;  // keys j < lim are visible
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t tO = tmem + lane_base + Cfg::O_COL0 + x * 128;
    const float c = p.scale_log2;
    float m_ref = -INFINITY, l = 0.f;
    bool ok = true;
    const int Tx = T[x];
    auto signal = [&](int id) {
      tc_fence_before();
      if (ok) named_arrive(id + x, 160);
      else named_sync(id + x, 160);
    };
    for (int j = 0; j < Tx; ++j) {
      const uint32_t tS = tmem + lane_base + Cfg::S_COL, tP = tmem + lane_base + Cfg::P_COL0 + x * 64;
      // (ok is the same in all lanes of a warp: the barriers and the tcgen05 operations are warp-collective)
      ok = __all_sync(0xffffffffu, ok && mbar_spin_wait(bar(BAR_S_FULL + x), j & 1, abort_flag, p.status));
      tc_fence_after();
      // columns >= nvalid are masked: the end of the prefix in its last tile, the causal limit afterwards
      const int nvalid = j < Tp ? p.prefix_len - j * TC_BN : lim - (j - Tp) * TC_BN;
      const bool masked = __any_sync(0xffffffffu, nvalid < TC_BN);
      softmax_tile_row<false, D>(
          tS, tP, tO, j, 4, masked, ColumnLimit{nvalid}, true, c, m_ref, l,
          [&] { return mbar_test_wait(bar(BAR_O_READY + x), (j - 1) & 1); },
          [&] { ok = ok && mbar_wait(bar(BAR_O_READY + x), (j - 1) & 1, abort_flag, p.status); },
          [&] { signal(NB_S_FREE); },
          [&] {
            ok = __all_sync(0xffffffffu, ok);
            signal(NB_P_EARLY);
          });
      signal(NB_P_FULL);
    }
    pdl_launch_dependents();  // the next kernel of the stream may start its own set-up now
    if (Tx > 0) {  // warpgroup-uniform: every thread of the tile reaches the named barriers below, even one that gave
                   // up on a wait (it only skips its global stores)
      ok = ok && mbar_wait(bar(BAR_O_READY + x), (Tx - 1) & 1, abort_flag, p.status);
      tc_fence_after();
      // O / l goes out through shared memory (this tile's Q buffer, free now) and tiled stores: two rounds of
      // D / 64 boxes of 128 rows x 32 columns; rows at or beyond q_len are clipped by the tensor map.
      const float inv = 1.f / l;
      float* stage = reinterpret_cast<float*>(smem_gen + Cfg::SMEM_Q + x * TILE_BYTES);
      const uint32_t stage_addr = sQ + x * TILE_BYTES;
      const int tid_t = threadIdx.x & 127;
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
#pragma unroll
        for (int q2 = 0; q2 < Cfg::PANELS; ++q2) {
          uint32_t o[32];
          tmem_ld32(tO + hh * (D / 2) + q2 * 32, o);
          tc_wait_ld();
          float v[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(o[i]) * inv;
          stage_box_row(stage + q2 * TC_BOX_FLOATS, row_in_tile, v);
        }
        fence_proxy_async();
        named_sync(NB_STORE + x, 128);
        if (tid_t == 0) {
          if (ok) {
#pragma unroll
            for (int c = 0; c < Cfg::PANELS; ++c)
              tma_store_4d(&tm_o, stage_addr + c * TC_BOX_FLOATS * 4, hh * (D / 2) + c * 32, h0, t0, b);
            tma_store_commit();
          }
          tma_store_wait_read();  // the boxes are rewritten next / shared memory is released at the end of the kernel
        }
        if (hh == 0) named_sync(NB_STORE + x, 128);
      }
      int hd;
      const int tok = t0 + p.pack.divmod(known_here(row_in_tile), hd);
      if (ok && p.lse && tok < min(p.q_len, t0 + p.tokens))
        p.lse[(static_cast<int64_t>(b) * p.q_heads + h0 + hd) * p.q_len + tok] =
            (m_ref + log2f(l)) * 0.69314718055994530942f;
    }
  }

  else {
    reg_dec<Cfg::REGS_OTHER>();  // the idle warp of the third warpgroup: the re-division is a warpgroup's decision
  }

  // ---- tear-down
  tc_fence_before();
  __syncthreads();
  if (warp == Cfg::QK_WARP) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace jup

#include "prefill_tc_frag.cuh"

namespace jup {

// ---------------------------------------------------------------- host side

// Log-sum-exps are results of 32 bits and want exact exponentials; without them only bf16 weights come of an exponential, and the
// form with a quarter of them on the FMA pipe is taken: four prompts of 8192 tokens in chunks of 128 2417 us against 2448, 2048
// tokens in chunks of 256 105.9 against 107.  With head_dim 64 it gains nothing (3000 tokens in chunks of 448 124 against 123).
template <int D>
static bool frag_exact(const float* lse) {
  return D == 64 || lse != nullptr;
}
template <int D, int C, bool EXACT>
static cudaError_t frag_set_attributes() {
  static PerDeviceOnce done;
  if (done.done()) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(prefill_frag_kernel<D, C, EXACT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       FragCfg<D>::SMEM_BYTES);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(prefill_frag_kernel<D, C, EXACT>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess) done.set();
  return e;
}
template <int D, int C, bool EXACT>
static cudaError_t launch_frag_as(int64_t units, cudaStream_t st, const CUtensorMap& tq, const CUtensorMap& tk,
                                  const CUtensorMap& tv, const CUtensorMap& tpk, const CUtensorMap& tpv,
                                  const CUtensorMap& tck, const CUtensorMap& tcv, const TcParams& p) {
  cudaError_t e = frag_set_attributes<D, C, EXACT>();
  if (e != cudaSuccess) return e;
  return launch_pdl_cluster(prefill_frag_kernel<D, C, EXACT>, dim3(static_cast<unsigned>(units * C)),
                            dim3(FragCfg<D>::THREADS), FragCfg<D>::SMEM_BYTES, st, static_cast<unsigned>(C), tq, tk, tv, tpk,
                            tpv, tck, tcv, p);
}
template <int D, int C, class... Args>
static cudaError_t launch_frag(const float* lse, Args&&... args) {
  if constexpr (D != 64)
    if (!frag_exact<D>(lse)) return launch_frag_as<D, C, false>(args...);
  return launch_frag_as<D, C, true>(args...);
}

// How many clusters of C CTAs of the fragment form can be resident at once on the current device (0 if the query fails; both
// forms take the same registers and shared memory).
template <int D, int C>
static int frag_resident_clusters() {
  static ResidentClusters clusters;
  if (frag_set_attributes<D, C, true>() != cudaSuccess) return 0;
  return clusters.get(reinterpret_cast<const void*>(prefill_frag_kernel<D, C, true>), C, FragCfg<D>::THREADS,
                      FragCfg<D>::SMEM_BYTES);
}

template <int D>
static cudaError_t launch_pairs(int64_t ctas, cudaStream_t st, const CUtensorMap& tq, const CUtensorMap& tk,
                                  const CUtensorMap& tv, const CUtensorMap& tpk, const CUtensorMap& tpv,
                                  const CUtensorMap& to, const CUtensorMap& tck, const CUtensorMap& tcv,
                                  const TcParams& p) {
  using Cfg = TcCfg<D>;
  static PerDeviceOnce done;
  if (!done.done()) {
    cudaError_t e =
        cudaFuncSetAttribute(prefill_tc_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM_BYTES);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(prefill_tc_kernel<D>, cudaFuncAttributePreferredSharedMemoryCarveout,
                               cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    done.set();
  }
  return launch_pdl_cluster(prefill_tc_kernel<D>, dim3(static_cast<unsigned>(ctas)),
                            dim3(Cfg::THREADS), Cfg::SMEM_BYTES, st, 1u, tq, tk, tv, tpk, tpv, to, tck,
                            tcv, p);
}

bool prefill_tc_supported(const CacheView& c, float scale) {
  // a positive finite scale, and strides a tensor map can carry (multiples of 16 bytes below 2^40;
  // the 16-byte rule is part of every cache descriptor already)
  return scale > 0.f && scale < INFINITY && encode_fn() != nullptr && stride_encodable(c.sr) &&
         stride_encodable(c.sh) && stride_encodable(c.sb);
}

// How a call is laid out: which kernel, how many of a kv head's query heads share a query tile, how many CTAs share its
// KV walk.
struct TcForm {
  bool pairs;  // two query tiles per CTA (prefill_tc_kernel), else one (prefill_frag_kernel)
  int pack, tokens, split;
};

// The layout with the shortest estimated time, in cycles of a CTA.
//  - A KV tile takes a CTA 2720 cycles with a pair of query tiles and 1700 with one (head_dim 128 and 64 alike); a CTA's
//    fixed time is about 6000.
//  - Heads of a group in one query tile: as many as make the fewest CTAs.  A chunk of 150 tokens with 4 heads per kv head
//    is 5 tiles of 32 tokens x 4 heads instead of 8 of 128 tokens x 1 head.
//  - Several CTAs per query tile (a cluster) when all of them run at once: the walk shrinks by the split, the exchange of the
//    partial results costs about 2.5 us and more with every CTA that takes part.  Measured (us a call, 1 CTA per query tile :
//    the chosen split, head_dim 128): 8 heads x 100 rows at position 192 8.1 : 8.1 (1), at 960 13.5 : 9.6 (8), at 3968
//    33.6 : 11.7 (8); 32 heads x 256 rows at 960 15.4 : 13.9 (2), at 3968 38.5 : 27.1 (2).  (A cluster of four CTAs sharing
//    a PAIR of query tiles, which this replaced, took 29.6 us for the last.)
template <int D>
static TcForm choose_form(int batch, int q_heads, int group, int q_len, int kv_tiles, size_t workspace_bytes, int sm_count) {
  constexpr int64_t PAIR = 2720, ONE = 1700, FIXED = 6000;
  TcForm best = {false, 1, TC_BM, 1};
  int64_t best_est = -1;
  for (int pairs = 0; pairs < 2; ++pairs) {
    int pack = 1;
    int64_t units = -1;
    for (int g = 1; g <= std::min(group, TC_BM); ++g) {
      if (group % g != 0) continue;
      const int tokens = TC_BM / g, tiles = (q_len + tokens - 1) / tokens;
      const int64_t u = static_cast<int64_t>(batch) * (q_heads / g) * (pairs ? (tiles + 1) / 2 : tiles);
      if (units < 0 || u < units) {
        units = u;
        pack = g;
      }
    }
    auto consider = [&](int split, int64_t at_once) {
      if (split > 1 && (at_once < units || kv_tiles < split ||
                        SCRATCH_COUNTER_BYTES + static_cast<size_t>(units) * split * FRAG_PART_F4<D> * 16 > workspace_bytes))
        return;
      const int64_t waves = (units + at_once - 1) / at_once, exchange = split > 1 ? 4500 + D / 6 * units * split : 0;
      const int64_t est = waves * ((kv_tiles + split - 1) / split * (pairs ? PAIR : ONE) + FIXED + exchange);
      if (best_est < 0 || est < best_est) {
        best_est = est;
        best = TcForm{pairs != 0, pack, TC_BM / pack, split};
      }
    };
    consider(1, sm_count);
    if (!pairs && 2 * units <= sm_count) {
      consider(2, frag_resident_clusters<D, 2>());
      consider(4, frag_resident_clusters<D, 4>());
      consider(8, frag_resident_clusters<D, 8>());
    }
  }
  return best;
}

// c: the attention's own segment (rows [0, pos + q_len) of every sequence); prefix (nullable): the segment in front
// of it, shared by all sequences or one per sequence (prefix_batched); copy_dst (nullable): cache that receives the
// own segment's rows at copy_pos (the own segment is then the chunk's token-major K/V).
template <int D>
static cudaError_t launch_tc(const bf16* q, const CacheView& c, const CacheView* prefix, int prefix_len,
                             bool prefix_batched, const CacheView* copy_dst, int copy_pos, int q_heads, int q_len,
                             int pos, float scale, float* out, float* lse, int* status, void* workspace,
                             size_t workspace_bytes, cudaStream_t st, LaunchInfo& li) {
  CUtensorMap tq, tk, tv, tpk, tpv, to, tck, tcv;
  if (!encode_fn()) return cudaErrorInvalidValue;
  if (!prefix) prefix_len = 0;
  const int kv_tiles = (prefix_len + TC_BN - 1) / TC_BN + (pos + q_len + TC_BN - 1) / TC_BN;
  const TcForm f = choose_form<D>(c.batch, q_heads, q_heads / c.kv_heads, q_len, kv_tiles, workspace ? workspace_bytes : 0,
                                  li.sm_count);
  {  // out: [batch][q_len][q_heads][D] fp32, boxes of a query tile's rows x 32 columns
    const uint64_t d[4] = {D, static_cast<uint64_t>(q_heads), static_cast<uint64_t>(q_len),
                           static_cast<uint64_t>(c.batch)};
    const uint64_t s[3] = {D * 4ull, static_cast<uint64_t>(q_heads) * D * 4ull,
                           static_cast<uint64_t>(q_len) * q_heads * D * 4ull};
    const uint32_t bx[4] = {32, static_cast<uint32_t>(f.pack), static_cast<uint32_t>(f.tokens), 1};
    if (!make_map_f32(&to, out, d, s, bx)) return cudaErrorInvalidValue;
  }
  const uint64_t rows_valid = static_cast<uint64_t>(pos) + q_len;  // rows above are dead: TMA zero-fills them
  {
    const uint64_t d[4] = {D, static_cast<uint64_t>(q_heads), static_cast<uint64_t>(q_len),
                           static_cast<uint64_t>(c.batch)};
    const uint64_t s[3] = {D * 2ull, static_cast<uint64_t>(q_heads) * D * 2ull,
                           static_cast<uint64_t>(q_len) * q_heads * D * 2ull};
    const uint32_t bx[4] = {64, static_cast<uint32_t>(f.pack), static_cast<uint32_t>(f.tokens), 1};
    if (!make_map_bf16(&tq, q, d, s, bx)) return cudaErrorInvalidValue;
  }
  {
    const uint64_t d[4] = {D, rows_valid, static_cast<uint64_t>(c.kv_heads), static_cast<uint64_t>(c.batch)};
    const uint64_t s[3] = {static_cast<uint64_t>(c.sr) * 2, static_cast<uint64_t>(c.sh) * 2,
                           static_cast<uint64_t>(c.sb) * 2};
    const uint32_t bx[4] = {64, TC_BN, 1, 1};
    if (!make_map_bf16(&tk, c.k, d, s, bx) || !make_map_bf16(&tv, c.v, d, s, bx)) return cudaErrorInvalidValue;
  }
  if (prefix && prefix_len > 0) {  // rows at or beyond prefix_len are zero-filled by TMA
    const uint64_t d[4] = {D, static_cast<uint64_t>(prefix_len), static_cast<uint64_t>(prefix->kv_heads),
                           static_cast<uint64_t>(prefix_batched ? prefix->batch : 1)};
    const uint64_t s[3] = {static_cast<uint64_t>(prefix->sr) * 2, static_cast<uint64_t>(prefix->sh) * 2,
                           static_cast<uint64_t>(prefix->sb) * 2};
    const uint32_t bx[4] = {64, TC_BN, 1, 1};
    if (!make_map_bf16(&tpk, prefix->k, d, s, bx) || !make_map_bf16(&tpv, prefix->v, d, s, bx)) return cudaErrorInvalidValue;
  } else {
    tpk = tk;  // never dereferenced when there is no prefix
    tpv = tv;
    prefix_len = 0;
  }
  TcParams p;
  p.q_heads = q_heads;
  p.q_len = q_len;
  p.pos = pos;
  p.prefix_len = prefix_len;
  p.scale_log2 = scale * 1.4426950408889634f;
  p.prefix_batched = prefix_batched ? 1 : 0;
  p.fused_write = copy_dst ? 1 : 0;
  p.copy_pos = copy_dst ? copy_pos : 0;
  tck = tk;  // never dereferenced without a fused write
  tcv = tv;
  if (copy_dst) {  // destination rows [0, copy_pos + q_len) of every sequence's cache; stores beyond are clipped
    const uint64_t d[4] = {D, static_cast<uint64_t>(copy_pos) + q_len, static_cast<uint64_t>(copy_dst->kv_heads),
                           static_cast<uint64_t>(copy_dst->batch)};
    const uint64_t s[3] = {static_cast<uint64_t>(copy_dst->sr) * 2, static_cast<uint64_t>(copy_dst->sh) * 2,
                           static_cast<uint64_t>(copy_dst->sb) * 2};
    const uint32_t bx[4] = {64, TC_BN, 1, 1};
    if (!make_map_bf16(&tck, copy_dst->k, d, s, bx) || !make_map_bf16(&tcv, copy_dst->v, d, s, bx)) return cudaErrorInvalidValue;
  }
  p.out = out;
  p.lse = lse;
  p.status = status;
  const int head_blocks = q_heads / f.pack;
  p.tokens = f.tokens;
  p.pack = FastDiv(f.pack);
  p.head_blocks = FastDiv(head_blocks);
  p.blocks_per_kv = FastDiv(head_blocks / c.kv_heads);
  p.batch_blocks = FastDiv(static_cast<uint32_t>(c.batch) * head_blocks);
  const int q_tiles = (q_len + f.tokens - 1) / f.tokens;
  p.q_blocks = f.pairs ? (q_tiles + 1) / 2 : q_tiles;
  p.scratch = f.split > 1 ? reinterpret_cast<float*>(static_cast<unsigned char*>(workspace) + SCRATCH_COUNTER_BYTES) : nullptr;
  const int64_t units = static_cast<int64_t>(p.q_blocks) * c.batch * head_blocks;
  cudaError_t e;
  if (f.pairs)
    e = launch_pairs<D>(units, st, tq, tk, tv, tpk, tpv, to, tck, tcv, p);
  else
    switch (f.split) {
      case 8: e = launch_frag<D, 8>(lse, units, st, tq, tk, tv, tpk, tpv, tck, tcv, p); break;
      case 4: e = launch_frag<D, 4>(lse, units, st, tq, tk, tv, tpk, tpv, tck, tcv, p); break;
      case 2: e = launch_frag<D, 2>(lse, units, st, tq, tk, tv, tpk, tpv, tck, tcv, p); break;
      default: e = launch_frag<D, 1>(lse, units, st, tq, tk, tv, tpk, tpv, tck, tcv, p);
    }
  li.launches += 1;
  return e;
}

cudaError_t launch_prefill_tc(const bf16* q, const CacheView& c, const CacheView* prefix, int prefix_len,
                              int q_heads, int q_len, int pos, float scale, float* out, float* lse, int* status,
                              void* workspace, size_t workspace_bytes, cudaStream_t st, LaunchInfo& li) {
  return (c.head_dim == 128 ? launch_tc<128> : launch_tc<64>)(q, c, prefix, prefix_len, false, nullptr, 0, q_heads, q_len, pos,
                                                              scale, out, lse, status, workspace, workspace_bytes, st, li);
}

cudaError_t launch_prefill_tc_fused(const bf16* q, const CacheView& c, const bf16* k_new, const bf16* v_new,
                                    int q_heads, int q_len, int pos, float scale, float* out, float* lse, int* status,
                                    void* workspace, size_t workspace_bytes, cudaStream_t st, LaunchInfo& li) {
  // own segment: the chunk itself, [batch][q_len][kv_heads][D] seen as a cache of q_len rows at position 0;
  // front segment: rows [0, pos) of each sequence's cache
  CacheView own;
  own.k = k_new;
  own.v = v_new;
  own.batch = c.batch;
  own.kv_heads = c.kv_heads;
  own.capacity = q_len;
  own.head_dim = c.head_dim;
  own.sr = static_cast<int64_t>(c.kv_heads) * c.head_dim;
  own.sh = c.head_dim;
  own.sb = static_cast<int64_t>(q_len) * own.sr;
  return (c.head_dim == 128 ? launch_tc<128> : launch_tc<64>)(q, own, pos > 0 ? &c : nullptr, pos, true, &c, pos, q_heads,
                                                              q_len, 0, scale, out, lse, status, workspace,
                                                              workspace_bytes, st, li);
}

}  // namespace jup
