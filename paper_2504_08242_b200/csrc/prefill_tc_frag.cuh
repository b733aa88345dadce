// Chunked-prefill attention, one query tile of 128 rows per CTA, both softmax warpgroups on that tile
// (included by prefill_tc.cu, which holds the parameters, the tensor maps and the dispatch).
//
// TMEM: S0 | S1 | S2 | O (128 columns each).  The MMA issuer runs S(j+3) = Q K(j+3)^T right after O += P(j) V(j),
// into the buffer P(j) is read from, so the scores of a tile are complete a whole tile before its softmax starts:
// the softmax never waits for the tensor pipe, and it can fetch the next tile's scores into registers and reduce
// them to their row maxima while the exponentials of the current tile keep the special-function unit busy.  A
// tile then costs about what its exponentials cost.  The two warpgroups split the tile by rows (warp w owns the 16
// rows 32 (w mod 4) + 16 (w / 4) ..., in the 16x256b fragment layout, see tc_softmax.cuh), so every warp scheduler
// works on every tile; a softmax thread holds two tiles' fragments (the register file is re-divided).
//   warps 0-7 : softmax;  warp 8: loader (TMA);  warp 9: MMA issuer;  warp 10: watcher;  warp 11: idle
// The issuer thread is blocked while the tensor pipe works through its queue, so whatever else it executes adds to
// the pipe's idle time: it tests no barrier and commits once per tile.  The watcher thread waits for each step's
// conditions in the issuer's program order and counts the cleared steps in shared memory (the issuer reads that
// word).  The loader needs no "slot empty" barriers: S(i) complete means S = Q K(i)^T has read K(i)'s slot and
// O += P V of tile i - 3, issued before it, has read V(i-3)'s slot.
#pragma once

namespace jup {

template <int D>
struct FragCfg {
  static constexpr int TILE_BYTES = TC_BM * D * 2;
  static constexpr int PANELS = D / 64;
  static constexpr int STAGES = 3;  // K slots = V slots = S buffers
  static constexpr int SOFTMAX_WARPS = 8, LOADER_WARP = 8, MMA_WARP = 9, WATCH_WARP = 10;
  static constexpr int THREADS = 384;
  static constexpr int REGS_SOFTMAX = 216, REGS_OTHER = 72;  // 2 x 128 x 216 + 128 x 72 = 384 x 168
  static constexpr int O_COL0 = 384;
  static constexpr int SMEM_Q = 0;
  static constexpr int SMEM_K = TILE_BYTES;
  static constexpr int SMEM_V = SMEM_K + STAGES * TILE_BYTES;
  static constexpr int SMEM_BAR = SMEM_V + STAGES * TILE_BYTES;
  static constexpr int SMEM_BYTES = SMEM_BAR + 256 + 1024;  // + slack for 1024-byte alignment
  static_assert(SMEM_BYTES <= 227 * 1024, "shared memory per CTA");
};
template <int D>
constexpr int FRAG_PART_F4 = 2 * TC_BM * D / 8 + TC_BM / 2;  // float4s of one CTA's partial: the accumulator, then (m, l)
enum {
  FB_Q_FULL = 0,
  FB_K_FULL = 1,    // [3] slot j % 3, phase j / 3
  FB_V_FULL = 4,    // [3]
  FB_S_FULL = 7,    // [3] buffer j % 3, phase j / 3
  FB_P_FULL = 10,   // [3] one arrival per softmax warp
  FB_O_READY = 13,  // [3] one barrier (a single phase) for each of the last (up to) three tiles' O += P V: a
                    // thread may come to them long after they completed, which one barrier's parity could not tell
  FB_DRAIN = 16,
  FB_COUNT = 17
};

// C > 1: a thread-block cluster of C CTAs shares a query tile; CTA r walks the r-th of C equal ranges of its KV tiles, and
// the partial (O, m, l) are exchanged through global scratch (L2) around one cluster barrier.
// EXACT: see frag_exp_store_max.
template <int D, int C, bool EXACT>
__global__ void __launch_bounds__(FragCfg<D>::THREADS, 1)
prefill_frag_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                    const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_pk,
                    const __grid_constant__ CUtensorMap tm_pv, const __grid_constant__ CUtensorMap tm_ck,
                    const __grid_constant__ CUtensorMap tm_cv, TcParams p) {
  using Cfg = FragCfg<D>;
  constexpr int TILE_BYTES = Cfg::TILE_BYTES;
  constexpr int STAGES = Cfg::STAGES;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t sQ = smem_base + Cfg::SMEM_Q, sK = smem_base + Cfg::SMEM_K, sV = smem_base + Cfg::SMEM_V;
  const uint32_t sBar = smem_base + Cfg::SMEM_BAR;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_gen + Cfg::SMEM_BAR + 8 * FB_COUNT);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + Cfg::SMEM_BAR + 8 * FB_COUNT + 8);
  const uint32_t go_count = sBar + 8u * FB_COUNT + 16u;  // steps the watcher has cleared for the issuer
  static_assert(8 * FB_COUNT + 24 <= 256, "barrier block");
  auto bar = [&](int i) { return sBar + 8u * i; };
  // barrier (of a family of three) and parity of tile j
  auto bar3 = [&](int family, int j) { return sBar + 8u * (family + j % STAGES); };
  auto par3 = [](int j) { return static_cast<uint32_t>(j / STAGES) & 1u; };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // ---- work assignment: heaviest query tiles first
  constexpr bool SPLIT = C > 1;
  const int crank = SPLIT ? static_cast<int>(cluster_ctarank()) : 0;
  const int work = blockIdx.x / C;
  // (recomputed behind the walk, so that the softmax does not carry it through)
  struct Place {
    int b, h0, hk, t0, t1;  // sequence, first head, kv head, tokens [t0, t1) of the query tile
    bool first_heads;       // of their group
  };
  auto place = [&](int w) {
    int bh, hb, hr;
    Place a;
    const int qblk = p.q_blocks - 1 - p.batch_blocks.divmod(w, bh);
    a.b = p.head_blocks.divmod(bh, hb);
    a.hk = p.blocks_per_kv.divmod(hb, hr);
    a.first_heads = hr == 0;
    a.h0 = hb * static_cast<int>(p.pack.d);
    a.t0 = qblk * p.tokens;
    a.t1 = min(p.q_len, a.t0 + p.tokens);
    return a;
  };
  const Place at = place(work);
  // KV tiles 0..Tp-1 come from the front segment (every row sees them, no causal limit), the rest from the own one
  const int Tp = (p.prefix_len + TC_BN - 1) / TC_BN;
  const int T_all = Tp + (p.pos + at.t1 + TC_BN - 1) / TC_BN;  // >= 1
  const int g0 = SPLIT ? T_all * crank / C : 0;  // this CTA's tiles are g0 .. g0 + T - 1 of them
  const int T = SPLIT ? T_all * (crank + 1) / C - g0 : T_all;  // (may be 0 with C > 1)
  // O += P V of tile j is followed by S(j+3), whose barrier then also says that the accumulator holds tile j; the
  // last tiles have no S(j+3) and complete one of the accumulator's own barriers instead, the first for tile o0
  const int o0 = max(T - STAGES, 0);

  if (threadIdx.x == 0) {
    for (int i = 0; i < FB_COUNT; ++i)
      mbar_init(bar(i), (i >= FB_P_FULL && i < FB_P_FULL + STAGES) ? static_cast<uint32_t>(Cfg::SOFTMAX_WARPS) : 1u);
    *abort_flag = 0;
    *reinterpret_cast<volatile int*>(smem_gen + Cfg::SMEM_BAR + 8 * FB_COUNT + 16) = 0;
    mbar_fence_init();
  }
  if (warp == Cfg::MMA_WARP) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
    tmem_relinquish();
  } else if (warp == Cfg::LOADER_WARP && lane == 0) {
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_k);
    tma_prefetch_desc(&tm_v);
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
      // (rows of the Q tile beyond its pack x tokens are never written: they belong to no query, and whatever the
      // tensor cores make of them is never used)
      mbar_expect_tx(bar(FB_Q_FULL), p.pack.d * p.tokens * (D * 2u));
#pragma unroll
      for (int c = 0; c < Cfg::PANELS; ++c) tma_load_4d(sQ + c * TC_PANEL_BYTES, &tm_q, bar(FB_Q_FULL), c * 64, at.h0, at.t0, at.b);
      bool ok = true;
      int k_issued = 0, v_issued = 0;
      auto load = [&](bool is_v, int j) {
        const int s = j % STAGES;
        const uint32_t full = bar3(is_v ? FB_V_FULL : FB_K_FULL, j);
        const uint32_t dst = (is_v ? sV : sK) + s * TILE_BYTES;
        const int g = g0 + j;
        const CUtensorMap* m = g < Tp ? (is_v ? &tm_pv : &tm_pk) : (is_v ? &tm_v : &tm_k);
        const int krow = (g < Tp ? g : g - Tp) * TC_BN, kb = (g < Tp && !p.prefix_batched) ? 0 : at.b;
        mbar_expect_tx(full, TILE_BYTES);
#pragma unroll
        for (int c = 0; c < Cfg::PANELS; ++c) tma_load_4d(dst + c * TC_PANEL_BYTES, m, full, c * 64, krow, at.hk, kb);
        if (is_v) v_issued = j + 1;
        else k_issued = j + 1;
      };
      // Fused KVCache write: a tile of the chunk's own K/V goes from its slots to the cache with tiled stores once it has
      // landed, before the slot is refilled: by the CTA whose query tile holds the tile's last token (of each group's
      // first heads; with C > 1 the CTA of the cluster that walks the tile); rows beyond copy_pos + q_len are clipped
      // by the tensor maps.
      const bool writer = p.fused_write != 0 && at.first_heads;
      const int own0 = Tp + at.t0 / TC_BN - g0, own1 = writer ? Tp + own_tiles_end(at.t1, p.q_len) - g0 : own0;
      auto own = [&](int j) { return j >= own0 && j < own1; };
      auto store_own = [&](bool is_v, int j) {
        ok = ok && mbar_wait(bar3(is_v ? FB_V_FULL : FB_K_FULL, j), par3(j), abort_flag, p.status);
        if (!ok) return;
        const uint32_t src = (is_v ? sV : sK) + (j % STAGES) * TILE_BYTES;
        const CUtensorMap* m = is_v ? &tm_cv : &tm_ck;
        const int row = p.copy_pos + (g0 + j - Tp) * TC_BN;
#pragma unroll
        for (int c = 0; c < Cfg::PANELS; ++c) tma_store_4d(m, src + c * TC_PANEL_BYTES, c * 64, row, at.hk, at.b);
        tma_store_commit();
        tma_store_wait_read();
      };
      for (int j = 0; j < STAGES && j < T; ++j) {
        load(false, j);
        load(true, j);
      }
      for (int i = 0; i < T && ok; ++i) {
        ok = mbar_wait(bar3(FB_S_FULL, i), par3(i), abort_flag, p.status);
        if (!ok) break;
        if (own(i)) store_own(false, i);
        if (i >= STAGES && own(i - STAGES)) store_own(true, i - STAGES);
        if (!ok) break;
        if (i + STAGES < T) load(false, i + STAGES);  // K(i)'s slot
        if (i >= STAGES) load(true, i);               // V(i-3)'s slot
      }
      for (int i = max(0, T - STAGES); i < T && ok; ++i)
        if (own(i)) store_own(true, i);
      if (*abort_flag) {
        // wait (bounded) until every copy this thread started has landed before shared memory is released
        int dummy = 0;
        volatile int* none = &dummy;
        for (int j = max(0, k_issued - STAGES); j < k_issued; ++j) mbar_wait(bar3(FB_K_FULL, j), par3(j), none, nullptr);
        for (int j = max(0, v_issued - STAGES); j < v_issued; ++j) mbar_wait(bar3(FB_V_FULL, j), par3(j), none, nullptr);
        mbar_wait(bar(FB_Q_FULL), 0, none, nullptr);
      }
    }
    __syncwarp();
  } else if (warp == Cfg::MMA_WARP) {
    // =============================================================== MMA issuer
    // Steps (each cleared by the watcher):  S(0), S(1), S(2);  then per tile j:  O += P(j) V(j),  S(j+3).
    reg_dec<Cfg::REGS_OTHER>();
    if (elect_one()) {
      constexpr uint32_t idesc_qk = tc_idesc_bf16(TC_BM, TC_BN, false, false);
      constexpr uint32_t idesc_pv = tc_idesc_bf16(TC_BM, D, false, true);
      const uint32_t q_lo = tc_desc_lo(sQ, 16), k_lo0 = tc_desc_lo(sK, 16), v_lo0 = tc_desc_lo(sV, TC_PANEL_BYTES);
      const uint32_t o_col = tmem + Cfg::O_COL0;
      // slot of K and V and S buffer are all j mod 3
      auto issue_qk = [&](int s) {  // S[s] = Q K[s]^T
        const uint32_t k_lo = k_lo0 + s * (TILE_BYTES >> 4);
        const uint32_t d = tmem + s * 128;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          const uint32_t off = ((ks >> 2) * TC_PANEL_BYTES + (ks & 3) * 32) >> 4;
          tc_mma_ss_lo(d, q_lo + off, k_lo + off, idesc_qk, ks > 0);
        }
      };
      auto issue_pv = [&](int s, bool first) {  // O (+)= P[s] V[s]
        const uint32_t v_lo = v_lo0 + s * (TILE_BYTES >> 4);
        const uint32_t a = tmem + s * 128;
#pragma unroll
        for (int ks = 0; ks < TC_BN / 16; ++ks)
          tc_mma_ts_lo(o_col, a + ks * 8, v_lo + ks * (2048 >> 4), idesc_pv, (!first || ks > 0));
      };
      int cleared = 0, step = 0;  // steps the watcher is known to have cleared / steps taken
      bool ok = true;
      auto next_step = [&] {
        ++step;
        if (cleared < step) {
          cleared = count_spin_wait(go_count, step, abort_flag, p.status);
          ok = cleared >= 0;
        }
        tc_fence_after();
        return ok;
      };
      for (int j = 0; j < STAGES && j < T && ok; ++j) {
        if (!next_step()) break;
        issue_qk(j);
        tc_commit(bar(FB_S_FULL + j));
      }
      int s = 0;
      for (int j = 0; j < T && ok; ++j) {
        if (!next_step()) break;
        issue_pv(s, j == 0);
        if (j + STAGES < T) {
          issue_qk(s);
          tc_commit(bar(FB_S_FULL + s));
        } else {
          tc_commit(bar(FB_O_READY + j - o0));
        }
        s = s + 1 == STAGES ? 0 : s + 1;
      }
      if (!ok) {  // make sure no MMA of this thread is still running before TMEM and smem go away
        int dummy = 0;
        tc_commit(bar(FB_DRAIN));
        mbar_wait(bar(FB_DRAIN), 0, &dummy, nullptr);
      }
    }
    __syncwarp();
  } else if (warp == Cfg::WATCH_WARP) {
    // =============================================================== watcher (see the MMA issuer)
    reg_dec<Cfg::REGS_OTHER>();
    if (lane == 0) {
      bool ok = mbar_wait(bar(FB_Q_FULL), 0, abort_flag, p.status);
      int step = 0;
      auto landed = [&](int family, int j) { return mbar_wait(bar3(family, j), par3(j), abort_flag, p.status); };
      for (int j = 0; j < STAGES && j < T && ok; ++j) {
        ok = landed(FB_K_FULL, j);
        if (ok) count_publish(go_count, ++step);
      }
      for (int j = 0; j < T && ok; ++j) {
        ok = landed(FB_V_FULL, j);
        if (ok && j + STAGES < T) ok = landed(FB_K_FULL, j + STAGES);
        ok = ok && mbar_spin_wait(bar3(FB_P_FULL, j), par3(j), abort_flag, p.status);
        if (!ok) break;
        count_publish(go_count, ++step);
      }
    }
    __syncwarp();
  } else if (warp < Cfg::SOFTMAX_WARPS) {
    // =============================================================== softmax: 16 rows per warp
    reg_inc<Cfg::REGS_SOFTMAX>();
    const int lane0 = (warp & 3) * 32 + (warp >> 2) * 16;  // first TMEM lane (row of the tile) of this warp
    const int col0 = 2 * (lane & 3);
    const uint32_t taddr = tmem + (static_cast<uint32_t>(lane0) << 16);
    const uint32_t tO = taddr + Cfg::O_COL0;
    // Columns of tile 0 that this thread's rows would see if they were all of the own segment (its causal limit), or all
    // of the front segment (its end); every tile further on it is 128 fewer.
    int own_cols[2];
#pragma unroll
    for (int e = 0; e < 2; ++e)
      own_cols[e] = p.pos + min(at.t0 + p.pack.div(lane0 + (lane >> 2) + 8 * e), p.q_len - 1) + 1 + (Tp - g0) * TC_BN;
    const int front_cols = p.prefix_len - g0 * TC_BN;
    const float c = p.scale_log2;
    float m_ref[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
    float mxs[2];
    bool ok = true;
    // the accumulator holds tile j - 1 (needed before its rows are rescaled at tile j)
    auto wait_o_before = [&](int j) {
      if (j + 2 < T) return mbar_wait(bar3(FB_S_FULL, j + 2), par3(j + 2), abort_flag, p.status);
      return mbar_wait(bar(FB_O_READY + j - 1 - o0), 0, abort_flag, p.status);
    };
    // Scores of tile j into fragments (asynchronous: the registers may only be used after the load was waited for).
    auto fetch = [&](int j, uint32_t (&sv)[64]) {
      ok = mbar_spin_wait(bar3(FB_S_FULL, j), par3(j), abort_flag, p.status);
      if (!ok) return;
      tc_fence_after();
      tmem_ld_16x256b_x16(taddr + (j % STAGES) * 128, sv);
    };
    // Columns >= nvalid of a row are hidden: the end of the front segment in its last tile, the causal limit afterwards.
    int nvalid[2];
    auto tile_masked = [&](int j) {  // warp-uniform; fills nvalid
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int front = front_cols - j * TC_BN;
        nvalid[e] = front > 0 ? front : own_cols[e] - j * TC_BN;
      }
      return __any_sync(0xffffffffu, nvalid[0] < TC_BN || nvalid[1] < TC_BN) != 0;
    };
    auto apply_mask = [&](uint32_t (&sv)[64]) {
#pragma unroll
      for (int k = 0; k < 16; ++k)
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (8 * k + col0 + (i & 1) >= nvalid[i >> 1]) sv[4 * k + i] = 0xff800000u;  // -inf
    };
    // One tile: cur holds its masked scores and mxs its maxima; nxt is the next tile's fetch in flight, whose maxima
    // are worked out between this tile's exponentials; afterwards the fetch of the tile after that goes into cur.
    auto tile = [&](int j, uint32_t (&cur)[64], uint32_t (&nxt)[64]) {
      if (!frag_decide<D>(mxs, m_ref, l, tO, j, [&] { return wait_o_before(j); })) {
        ok = false;
        return;
      }
      const bool next_masked = j + 1 < T && tile_masked(j + 1);
      float mxs_next[2];
      frag_exp_store_max<EXACT>(cur, taddr + (j % STAGES) * 128, c, m_ref, l, nxt, next_masked, [&] { apply_mask(nxt); }, mxs_next);
      mxs[0] = mxs_next[0];
      mxs[1] = mxs_next[1];
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar3(FB_P_FULL, j));
      if (j + 2 < T) fetch(j + 2, cur);
    };
    uint32_t fa[64], fb[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) fb[i] = 0u;  // read (and ignored) as "next tile" when there is none
    if (!SPLIT || T > 0) fetch(0, fa);
    if (ok && (!SPLIT || T > 0)) {
      tc_wait_ld_into(fa);
      const bool masked0 = tile_masked(0);
      frag_mask_max(fa, masked0, [&](int e, int col) { return col < nvalid[e]; }, col0, c, mxs);
      if (T > 1) fetch(1, fb);
    }
    for (int j = 0; j < T && ok; j += 2) {
      tile(j, fa, fb);
      if (j + 1 < T && ok) tile(j + 1, fb, fa);
    }
    tc_wait_ld();  // (no fetch is left in flight; the registers are dead)
    pdl_launch_dependents();  // the next kernel of the stream may start its own set-up now
    if (!SPLIT || T > 0)
      ok = ok && mbar_wait(bar(FB_O_READY + T - 1 - o0), 0, abort_flag, p.status);  // the accumulator is final
    tc_fence_after();
    float inv[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      l[e] += __shfl_xor_sync(0xffffffffu, l[e], 1);
      l[e] += __shfl_xor_sync(0xffffffffu, l[e], 2);
      inv[e] = 1.f / l[e];
    }
    if constexpr (SPLIT) {
      const int work = known_here(blockIdx.x) / C, crank = static_cast<int>(cluster_ctarank());
      // ---- this CTA's unnormalised partial -> scratch, in fragment order ([column step][thread] float4, so that every
      // store of a warp writes 512 contiguous bytes), and (m, l) per row
      float4* gpart = reinterpret_cast<float4*>(p.scratch) + (static_cast<size_t>(work) * C + crank) * FRAG_PART_F4<D>;
      float2* gml = reinterpret_cast<float2*>(gpart + 2 * TC_BM * D / 8);
#pragma unroll
      for (int hh = 0; hh < Cfg::PANELS; ++hh) {
        uint32_t o[32];
        if (T > 0) {
          tmem_ld_16x256b_x8(tO + hh * 64, o);
          tc_wait_ld();
        } else {  // (a CTA without tiles never wrote its accumulator)
#pragma unroll
          for (int k = 0; k < 32; ++k) o[k] = 0u;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
          gpart[(hh * 8 + k) * 256 + threadIdx.x] =
              make_float4(__uint_as_float(o[4 * k]), __uint_as_float(o[4 * k + 1]), __uint_as_float(o[4 * k + 2]),
                          __uint_as_float(o[4 * k + 3]));
      }
      if ((lane & 3) == 0) {
#pragma unroll
        for (int e = 0; e < 2; ++e) gml[lane0 + (lane >> 2) + 8 * e] = make_float2(T > 0 ? m_ref[e] : -INFINITY, l[e]);
      }
      __threadfence();  // visible to the cluster before its barrier is passed
      cluster_sync_all();  // release / acquire over the cluster: the partials of every CTA are visible
      // ---- merge over the cluster (here and not behind the role branches, where the code would have to make do with the
      // other roles' registers).  CTA r finishes the fragments of the softmax threads [256 r / C, 256 (r + 1) / C), i.e.
      // the rows of 8 / C warps: thread t of them every C-th column step, all loads in flight at once; the sums run in
      // CTA order.
      const bool cta_ok = *abort_flag == 0 && *reinterpret_cast<volatile int*>(p.status) == 0;  // nobody gave up on a wait
      constexpr int PER = 256 / C, STEPS = D / 8, MINE = STEPS / C;
      const int sub = threadIdx.x / PER, t = PER * crank + threadIdx.x % PER;
      const int w_t = t >> 5, l_t = t & 31;
      const int r0 = (w_t & 3) * 32 + (w_t >> 2) * 16 + (l_t >> 2);  // rows r0 and r0 + 8 of the tile
      const float4* upart = reinterpret_cast<const float4*>(p.scratch) + static_cast<size_t>(work) * C * FRAG_PART_F4<D>;
      float2 ml[2][C];
      float4 v[MINE][C];
#pragma unroll
      for (int cr = 0; cr < C; ++cr)
#pragma unroll
        for (int e = 0; e < 2; ++e)
          ml[e][cr] = __ldcg(reinterpret_cast<const float2*>(upart + cr * FRAG_PART_F4<D> + 2 * TC_BM * D / 8) + r0 + 8 * e);
#pragma unroll
      for (int u = 0; u < MINE; ++u)
#pragma unroll
        for (int cr = 0; cr < C; ++cr) v[u][cr] = __ldcg(upart + cr * FRAG_PART_F4<D> + (u * C + sub) * 256 + t);
      float wgt[2][C], m[2], lsum[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        m[e] = -INFINITY;
#pragma unroll
        for (int cr = 0; cr < C; ++cr) m[e] = fmaxf(m[e], ml[e][cr].x);  // (-inf: all its tiles were hidden from the row)
        lsum[e] = 0.f;
#pragma unroll
        for (int cr = 0; cr < C; ++cr) {
          wgt[e][cr] = fast_exp2(ml[e][cr].x - m[e]);
          lsum[e] = fmaf(wgt[e][cr], ml[e][cr].y, lsum[e]);
        }
        const float inv = 1.f / lsum[e];
#pragma unroll
        for (int cr = 0; cr < C; ++cr) wgt[e][cr] *= inv;
      }
      int tok[2], hd[2];
      float* dst[2];
      const Place at = place(known_here(blockIdx.x) / C);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        tok[e] = at.t0 + p.pack.divmod(known_here(r0 + 8 * e), hd[e]);
        hd[e] += at.h0;
        dst[e] = p.out + ((static_cast<int64_t>(at.b) * p.q_len + tok[e]) * p.q_heads + hd[e]) * D + 2 * (l_t & 3);
      }
#pragma unroll
      for (int u = 0; u < MINE; ++u) {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int cr = 0; cr < C; ++cr) {
          acc.x = fmaf(wgt[0][cr], v[u][cr].x, acc.x);
          acc.y = fmaf(wgt[0][cr], v[u][cr].y, acc.y);
          acc.z = fmaf(wgt[1][cr], v[u][cr].z, acc.z);
          acc.w = fmaf(wgt[1][cr], v[u][cr].w, acc.w);
        }
        const int col = 8 * (u * C + sub);
        if (cta_ok && tok[0] < at.t1) *reinterpret_cast<float2*>(dst[0] + col) = make_float2(acc.x, acc.y);
        if (cta_ok && tok[1] < at.t1) *reinterpret_cast<float2*>(dst[1] + col) = make_float2(acc.z, acc.w);
      }
      if (cta_ok && p.lse && sub == 0 && (l_t & 3) == 0) {
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (tok[e] < at.t1)
            p.lse[(static_cast<int64_t>(at.b) * p.q_heads + hd[e]) * p.q_len + tok[e]] =
                (m[e] + log2f(lsum[e])) * 0.69314718055994530942f;
      }
    } else {
      // ---- output: O / l straight from the fragments (a row's four threads write 32 contiguous bytes per repeat)
      int tok[2], hd[2];  // token and head of this thread's rows
      float* dst[2];
      const Place at = place(known_here(blockIdx.x) / C);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        tok[e] = at.t0 + p.pack.divmod(known_here(lane0 + (lane >> 2) + 8 * e), hd[e]);
        hd[e] += at.h0;
        dst[e] = p.out + ((static_cast<int64_t>(at.b) * p.q_len + tok[e]) * p.q_heads + hd[e]) * D + col0;
      }
#pragma unroll
      for (int hh = 0; hh < Cfg::PANELS; ++hh) {
        uint32_t o[32];
        tmem_ld_16x256b_x8(tO + hh * 64, o);
        tc_wait_ld();
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (!ok || tok[e] >= at.t1) continue;
#pragma unroll
          for (int k = 0; k < 8; ++k)
            *reinterpret_cast<float2*>(dst[e] + hh * 64 + 8 * k) =
                make_float2(__uint_as_float(o[4 * k + 2 * e]) * inv[e], __uint_as_float(o[4 * k + 2 * e + 1]) * inv[e]);
        }
      }
      if (ok && p.lse && (lane & 3) == 0) {
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (tok[e] < at.t1)
            p.lse[(static_cast<int64_t>(at.b) * p.q_heads + hd[e]) * p.q_len + tok[e]] =
                (m_ref[e] + log2f(l[e])) * 0.69314718055994530942f;
      }
    }
  } else {
    reg_dec<Cfg::REGS_OTHER>();  // the idle warp of the third warpgroup: the re-division is a warpgroup's decision
  }

  // (every thread of every CTA passes the cluster's barrier, whatever happened above)
  if constexpr (SPLIT)
    if (warp >= Cfg::SOFTMAX_WARPS) cluster_sync_all();

  // ---- tear-down
  tc_fence_before();
  __syncthreads();
  if (warp == Cfg::MMA_WARP) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace jup
