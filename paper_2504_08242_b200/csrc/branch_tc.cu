// Branch attention with many stacked query rows per kv head on the 5th-generation tensor cores (paper Sec. V-A,
// Fig. 7 step 3: the k draft tokens of every request are verified in one pass; Sec. V-B, Fig. 8: all
// point-extending requests share the prompt's KVCache).
//
// The stacked rows of a kv head -- (branch, draft token, head of the group), in that order -- are
// cut into row tiles of at most 128 rows: whole branches while a branch has at most 128 rows (the same number
// of branches in every tile, so that the tiles carry equal work), else 128-row slices of one branch.
// A unit = (kv head, row tile).  Every row belongs to one branch and may see the shared prefix plus that
// branch's suffix, so a row keeps ONE online-softmax state in its TMEM lane while the unit walks
//     prefix | suffix of the tile's first branch | ... | suffix of its last branch
// in tiles of 128 keys: a prefix tile is visible to every row, a suffix tile to the rows of its branch below
// their causal limit (or tree mask).  A prefix K/V tile is therefore fetched once per row tile, not once per branch.
//
// A unit is walked by one CTA or shared by C CTAs, a thread-block cluster: the prefix tiles are cut into equal contiguous
// ranges, one per CTA, and so are the suffix tiles (the prefix share does not depend on the device-side lengths,
// so its first loads are in flight while the lengths arrive).  Inside a CTA:
//   loader warp  : TMA (tiled, 128-byte swizzle) Q once -- one box [tokens][G heads][64] lands in stacked-row
//                  order -- then the K/V tiles of the CTA's list, in the order of their use, into one ring of slots
//   patch warp   : passes landed V tiles on to the MMA issuer, after zeroing the rows of a last, partial 16-key group
//                  that are no keys (rows at or beyond a branch's device-side length, which TMA cannot know: their
//                  weights are 0, but 0 x NaN must not reach an accumulator)
//   MMA warps    : one thread issues S = Q K^T, another O += P V (tcgen05.mma over the 16-key groups that hold keys)
//   softmax WGs  : two warpgroups run two independent online-softmax streams over the even and the odd tiles of
//                  the CTA's list, which mixes prefix and suffix tiles (one thread per row); a warp none of whose rows sees a tile only zeroes its P
// TMEM (512 columns): O_0 | O_1 (128 each) | S (128) | P_0 | P_1 (64 each); the one S buffer goes back and forth between
// the streams, as in the two-tile prefill kernel.
// With the fused KVCache write the step's K/V block of all the tile's branches is one more tile, fetched from k_new /
// v_new with one box (their rows lie there as [token][kv head], so the tile's branches follow one another) and masked by
// branch; the unit that owns a branch also copies the block's rows into the cache.
// At the end the two streams of a CTA are merged in registers.  With one CTA per unit the rows are normalised
// and written out.  Otherwise every CTA writes its rows' unnormalised (O, m, l) to scratch (L2), and behind ONE
// cluster barrier CTA r of the cluster finishes a contiguous slice of the rows: it adds the partials in CTA
// order -- the result never depends on timing -- normalises and writes the output.  (Pushing the partials into the
// owner's shared memory instead was measured: 64 KB per CTA took 2.3 us over distributed shared memory, twice the
// trip through L2.)  No atomics, no second launch, nothing waits on a flag.
// All mbarrier waits are bounded; on expiry the CTA sets the status word, drains its own copies and MMAs,
// frees TMEM and returns (every thread still passes the cluster barriers).
#include <algorithm>

#include "host_checks.h"
#include "kernels.h"
#include "tc_common.cuh"
#include "tc_softmax.cuh"
#include "tile_ring.h"
#include "tmap.h"

namespace jup {

constexpr int BT_BM = 128;             // stacked rows per tile (at most)
constexpr int BT_BN = 128;             // keys per KV tile
constexpr int BT_PANEL_BYTES = 16384;  // 128 rows x 64 elements
constexpr int BT_MAX_SLOTS = 12;
constexpr int BT_MAX_BRANCHES = 32;    // branches in one row tile
constexpr int BT_ML_FLOATS = BT_BM * 2;  // one CTA's (m, l) pairs
// Layers of one call share a launch from this many on.
constexpr int BT_MIN_BATCHED_LAYERS = 3;

struct BtParams {
  int n_branches, q_len, q_heads, group, kv_heads;
  FastDiv by_group, by_q_len, by_row_tiles, by_layer_units;
  int prefix_len, max_suffix_len;
  int whole_units;        // units of all layers that one CTA walks
  int branches_per_tile;  // whole branches per row tile (slices_per_branch == 1)
  int slices_per_branch;  // > 1: a branch has more than 128 rows and is cut into 128-row slices
  int box_tokens;         // tokens in the Q box
  int box_keys;           // keys in the box of the step's block: all of the row tile's branches
  float scale_log2;
  long long wait_limit;
  const int32_t* d_suffix_len;
  const uint32_t* tree_mask;  // nullable: [n_branches][q_len] ancestor bit masks of the draft block
  int64_t sb, sh, sr;         // strides of the suffix cache
  int* status;
  float* part;  // [shared units][C][D / 4 column chunks][128 rows] float4, a CTA's partial accumulator
  float* ml;    // [shared units][C][128 rows] (m, l)
};

// What differs between the layers of one launch.
struct BtLayer {
  CUtensorMap tm_q, tm_pk, tm_pv, tm_sk, tm_sv;
  CUtensorMap tm_nk, tm_nv;  // k_new / v_new
  const bf16* k_new;  // nullable: fused KVCache write, [n_branches][q_len][kv_heads][D]
  const bf16* v_new;
  bf16* k_cache;      // the suffix cache (written only with the fused write)
  bf16* v_cache;
  float* out;
  float* lse;
};
template <int NL>
struct BtLayers {
  BtLayer l[NL];
};

// shared memory: [Q][K/V slots][barriers, flags][lengths and tile counts of the row tile's branches]
template <int D>
struct BtCfg {
  static constexpr int SLOTS = D == 128 ? 6 : 12;
  // Prefix tiles at the front of a CTA's list: as many as the first SLOTS loads belong to (K_0 K_1 V_0 K_2 V_1 ..
  // K_SLOTS/2), and even: a pair of tiles is one per stream.  (head_dim 64, 16 branches x 20 rows, 8 layers, prefix 3000,
  // 73.0 us; with 4 tiles in front and only their loads early 73.5.)
  static constexpr int LEAD = D == 128 ? 4 : 8;
  static_assert(LEAD % 2 == 0 && 2 * LEAD - 1 >= SLOTS, "every slot is filled before the lengths are known");
  static constexpr int TILE_BYTES = BT_BN * D * 2;
  static constexpr int PANELS = D / 64;
  static constexpr int CH = D / 8;  // 16-byte pieces per K/V row
  static constexpr int RECV_STRIDE = D + 4;  // one CTA per unit: floats per staged row: O, then (m, l), padded against bank conflicts
  static constexpr int PART_FLOATS = BT_BM * D;  // one CTA's partial accumulator
  static constexpr int SMEM_Q = 0;
  static constexpr int SMEM_KV = TILE_BYTES;
  static constexpr int SMEM_BAR = SMEM_KV + SLOTS * TILE_BYTES;
  static constexpr int SMEM_LEN = SMEM_BAR + 512;
  static constexpr int SMEM_BYTES = SMEM_LEN + 2 * BT_MAX_BRANCHES * 4 + 1024;  // + slack for 1024-byte alignment
  static_assert(SMEM_BYTES <= 227 * 1024, "shared memory per CTA");
  static_assert(SLOTS <= BT_MAX_SLOTS && BT_BM * RECV_STRIDE * 4 <= SLOTS * TILE_BYTES, "the staged rows fit in the slots");
};
// TMEM columns: O_0 | O_1 | S | P_0 | P_1
constexpr int BT_O_COL0 = 0, BT_S_COL = 256, BT_P_COL0 = 384;
// The register file is re-divided: a softmax thread holds a whole score row; 2 x 128 x 208 + 128 x 88 = 384 x 168.
constexpr int BT_REGS_SOFTMAX = 208, BT_REGS_OTHER = 88;
constexpr int BT_LOADER_WARP = 8,  // warps 0..7: the two softmax warpgroups
              BT_QK_WARP = 9, BT_PV_WARP = 10, BT_PATCH_WARP = 11;
constexpr int BT_THREADS = 32 * 12;

enum {
  BT_Q_FULL = 0,
  BT_FULL = 1,                           // [SLOTS] a K or V tile has landed
  BT_EMPTY = BT_FULL + BT_MAX_SLOTS,     // [SLOTS] and its MMAs are done
  BT_S_FULL = BT_EMPTY + BT_MAX_SLOTS,   // [2] one per stream
  BT_O_READY = BT_S_FULL + 2,            // [2]
  BT_DRAIN = BT_O_READY + 2,             // [2] one per issuing thread
  BT_K_SEEN = BT_DRAIN + 2,              // [2] K_0, and the K tile in front of the last V tile, have landed (a single phase)
  BT_BAR_COUNT = BT_K_SEEN + 2
};

// One entry of a CTA's tile list.
constexpr int BT_PREFIX = -1, BT_NEW = -2;
struct BtTile {
  int seg;    // branch as an index into the row tile's branches; BT_PREFIX; BT_NEW: the step's block of all of them
  int tile;   // tile number inside the segment
  int valid;  // keys in it (1..128): the tensor cores work on the 16-key groups that hold them
  // V rows in the last group that are no keys (dead cache rows, or not loaded at all) and must read as zero, so that
  // 0 x NaN never reaches an accumulator.  (The prefix's tensor map ends with the prefix and zero-fills.)
  __device__ __forceinline__ bool patch() const { return seg != BT_PREFIX && (valid & 15) != 0; }
  __device__ __forceinline__ int groups() const { return (valid + 15) >> 4; }
};

// C: cluster size = CTAs per shared unit.  The units of all layers are numbered through; the first whole_units of them are
// walked by one CTA each (C of them make a cluster only in name), the others by a cluster each.
template <int D, int NL, int C>
__global__ void __launch_bounds__(BT_THREADS, 1)
branch_tc_kernel(const __grid_constant__ BtLayers<NL> layers, const BtParams p) {
  using Cfg = BtCfg<D>;
  constexpr int TILE_BYTES = Cfg::TILE_BYTES;
  constexpr int SLOTS = Cfg::SLOTS;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t sQ = smem_base + Cfg::SMEM_Q, sKV = smem_base + Cfg::SMEM_KV;
  const uint32_t sBar = smem_base + Cfg::SMEM_BAR;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_gen + Cfg::SMEM_BAR + 8 * BT_BAR_COUNT);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + Cfg::SMEM_BAR + 8 * BT_BAR_COUNT + 8);
  volatile int* suffix_share = reinterpret_cast<volatile int*>(smem_gen + Cfg::SMEM_BAR + 8 * BT_BAR_COUNT + 16);  // [2]
  const uint32_t v_ready = sBar + 8 * BT_BAR_COUNT + 24;  // how many V tiles of the list have landed and are patched
  const uint32_t qk_turn = v_ready + 4;  // odd while a batch of scores is being issued
  int* len_s = reinterpret_cast<int*>(smem_gen + Cfg::SMEM_LEN);  // clamped suffix length of the tile's branches
  int* cum_s = len_s + BT_MAX_BRANCHES;                         // one past the last suffix tile of each
  auto bar = [&](int i) { return sBar + 8u * i; };
  const long long wl = p.wait_limit;

  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const bool shared = C > 1 && blockIdx.x >= static_cast<unsigned>(p.whole_units);
  const int share = shared ? (blockIdx.x - p.whole_units) / C : 0;  // number among the shared units
  const int crank = shared ? blockIdx.x % C : 0;                    // rank in its cluster (whole_units is a multiple of C)
  const int log2c = shared ? (C == 8 ? 3 : C / 2) : 0;              // log2 of the CTAs that walk this unit
  int unit = shared ? p.whole_units + share : blockIdx.x, rt;
  const BtLayer& L_ = layers.l[NL == 1 ? 0 : p.by_layer_units.divmod(unit, unit)];
  const int hk = p.by_row_tiles.divmod(unit, rt);
  const int n = p.q_len, G = p.group;
  // ---- the row tile: tokens [tok0, tok0 + ntok) of the stacked (branch, draft row) order, all heads of the group
  int b_first, nb, tok0, ntok;
  if (p.slices_per_branch == 1) {
    b_first = rt * p.branches_per_tile;
    nb = min(p.branches_per_tile, p.n_branches - b_first);
    tok0 = b_first * n;
    ntok = nb * n;
  } else {
    b_first = rt / p.slices_per_branch;
    nb = 1;
    const int first = (rt % p.slices_per_branch) * (BT_BM / G);
    tok0 = b_first * n + first;
    ntok = min(BT_BM / G, n - first);
  }
  const int rows_here = ntok * G;
  const int P = p.prefix_len;
  const bool fused = L_.k_new != nullptr;
  // this CTA's share of the prefix tiles: known without any memory access
  const int Tp = (P + BT_BN - 1) / BT_BN;
  const int p0 = (Tp * crank) >> log2c, npre = ((Tp * (crank + 1)) >> log2c) - p0;

  // ---- set-up
  if (threadIdx.x == 0) {
    for (int i = 0; i < BT_BAR_COUNT; ++i) mbar_init(bar(i), 1u);
    *abort_flag = 0;
    count_publish(v_ready, 0);
    count_publish(qk_turn, 0);
    mbar_fence_init();
  }
  if (warp == BT_QK_WARP) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
    tmem_relinquish();
  } else if (warp == BT_LOADER_WARP && lane == 0) {
    tma_prefetch_desc(&L_.tm_q);
    tma_prefetch_desc(&L_.tm_sk);
    tma_prefetch_desc(&L_.tm_sv);
    if (fused) {
      tma_prefetch_desc(&L_.tm_nk);
      tma_prefetch_desc(&L_.tm_nv);
    }
    if (Tp > 0) {
      tma_prefetch_desc(&L_.tm_pk);
      tma_prefetch_desc(&L_.tm_pv);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = warp_uniform(*tmem_slot);
  pdl_wait();  // everything above overlapped the previous kernel's tail; global memory is touched from here on

  // K (V) of list entry e into a slot
  auto load_kv = [&](bool is_v, int slot, const BtTile& e) {
    const uint32_t dst = sKV + slot * TILE_BYTES, full = bar(BT_FULL + slot);
    if (e.seg == BT_NEW) {  // token-major rows of the row tile's branches, one box
      mbar_expect_tx(full, static_cast<uint32_t>(p.box_keys) * (D * 2u));
      const CUtensorMap* m = is_v ? &L_.tm_nv : &L_.tm_nk;
#pragma unroll
      for (int c = 0; c < Cfg::PANELS; ++c) tma_load_4d(dst + c * BT_PANEL_BYTES, m, full, c * 64, hk, b_first * n, 0);
    } else {
      mbar_expect_tx(full, TILE_BYTES);
      const CUtensorMap* m = e.seg == BT_PREFIX ? (is_v ? &L_.tm_pv : &L_.tm_pk) : (is_v ? &L_.tm_sv : &L_.tm_sk);
#pragma unroll
      for (int c = 0; c < Cfg::PANELS; ++c)
        tma_load_4d(dst + c * BT_PANEL_BYTES, m, full, c * 64, e.tile * BT_BN, hk, e.seg == BT_PREFIX ? 0 : b_first + e.seg);
    }
  };
  // K and V share one ring: loaded in the order of their use, K_0 K_1 V_0 K_2 V_1 .. K_T-1 V_T-2 V_T-1, each
  // into the slot of the load SLOTS before it.  (With a ring of three for either, a V tile arrived with its K tile, held
  // its slot for the whole softmax of that tile, and the next V was asked for late.  8 layers x 8 kv heads, prefix 2048,
  // 16 branches x 20 rows 94.1 -> 90.4 us; head_dim 64, with twice as many slots, 16 branches x 20 rows, prefix 1500
  // 16.0 -> 15.4 us.)
  using Ring = TileRing<SLOTS>;
  // The list starts with `lead` prefix tiles (see tile_at): their loads, but for the last one's V tile, have places in that
  // order that do not depend on the lengths.
  const int lead = min(npre, Cfg::LEAD), pre_issued = min(max(2 * lead - 1, 0), SLOTS);
  if (warp == BT_LOADER_WARP) {
    if (elect_one()) {
      // Q: box_tokens tokens from tok0 on, heads hk G .. hk G + G - 1, one box per 64-column panel; the box lands as
      // rows (token, head) = stacked-row order.  Rows of the Q buffer beyond the box are never written: they belong
      // to no row of this tile and whatever the tensor cores make of them is never used.
      mbar_expect_tx(bar(BT_Q_FULL), static_cast<uint32_t>(p.box_tokens) * G * (D * 2u));
#pragma unroll
      for (int c = 0; c < Cfg::PANELS; ++c)
        tma_load_4d(sQ + c * BT_PANEL_BYTES, &L_.tm_q, bar(BT_Q_FULL), c * 64, hk * G, tok0, 0);
      for (int i = 0; i < pre_issued; ++i) {
        const bool is_v = i > 0 && (i & 1) == 0;
        load_kv(is_v, i, BtTile{BT_PREFIX, p0 + (is_v ? i / 2 - 1 : (i + 1) / 2), 0});
      }
    }
  } else if (warp == 0) {
    // ---- lengths and tile counts of the row tile's branches
    int L = 0;
    if (lane < nb) {
      L = __ldg(p.d_suffix_len + b_first + lane);
      L = L < n ? n : (L > p.max_suffix_len ? p.max_suffix_len : L);
    }
    // with the fused write the step's block is an entry of its own, the first of the suffix part
    int cum = ((fused ? max(L - n, 0) : L) + BT_BN - 1) / BT_BN;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, cum, o);
      if (lane >= o) cum += t;
    }
    len_s[lane] = L;
    cum_s[lane] = cum;
    if (lane == 31) {  // this CTA's share of the unit's suffix part
      cum += fused ? 1 : 0;
      const int s0 = static_cast<int>((static_cast<int64_t>(cum) * crank) >> log2c);
      suffix_share[0] = s0;
      suffix_share[1] = static_cast<int>((static_cast<int64_t>(cum) * (crank + 1)) >> log2c) - s0;
    }
  }
  __syncthreads();
  const int s0 = suffix_share[0], nsuf = suffix_share[1];
  const int Tall = npre + nsuf;
  // branch `lane` of the row tile: its rows in the suffix tiles, the number of its first tile, one past its last
  const int lane_rows = fused ? len_s[lane] - n : len_s[lane], lane_end = cum_s[lane];
  const int lane_first = lane > 0 ? cum_s[lane - 1] : 0;
  // Entry `s` of this CTA's list, for a whole warp.  `lead` prefix tiles, whose loads need no lengths, then two tiles of the
  // suffix part and two of the prefix in turn (one per stream) while both last, then the rest.  The suffix part is the step's
  // block (fused write only), then the suffix tiles of the row tile's branches.
  // The lookup is on the issuers' path, where an access to shared memory takes 100 to 200 cycles: it works on what the lanes
  // hold.  The prefix comes from L2 (other row tiles read it too), the suffix from HBM: one after the other, HBM was idle
  // first and then what every tile waited for.  6 layers x 8 kv heads, 16 branches x 20 rows of 69 .. 517, prefix 2048: lookup in
  // shared memory and one after the other 53.4 us, lookup in the lanes 50.5, and mixed 46.
  const int mixed = min(npre - lead, nsuf) >> 1;
  auto tile_at = [&](int s) {
    bool prefix = s < lead;
    int g = s;  // its number among the entries of its kind
    if (!prefix) {
      const int q = s - lead, left = npre - lead - 2 * mixed;
      if (q < 4 * mixed) {
        prefix = q & 2;
        g = (q >> 2) * 2 + (q & 1) + (prefix ? lead : 0);
      } else {
        prefix = q - 4 * mixed < left;
        g = q - 2 * mixed + (prefix ? lead : -left);
      }
    }
    if (prefix) return BtTile{BT_PREFIX, p0 + g, min(P - (p0 + g) * BT_BN, BT_BN)};
    g += s0;
    if (fused) {
      if (g == 0) return BtTile{BT_NEW, 0, nb * n};
      --g;
    }
    const int j = __popc(__ballot_sync(0xffffffffu, lane_end <= g));
    const int tile = g - __shfl_sync(0xffffffffu, lane_first, j);
    return BtTile{j, tile, min(__shfl_sync(0xffffffffu, lane_rows, j) - tile * BT_BN, BT_BN)};
  };
  const Ring ring{Tall};
  const int T[2] = {(Tall + 1) >> 1, Tall >> 1};  // stream x takes the sequence numbers 2 i + x

  if (warp == BT_LOADER_WARP) {
    // =============================================================== loader
    reg_dec<BT_REGS_OTHER>();
    const bool leader = elect_one();
    bool ok = true;
    int i = pre_issued;
    for (; i < ring.loads(); ++i) {
      const bool is_v = ring.is_v(i);
      const BtTile e = tile_at(ring.tile(i));
      const int slot = Ring::slot(i);
      if (i >= SLOTS) ok = __all_sync(0xffffffffu, mbar_wait(bar(BT_EMPTY + slot), (i / SLOTS - 1) & 1, abort_flag, p.status, wl));
      if (!ok) break;
      if (leader) load_kv(is_v, slot, e);
    }
    if (leader && *abort_flag) {
      // wait (bounded) until every copy this thread started has landed before shared memory is released
      int dummy = 0;
      volatile int* none = &dummy;
      for (int j = max(0, i - SLOTS); j < i; ++j)
        mbar_wait(bar(BT_FULL + Ring::slot(j)), Ring::parity(j), none, nullptr);
      mbar_wait(bar(BT_Q_FULL), 0, none, nullptr);
    }
    __syncwarp();
  } else if (warp == BT_PATCH_WARP) {
    // =============================================================== patcher
    // Passes every landed V tile on, in list order (a count, which unlike a barrier's parity cannot be mistaken for an
    // older one); before that, where the last 16-key group of a tile is not full, zeros into the rest of the group.
    reg_dec<BT_REGS_OTHER>();
    bool ok = true;
    for (int s = 0; s < Tall && ok; ++s) {
      const BtTile e = tile_at(s);
      const int i = ring.v_load(s), slot = Ring::slot(i), k_before = ring.k_before_v(s);
      ok = k_before < 0 || mbar_wait(bar(BT_K_SEEN + (k_before > 0)), 0, abort_flag, p.status, wl);
      ok = __all_sync(0xffffffffu, ok && mbar_wait(bar(BT_FULL + slot), Ring::parity(i), abort_flag, p.status, wl));
      if (!ok) break;
      if (e.patch()) {
        const uint32_t tile_addr = sKV + slot * TILE_BYTES;
        constexpr int CH = Cfg::CH;
        for (int idx = lane; idx < (16 - (e.valid & 15)) * CH; idx += 32) {
          const int r = e.valid + idx / CH, c = idx % CH;  // 16-byte piece c of row r in the 128-byte-swizzled panels
          asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};\n" ::"r"(tile_addr + (c >> 3) * BT_PANEL_BYTES + r * 128 +
                                                                          (((c & 7) ^ (r & 7)) << 4)),
                       "r"(0u)
                       : "memory");
        }
        fence_proxy_async();  // the tensor cores read the slot through the async proxy
        __syncwarp();
      }
      if (lane == 0) count_publish(v_ready, s + 1);
    }
  } else if (warp == BT_QK_WARP) {
    // =============================================================== issuer of S = Q K^T, tiles in list order
    // (two issuing threads and one S buffer handed back by the softmax as soon as it has read its scores: see
    // prefill_tc.cu)
    reg_dec<BT_REGS_OTHER>();
    const bool leader = elect_one();
    const uint32_t s_col = tmem + BT_S_COL, q_lo = tc_desc_lo(sQ, 16);
    bool ok = true;
    int turn = 0;
    ok = mbar_wait(bar(BT_Q_FULL), 0, abort_flag, p.status, wl);  // (also when the list is empty: the copy must land)
    for (int s = 0; s < Tall; ++s) {
      const int i = Ring::k_load(s), slot = Ring::slot(i);
      const BtTile e = tile_at(s);
      const uint32_t idesc_qk = tc_idesc_bf16(BT_BM, e.groups() * 16, false, false);
      ok = __all_sync(0xffffffffu, ok && mbar_wait(bar(BT_FULL + slot), Ring::parity(i), abort_flag, p.status, wl));
      if (leader && ok && ring.v_after_k(s)) mbar_arrive(bar(BT_K_SEEN + (s > 0)));
      if (s > 0) named_sync(NB_S_FREE + ((s - 1) & 1), 160);
      if (leader && ok) {
        flag_write(qk_turn, ++turn);  // odd: a batch of scores is being issued
        tc_fence_after();
        const uint32_t k_lo = tc_desc_lo(sKV + slot * TILE_BYTES, 16);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          const uint32_t off = ((ks >> 2) * BT_PANEL_BYTES + (ks & 3) * 32) >> 4;
          tc_mma_ss_lo(s_col, q_lo + off, k_lo + off, idesc_qk, ks > 0);
        }
        tc_commit(bar(BT_S_FULL + (s & 1)));
        flag_write(qk_turn, ++turn);
        tc_commit(bar(BT_EMPTY + slot));
      }
      __syncwarp();
    }
    if (Tall > 0) named_sync(NB_S_FREE + ((Tall - 1) & 1), 160);
    if (leader && !ok) {  // make sure no MMA of this thread is still running before TMEM and smem go away
      int dummy = 0;
      tc_commit(bar(BT_DRAIN));
      mbar_wait(bar(BT_DRAIN), 0, &dummy, nullptr);
    }
    __syncwarp();
  } else if (warp == BT_PV_WARP) {
    // =============================================================== issuer of O += P V, tiles in list order
    reg_dec<BT_REGS_OTHER>();
    constexpr uint32_t idesc_pv = tc_idesc_bf16(BT_BM, D, false, true);
    const bool leader = elect_one();
    bool ok = true;
    for (int s = 0; s < Tall; ++s) {
      const int slot = Ring::slot(ring.v_load(s)), x = s & 1;
      const uint32_t v_lo = tc_desc_lo(sKV + slot * TILE_BYTES, BT_PANEL_BYTES);
      const uint32_t o_col = tmem + BT_O_COL0 + x * 128, p_col = tmem + BT_P_COL0 + x * 64;
      const BtTile e = tile_at(s);
      const int groups = e.groups();
      ok = __all_sync(0xffffffffu, ok && count_spin_wait(v_ready, s + 1, abort_flag, p.status, wl) >= 0);
      named_sync(NB_P_EARLY + x, 160);  // the first 96 keys while the softmax finishes the last 32
      if (leader && ok) {
        for (int it = 0; it < 4096 && (flag_read(qk_turn) & 1); ++it) {}  // stand back for the scores
        tc_fence_after();
#pragma unroll
        for (int ks = 0; ks < 6; ++ks)
          if (ks < groups) tc_mma_ts_lo(o_col, p_col + ks * 8, v_lo + ks * (2048 >> 4), idesc_pv, (s > 1 || ks > 0));
      }
      __syncwarp();
      named_sync(NB_P_FULL + x, 160);
      if (leader && ok) {
        tc_fence_after();
#pragma unroll
        for (int ks = 6; ks < 8; ++ks)
          if (ks < groups) tc_mma_ts_lo(o_col, p_col + ks * 8, v_lo + ks * (2048 >> 4), idesc_pv, 1);
        tc_commit(bar(BT_O_READY + x));
        tc_commit(bar(BT_EMPTY + slot));
      }
      __syncwarp();
    }
    if (leader && !ok) {
      int dummy = 0;
      tc_commit(bar(BT_DRAIN + 1));
      mbar_wait(bar(BT_DRAIN + 1), 0, &dummy, nullptr);
    }
    __syncwarp();
  } else {
    // =============================================================== softmax warpgroups (streams)
    reg_inc<BT_REGS_SOFTMAX>();
    const int x = warp >> 2;
    const int row_in_tile = (warp & 3) * 32 + lane;
    const bool row_valid = row_in_tile < rows_here;
    int ri;
    const int rb = p.by_q_len.divmod(tok0 + p.by_group.div(row_in_tile), ri);  // branch and draft row of this row
    const int rj = row_valid ? rb - b_first : -1;    // the row's branch as an index into the tile's branches
    const int own_rows = row_valid ? len_s[rj] - n : 0;  // rows of its branch before the step's block
    // draft rows of the block this row may see, as bits: its ancestors and itself (a chain: rows 0..i)
    const uint32_t tm = !row_valid ? 0u
                        : (p.tree_mask ? __ldg(p.tree_mask + static_cast<int64_t>(rb) * n + ri) : (2u << ri) - 1u) &
                              ((1u << n) - 1u);
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t tS = tmem + lane_base + BT_S_COL, tP = tmem + lane_base + BT_P_COL0 + x * 64;
    const uint32_t tO = tmem + lane_base + BT_O_COL0 + x * 128;
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
      // ---- which columns of the tile this row sees (a row beyond the tile's rows sees nothing); worked out while
      // the tensor cores still compute the tile's scores
      const BtTile e = tile_at(2 * j + x);
      const int key0 = e.tile * BT_BN;
      ColumnBits allow = {0u, 0u, 0u, 0u};
      // a whole prefix tile is seen by every row there is
      bool row_sees = true, warp_sees = (warp & 3) * 32 < rows_here, masked = false;
      if (e.seg != BT_PREFIX || e.valid < BT_BN) {
        // by 32-column words: the first `cnt` columns, and the block's rows by the mask from column `col` on (which may
        // lie outside the tile)
        auto word = [&](int w, int cnt, int col) {
          const int k = cnt - 32 * w, c0 = col - 32 * w;
          const uint32_t before = k >= 32 ? 0xffffffffu : (k <= 0 ? 0u : (1u << k) - 1u);
          const uint32_t block = c0 >= 32 ? 0u : (c0 >= 0 ? tm << c0 : (c0 > -32 ? tm >> (-c0) : 0u));
          return before | block;
        };
        // shared prefix: up to its end; the step's block: the rows of this row's branch; the row's own branch: the rows
        // before the block, then (without the fused write) the block; another branch's suffix: nothing
        constexpr int NONE = 0x100000;
        int cnt = 0, col = NONE;
        if (e.seg == BT_PREFIX) {
          cnt = e.valid;
        } else if (e.seg == BT_NEW) {
          col = rj * n;
        } else if (e.seg == rj) {
          cnt = own_rows - key0;
          col = fused ? NONE : cnt;
        }
        if (!row_valid) cnt = 0, col = NONE;
        allow = ColumnBits{word(0, cnt, col), word(1, cnt, col), word(2, cnt, col), word(3, cnt, col)};
        row_sees = (allow.w0 | allow.w1 | allow.w2 | allow.w3) != 0u;
        warp_sees = __any_sync(0xffffffffu, row_sees);
        // columns are only masked for the rows that see some of the tile but not all of it
        masked = !__all_sync(0xffffffffu, !row_sees || (allow.w0 & allow.w1 & allow.w2 & allow.w3) == 0xffffffffu);
      }
      // (ok is the same in all lanes of a warp: the barriers and the tcgen05 operations are warp-collective)
      ok = __all_sync(0xffffffffu, ok && mbar_spin_wait(bar(BT_S_FULL + x), j & 1, abort_flag, p.status, wl));
      tc_fence_after();
      auto test_o = [&] { return mbar_test_wait(bar(BT_O_READY + x), (j - 1) & 1); };
      auto wait_o = [&] { ok = ok && mbar_wait(bar(BT_O_READY + x), (j - 1) & 1, abort_flag, p.status, wl); };
      auto release_early = [&] {
        ok = __all_sync(0xffffffffu, ok);
        signal(NB_P_EARLY);
      };
      if (warp_sees) {
        softmax_tile_row<true, D>(tS, tP, tO, j, (e.groups() + 1) >> 1, masked, allow, row_sees, c, m_ref, l, test_o, wait_o,
                                  [&] { signal(NB_S_FREE); }, release_early);
      } else {  // no row of this warp sees the tile: P = 0, nothing else changes
        signal(NB_S_FREE);
        if (j > 0 && !test_o()) wait_o();  // the previous P has been read
        tc_fence_after();
        uint32_t z[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) z[i] = 0u;
#pragma unroll 1
        for (int q4 = 0; q4 < 4; ++q4) tmem_st16(tP + q4 * 16, z);
        tc_wait_st();
        release_early();
      }
      signal(NB_P_FULL);
    }
    // With the fused write the block's rows go into the cache once per (branch, kv head): by the unit whose row tile
    // starts the branch, its branches dealt to the CTAs, all threads and all loads at once (one warp going through
    // the branches took 10 us).  Nobody reads those rows of the cache in this launch.
    if (ok && fused && (p.slices_per_branch == 1 || rt % p.slices_per_branch == 0)) {
      constexpr int CH = Cfg::CH;
      const int pieces = nb > crank ? ((nb - crank + (1 << log2c) - 1) >> log2c) * n * CH : 0;
#pragma unroll 2
      for (int idx = threadIdx.x; idx < pieces; idx += 256) {
        const int c16 = idx % CH, t = idx / CH, jb = crank + (t / n << log2c), r = t % n, b = b_first + jb;
        const int64_t src = ((static_cast<int64_t>(b) * n + r) * p.kv_heads + hk) * D + c16 * 8;
        const int64_t dst = b * p.sb + hk * p.sh + static_cast<int64_t>(len_s[jb] - n + r) * p.sr + c16 * 8;
        const uint4 kk = __ldg(reinterpret_cast<const uint4*>(L_.k_new + src));
        const uint4 vv = __ldg(reinterpret_cast<const uint4*>(L_.v_new + src));
        *reinterpret_cast<uint4*>(L_.k_cache + dst) = kk;
        *reinterpret_cast<uint4*>(L_.v_cache + dst) = vv;
      }
    }
    pdl_launch_dependents();  // the next kernel of the stream may start its own set-up now

    // ---- the two streams' (m, l) of a row cross through shared memory: the K slot of the stream's last tile,
    // free once its accumulator is complete and not filled again; a stream without tiles takes slot 2 + x, never filled then
    auto ml_of = [&](int y) {
      const int slot = T[y] > 0 ? Ring::slot(Ring::k_load(2 * (T[y] - 1) + y)) : 2 + y;
      return reinterpret_cast<float2*>(smem_gen + Cfg::SMEM_KV + slot * TILE_BYTES);
    };
    if (Tx > 0) ok = mbar_wait(bar(BT_O_READY + x), (Tx - 1) & 1, abort_flag, p.status, wl) && ok;
    ml_of(x)[row_in_tile] = make_float2(m_ref, l);
    tc_fence_before();
    named_sync(NB_MERGE, 256);
    tc_fence_after();
    const float2 oth = ml_of(1 - x)[row_in_tile];
    // a stream whose tiles were all hidden from this row has l = 0 and takes no part
    const float m_own = l > 0.f ? m_ref : -INFINITY, m_oth = oth.y > 0.f ? oth.x : -INFINITY;
    const float fin_m = fmaxf(m_own, m_oth);
    float w_own = l > 0.f ? fast_exp2(m_own - fin_m) : 0.f, w_oth = oth.y > 0.f ? fast_exp2(m_oth - fin_m) : 0.f;
    const float fin_l = l * w_own + oth.y * w_oth;
    // columns [D/2 x, D/2 x + D/2) of both streams combined, handed to put(column, value) by fours
    const bool has_own = Tx > 0, has_oth = T[1 - x] > 0;  // a stream without tiles never wrote its accumulator
    auto combine = [&](auto&& put) {
      const uint32_t tOwn = tmem + lane_base + BT_O_COL0 + x * 128 + x * (D / 2);
      const uint32_t tOth = tmem + lane_base + BT_O_COL0 + (1 - x) * 128 + x * (D / 2);
#pragma unroll
      for (int q2 = 0; q2 < D / 64; ++q2) {
        uint32_t o[32], o2[32];
        if (has_own) tmem_ld32(tOwn + q2 * 32, o);
        if (has_oth) tmem_ld32(tOth + q2 * 32, o2);
        tc_wait_ld();
#pragma unroll
        for (int cc = 0; cc < 8; ++cc) {
          float v[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            v[i] = has_own ? __uint_as_float(o[4 * cc + i]) * w_own : 0.f;
            if (has_oth) v[i] = fmaf(__uint_as_float(o2[4 * cc + i]), w_oth, v[i]);
          }
          put(x * (D / 2) + q2 * 32 + cc * 4, make_float4(v[0], v[1], v[2], v[3]));
        }
      }
    };
    const bool warp_has_row = (warp & 3) * 32 < rows_here;  // warp-uniform (the TMEM loads are warp-collective)
    // token and head of a row of the tile
    auto place = [&](int row, int& hq) {
      const int tok = tok0 + p.by_group.divmod(row, hq);
      hq += hk * G;
      return tok;
    };
    auto store_lse = [&](int tok, int hq, float value) {
      int i;
      const int b = p.by_q_len.divmod(tok, i);
      L_.lse[(static_cast<int64_t>(b) * p.q_heads + hq) * n + i] = value * 0.69314718055994530942f;
    };
    if (shared) {
      // ---- this CTA's partial of the row -> scratch, unnormalised, relative to the row's maximum over this CTA's tiles, as
      // [column chunk][row] float4 so that a warp writes 512 contiguous bytes
      float4* gpart = reinterpret_cast<float4*>(p.part + (static_cast<size_t>(share) * C + crank) * Cfg::PART_FLOATS);
      float2* gml = reinterpret_cast<float2*>(p.ml + (static_cast<size_t>(share) * C + crank) * BT_ML_FLOATS);
      if (warp_has_row) {
        combine([&](int col, float4 v) {
          if (row_valid) gpart[col / 4 * BT_BM + row_in_tile] = v;
        });
        if (row_valid && x == 0) gml[row_in_tile] = make_float2(fin_l > 0.f ? fin_m : -INFINITY, fin_l);
      }
      __threadfence();  // visible to the cluster before its barrier is passed
      tc_fence_before();
      cluster_sync_all();
      // ---- behind the cluster barrier every CTA's partial is in the scratch (L2).  This CTA finishes the rows
      // [128 crank / C, 128 (crank + 1) / C): a thread takes every 2C-th column chunk of one row, all its loads in flight
      // at once; the sums run in CTA order, so the result never depends on timing.
      const bool clean = *abort_flag == 0 && *reinterpret_cast<volatile int*>(p.status) == 0;  // nobody gave up on a wait
      constexpr int PER = BT_BM / C, MINE = D / 4 / (2 * C);
      const int row = PER * crank + known_here(threadIdx.x) % PER, sub = known_here(threadIdx.x) / PER;
      if (row < rows_here) {
        const float2* uml = reinterpret_cast<const float2*>(p.ml + static_cast<size_t>(share) * C * BT_ML_FLOATS);
        const float4* upart = reinterpret_cast<const float4*>(p.part + static_cast<size_t>(share) * C * Cfg::PART_FLOATS);
        float2 ml[C];
        float4 v[MINE][C];
#pragma unroll
        for (int cr = 0; cr < C; ++cr) ml[cr] = __ldcg(uml + cr * BT_BM + row);
#pragma unroll
        for (int u = 0; u < MINE; ++u)
#pragma unroll
          for (int cr = 0; cr < C; ++cr)
            v[u][cr] = __ldcg(upart + cr * (Cfg::PART_FLOATS / 4) + (u * 2 * C + sub) * BT_BM + row);
        float M = -INFINITY, w[C], lall = 0.f;
#pragma unroll
        for (int cr = 0; cr < C; ++cr) M = fmaxf(M, ml[cr].x);  // (-inf: all of that CTA's tiles were hidden from the row)
#pragma unroll
        for (int cr = 0; cr < C; ++cr) {
          w[cr] = fast_exp2(ml[cr].x - M);
          lall = fmaf(w[cr], ml[cr].y, lall);
        }
        const float inv = 1.f / lall;
        int hq;
        const int tok = place(row, hq);
        float* dst = L_.out + (static_cast<int64_t>(tok) * p.q_heads + hq) * D;
#pragma unroll
        for (int u = 0; u < MINE; ++u) {
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int cr = 0; cr < C; ++cr) {
            acc.x = fmaf(w[cr], v[u][cr].x, acc.x);
            acc.y = fmaf(w[cr], v[u][cr].y, acc.y);
            acc.z = fmaf(w[cr], v[u][cr].z, acc.z);
            acc.w = fmaf(w[cr], v[u][cr].w, acc.w);
          }
          if (clean)
            *reinterpret_cast<float4*>(dst + (u * 2 * C + sub) * 4) = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        }
        if (clean && L_.lse && sub == 0) store_lse(tok, hq, M + log2f(lall));
      }
    } else {
      // ---- one CTA per unit: the rows are staged in shared memory (every MMA and copy of the CTA is complete behind
      // the barrier above, so the K/V slots are free once the (m, l) have been read) and written out as whole rows
      float* stage = reinterpret_cast<float*>(smem_gen + Cfg::SMEM_KV);  // [row][Cfg::RECV_STRIDE]
      named_sync(NB_MERGE, 256);
      if (warp_has_row) {
        const float inv = 1.f / fin_l;
        w_own *= inv;
        w_oth *= inv;
        combine([&](int col, float4 v) {
          *reinterpret_cast<float4*>(stage + row_in_tile * Cfg::RECV_STRIDE + col) = v;
        });
        if (x == 0) *reinterpret_cast<float2*>(stage + row_in_tile * Cfg::RECV_STRIDE + D) = make_float2(fin_m, fin_l);
      }
      named_sync(NB_MERGE, 256);
      const bool clean = *abort_flag == 0 && *reinterpret_cast<volatile int*>(p.status) == 0;  // nobody gave up on a wait
#pragma unroll 4
      for (int idx = threadIdx.x; idx < rows_here * (D / 4) && clean; idx += 256) {
        const int row = idx / (D / 4), chunk = idx % (D / 4);
        int hq;
        const int tok = place(row, hq);
        *reinterpret_cast<float4*>(L_.out + (static_cast<int64_t>(tok) * p.q_heads + hq) * D + chunk * 4) =
            *reinterpret_cast<const float4*>(stage + row * Cfg::RECV_STRIDE + chunk * 4);
        if (chunk == 0 && L_.lse) {
          const float2 ml = *reinterpret_cast<const float2*>(stage + row * Cfg::RECV_STRIDE + D);
          store_lse(tok, hq, ml.x + log2f(ml.y));
        }
      }
    }
  }
  // (every thread of every CTA passes the cluster's barrier, whatever happened above; the output above is part of the
  // softmax branch because code behind the branches would have to make do with the other roles' registers)
  if (shared && warp >= 8) cluster_sync_all();

  // ---- tear-down
  tc_fence_before();
  __syncthreads();
  if (warp == BT_QK_WARP) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ---------------------------------------------------------------- host side

struct BtPlan {
  int row_tiles, branches_per_tile, slices_per_branch, box_tokens, units;
  int cluster, whole_units;  // of the units of all layers, the first whole_units have a CTA each, the others a cluster
  bool ok;
  int64_t estimate_ns;
};

template <int D, int NL, int C>
static cudaError_t bt_set_attributes() {
  static PerDeviceOnce attr_done;
  if (attr_done.done()) return cudaSuccess;
  cudaError_t e =
      cudaFuncSetAttribute(branch_tc_kernel<D, NL, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, BtCfg<D>::SMEM_BYTES);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(branch_tc_kernel<D, NL, C>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess) attr_done.set();
  return e;
}

// How many clusters of C CTAs of the kernel can be resident at once on the current device (0 if the query fails).
template <int D, int NL, int C>
static int bt_resident_clusters() {
  static ResidentClusters clusters;
  if (bt_set_attributes<D, NL, C>() != cudaSuccess) return 0;
  return clusters.get(reinterpret_cast<const void*>(branch_tc_kernel<D, NL, C>), C, BT_THREADS, BtCfg<D>::SMEM_BYTES);
}

// The tiling of one problem and the CTAs per unit, for `layers` problems in one launch: the form with the shortest
// estimated time.  A CTA takes 1.15 us per tile of 128 keys (0.85 with head_dim 64; a branch's suffix counted at 0.6 of its
// longest possible walk) and a fixed time, larger when a cluster has to exchange partials; more, smaller row tiles walk
// the prefix more often but may fill the machine better.  Where the units fill the machine more than once, the full waves
// have a CTA per unit and the rest a cluster each, if these fit in one wave.  Measured (us, tiles per CTA in brackets):
// 8 kv heads, 128 rows, prefix 1000 11.5 (3), prefix 4000 13.6 (6); 6 layers x 8 kv heads x 3 row tiles, one wave 46 (34); 8
// layers, two waves of CTAs 75 (2 x 28), one and a rest of 48 units in clusters of two 70 (34 + 17); the same with short
// suffixes, prefix 3000 71 and 64.
template <int D, int NL>
static BtPlan bt_plan(int prefix_len, int max_suffix_len, int n_branches, int q_heads, int kv_heads, int q_len,
                      int sm_count, int layers) {
  constexpr int64_t TILE_NS = D == 128 ? 1150 : 850, ALONE_NS = D == 128 ? 6800 : 6000, CLUSTER_NS = D == 128 ? 8100 : 7600;
  BtPlan pl = {0, 0, 1, 0, 0, 1, 0, false, 0};
  const int G = q_heads / kv_heads, nG = q_len * G;
  const int64_t Tp = (static_cast<int64_t>(prefix_len) + BT_BN - 1) / BT_BN;
  const int64_t ts_max = (max_suffix_len + BT_BN - 1) / BT_BN;
  const int64_t ts_est = std::max<int64_t>(1, (ts_max * 6 + 9) / 10);
  int64_t best = -1;
  auto consider = [&](int64_t row_tiles, int per_tile, int slices, int box_tokens) {
    const int64_t units = row_tiles * kv_heads, all = units * layers;
    if (all > (1 << 30)) return;
    const int64_t walk = Tp + per_tile * ts_est;
    for (int c = 1; c <= 8; c *= 2) {
      if (c > 1 && 2 * c > Tp + ts_max + 1) break;  // no more CTAs than pairs of tiles a unit certainly has
      const int64_t at_once = c == 1   ? sm_count
                              : c == 2 ? bt_resident_clusters<D, NL, 2>()
                              : c == 4 ? bt_resident_clusters<D, NL, 4>()
                                       : bt_resident_clusters<D, NL, 8>();
      if (at_once == 0) continue;
      const int64_t full_waves = all / (at_once * c), whole = c == 1 ? all : full_waves * at_once * c;
      if (c > 1 && (whole == all || all - whole > at_once)) continue;  // (clusters: one wave, after those of whole units)
      const int64_t est = c == 1 ? (all + at_once - 1) / at_once * (walk * TILE_NS + ALONE_NS)
                                 : full_waves * (walk * TILE_NS + ALONE_NS) + (walk + c - 1) / c * TILE_NS + CLUSTER_NS;
      if (best < 0 || est < best) {
        best = est;
        pl = BtPlan{static_cast<int>(row_tiles), per_tile, slices, box_tokens, static_cast<int>(units), c, static_cast<int>(whole), true, est};
      }
    }
  };
  if (nG <= BT_BM) {  // whole branches per row tile, the same number in every tile
    const int per_tile_max = std::min(BT_MAX_BRANCHES, BT_BM / nG);
    const int tiles_min = (n_branches + per_tile_max - 1) / per_tile_max;
    for (int tiles = tiles_min; tiles <= std::min(n_branches, 2 * tiles_min); ++tiles) {
      const int per_tile = (n_branches + tiles - 1) / tiles;
      if (per_tile > per_tile_max || static_cast<int64_t>(tiles - 1) * per_tile >= n_branches) continue;
      consider(tiles, per_tile, 1, per_tile * q_len);
    }
  } else if (BT_BM % G == 0) {  // a branch has more than 128 rows: 128-row slices, which must start on a token
    const int slices = (nG + BT_BM - 1) / BT_BM;
    consider(static_cast<int64_t>(n_branches) * slices, 1, slices, BT_BM / G);
  }
  return pl;
}

template <int D>
static size_t bt_scratch_bytes(const BtPlan& pl, int layers) {
  if (pl.cluster <= 1) return 0;
  return SCRATCH_COUNTER_BYTES + static_cast<size_t>(layers * pl.units - pl.whole_units) * pl.cluster *
                                     (BtCfg<D>::PART_FLOATS + BT_ML_FLOATS) * sizeof(float);
}

bool branch_tc_supported(const CacheView& prefix, const CacheView& suffix, int n_branches, int q_heads, int q_len,
                         float scale) {
  if (!(scale > 0.f) || !(scale < INFINITY) || !encode_fn() || !replace_fn()) return false;
  // (a stride that no tensor map carries, as of the batch of a cache for one branch, which nothing else looks at: the other
  // kernels take the call)
  if (!stride_encodable(suffix.sr) || !stride_encodable(suffix.sh) || !stride_encodable(suffix.sb) ||
      !stride_encodable(prefix.sr) || !stride_encodable(prefix.sh))
    return false;
  const int G = q_heads / suffix.kv_heads;
  const int64_t nG = static_cast<int64_t>(q_len) * G;
  if (nG > BT_BM && BT_BM % G != 0) return false;
  const int64_t tiles = nG > BT_BM ? static_cast<int64_t>(n_branches) * ((nG + BT_BM - 1) / BT_BM) : n_branches;
  return tiles * suffix.kv_heads <= (1 << 30);
}

int64_t branch_tc_estimate_ns(int n_branches, int q_heads, int kv_heads, int q_len, int head_dim, int prefix_len,
                              int max_suffix_len, int layers, int sm_count) {
  const bool batched = layers >= BT_MIN_BATCHED_LAYERS;
  auto estimate = [&](auto plan) {
    const BtPlan pl = plan(prefix_len, max_suffix_len, n_branches, q_heads, kv_heads, q_len, sm_count, batched ? layers : 1);
    return pl.ok ? pl.estimate_ns * (batched ? 1 : layers) : INT64_MAX;
  };
  if (head_dim == 128) return batched ? estimate(bt_plan<128, kBranchMaxLayersPerLaunch>) : estimate(bt_plan<128, 1>);
  return batched ? estimate(bt_plan<64, kBranchMaxLayersPerLaunch>) : estimate(bt_plan<64, 1>);
}

template <int D, int NL>
static cudaError_t launch_bt(const BranchLayerTensors* t, int layers, const CacheView& prefix, int prefix_len,
                             const CacheView& suffix, const int32_t* d_suffix_len, const uint32_t* d_tree_mask,
                             int max_suffix_len, int n_branches, int q_heads, int q_len, float scale, int* status,
                             long long wait_limit, void* workspace, size_t workspace_bytes, cudaStream_t st,
                             LaunchInfo& li) {
  BtPlan pl = bt_plan<D, NL>(prefix_len, max_suffix_len, n_branches, q_heads, suffix.kv_heads, q_len, li.sm_count, layers);
  if (!pl.ok) return cudaErrorInvalidValue;
  // several CTAs per unit exchange partials through the scratch; without enough of it a unit is walked by one CTA
  const int all_units = layers * pl.units;
  if (pl.cluster > 1 && (!workspace || bt_scratch_bytes<D>(pl, layers) > workspace_bytes)) pl.cluster = 1, pl.whole_units = all_units;
  const int G = q_heads / suffix.kv_heads;
  const uint64_t tokens = static_cast<uint64_t>(n_branches) * q_len;
  BtLayers<NL> L;
  {  // layer 0's maps; the other layers' differ in their addresses only, and so do V's from K's.  (Encoding all seven maps of
     // a layer took the host 100 us for a call of 32 layers, more than small layers take on the GPU; replaced addresses 90.)
    BtLayer& l = L.l[0];
    {  // q: [tokens][q_heads][D]; a box is [box_tokens tokens][G heads][64 columns]: the tile's stacked rows in order
      const uint64_t d[4] = {D, static_cast<uint64_t>(q_heads), tokens, 1};
      const uint64_t s[3] = {D * 2ull, static_cast<uint64_t>(q_heads) * D * 2ull, 0};
      const uint32_t bx[4] = {64, static_cast<uint32_t>(G), static_cast<uint32_t>(pl.box_tokens), 1};
      if (!make_map_bf16(&l.tm_q, t[0].q, d, s, bx)) return cudaErrorInvalidValue;
    }
    {  // suffix caches: rows at or beyond max_suffix_len read as zero
      const uint64_t d[4] = {D, static_cast<uint64_t>(max_suffix_len), static_cast<uint64_t>(suffix.kv_heads),
                             static_cast<uint64_t>(suffix.batch)};
      const uint64_t s[3] = {static_cast<uint64_t>(suffix.sr) * 2, static_cast<uint64_t>(suffix.sh) * 2,
                             static_cast<uint64_t>(suffix.sb) * 2};
      const uint32_t bx[4] = {64, BT_BN, 1, 1};
      if (!make_map_bf16(&l.tm_sk, t[0].sk, d, s, bx)) return cudaErrorInvalidValue;
    }
    if (prefix_len > 0) {  // rows at or beyond prefix_len read as zero
      const uint64_t d[4] = {D, static_cast<uint64_t>(prefix_len), static_cast<uint64_t>(prefix.kv_heads), 1};
      const uint64_t s[3] = {static_cast<uint64_t>(prefix.sr) * 2, static_cast<uint64_t>(prefix.sh) * 2, 0};
      const uint32_t bx[4] = {64, BT_BN, 1, 1};
      if (!make_map_bf16(&l.tm_pk, t[0].pk, d, s, bx)) return cudaErrorInvalidValue;
    }
    if (t[0].k_new) {  // the step's block, [tokens][kv_heads][D]: a box is the tokens of a row tile's branches
      const uint64_t d[4] = {D, static_cast<uint64_t>(suffix.kv_heads), tokens, 1};
      const uint64_t s[3] = {D * 2ull, static_cast<uint64_t>(suffix.kv_heads) * D * 2ull, 0};
      const uint32_t bx[4] = {64, 1, static_cast<uint32_t>(pl.branches_per_tile * q_len), 1};
      if (!make_map_bf16(&l.tm_nk, t[0].k_new, d, s, bx)) return cudaErrorInvalidValue;
    }
  }
  for (int i = 0; i < layers; ++i) {
    BtLayer& l = L.l[i];
    const BtLayer& l0 = L.l[0];
    if (i > 0 && (!make_map_like(&l.tm_q, l0.tm_q, t[i].q) || !make_map_like(&l.tm_sk, l0.tm_sk, t[i].sk)))
      return cudaErrorInvalidValue;
    if (!make_map_like(&l.tm_sv, l0.tm_sk, t[i].sv)) return cudaErrorInvalidValue;
    if (prefix_len > 0) {
      if (i > 0 && !make_map_like(&l.tm_pk, l0.tm_pk, t[i].pk)) return cudaErrorInvalidValue;
      if (!make_map_like(&l.tm_pv, l0.tm_pk, t[i].pv)) return cudaErrorInvalidValue;
    } else {
      l.tm_pk = l.tm_sk;  // never dereferenced without a prefix
      l.tm_pv = l.tm_sv;
    }
    if (t[i].k_new) {
      if (i > 0 && !make_map_like(&l.tm_nk, l0.tm_nk, t[i].k_new)) return cudaErrorInvalidValue;
      if (!make_map_like(&l.tm_nv, l0.tm_nk, t[i].v_new)) return cudaErrorInvalidValue;
    } else {
      l.tm_nk = l.tm_sk;  // never dereferenced without a fused write
      l.tm_nv = l.tm_sv;
    }
    l.k_new = t[i].k_new;
    l.v_new = t[i].v_new;
    l.k_cache = const_cast<bf16*>(t[i].sk);
    l.v_cache = const_cast<bf16*>(t[i].sv);
    l.out = t[i].out;
    l.lse = t[i].lse;
  }
  BtParams p;
  p.n_branches = n_branches;
  p.q_len = q_len;
  p.q_heads = q_heads;
  p.group = G;
  p.kv_heads = suffix.kv_heads;
  p.prefix_len = prefix_len;
  p.max_suffix_len = max_suffix_len;
  p.branches_per_tile = pl.branches_per_tile;
  p.slices_per_branch = pl.slices_per_branch;
  p.box_tokens = pl.box_tokens;
  p.box_keys = pl.branches_per_tile * q_len;
  p.by_group = FastDiv(G);
  p.by_q_len = FastDiv(q_len);
  p.by_row_tiles = FastDiv(pl.row_tiles);
  p.by_layer_units = FastDiv(pl.units);
  p.whole_units = pl.whole_units;
  p.scale_log2 = scale * 1.4426950408889634f;
  p.wait_limit = wait_limit;
  p.d_suffix_len = d_suffix_len;
  p.tree_mask = d_tree_mask;
  p.sb = suffix.sb;
  p.sh = suffix.sh;
  p.sr = suffix.sr;
  p.status = status;
  const int shares = (all_units - pl.whole_units) * pl.cluster;  // CTAs that share a unit
  p.part = shares > 0 ? reinterpret_cast<float*>(static_cast<unsigned char*>(workspace) + SCRATCH_COUNTER_BYTES) : nullptr;
  p.ml = shares > 0 ? p.part + static_cast<size_t>(shares) * BtCfg<D>::PART_FLOATS : nullptr;
  auto launch = [&](auto set_attributes, auto kernel) {
    cudaError_t e = set_attributes();
    if (e != cudaSuccess) return e;
    li.launches += 1;
    return launch_pdl_cluster(kernel, dim3(static_cast<unsigned>(pl.whole_units + shares)), dim3(BT_THREADS), BtCfg<D>::SMEM_BYTES,
                              st, static_cast<unsigned>(pl.cluster), L, p);
  };
  switch (pl.cluster) {
    case 8: return launch(bt_set_attributes<D, NL, 8>, branch_tc_kernel<D, NL, 8>);
    case 4: return launch(bt_set_attributes<D, NL, 4>, branch_tc_kernel<D, NL, 4>);
    case 2: return launch(bt_set_attributes<D, NL, 2>, branch_tc_kernel<D, NL, 2>);
  }
  return launch(bt_set_attributes<D, NL, 1>, branch_tc_kernel<D, NL, 1>);
}

cudaError_t launch_branch_tc_layers(const BranchLayerTensors* t, int n_layers, const CacheView& prefix, int prefix_len,
                                    const CacheView& suffix, const int32_t* d_suffix_len, const uint32_t* d_tree_mask,
                                    int max_suffix_len, int n_branches, int q_heads, int q_len, float scale, int* status,
                                    long long wait_limit, void* workspace, size_t workspace_bytes, cudaStream_t st,
                                    LaunchInfo& li) {
  const int at_once = n_layers >= BT_MIN_BATCHED_LAYERS ? kBranchMaxLayersPerLaunch : 1;
  for (int first = 0; first < n_layers; first += at_once) {
    const int n = std::min(at_once, n_layers - first);
    auto launch = [&](auto kernel_launch) {
      return kernel_launch(t + first, n, prefix, prefix_len, suffix, d_suffix_len, d_tree_mask, max_suffix_len, n_branches,
                           q_heads, q_len, scale, status, wait_limit, workspace, workspace_bytes, st, li);
    };
    cudaError_t e;
    if (suffix.head_dim == 128)
      e = n == 1 ? launch(launch_bt<128, 1>) : launch(launch_bt<128, kBranchMaxLayersPerLaunch>);
    else
      e = n == 1 ? launch(launch_bt<64, 1>) : launch(launch_bt<64, kBranchMaxLayersPerLaunch>);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace jup
