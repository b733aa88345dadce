// The order in which the tensor-core branch kernel loads the K and V tiles of a CTA's list into one ring of slots.  Plain
// integers, so that the host can check it for every length of the list.
#pragma once

#ifdef __CUDACC__
#define JUP_HD __host__ __device__ __forceinline__
#else
#define JUP_HD inline
#endif

namespace jup {

// Tiles 0 .. tiles - 1 are loaded in the order of their use, K_0 K_1 V_0 K_2 V_1 .. K_T-1 V_T-2 V_T-1, load i into slot
// i % SLOTS.
template <int SLOTS>
struct TileRing {
  static_assert(SLOTS % 2 == 0, "a slot's loads are all odd or all even");
  int tiles;
  static JUP_HD int slot(int load) { return load % SLOTS; }
  static JUP_HD int parity(int load) { return (load / SLOTS) & 1; }  // of the phase in which the slot's barrier says that it landed
  JUP_HD int loads() const { return 2 * tiles; }
  static JUP_HD int k_load(int s) { return s > 0 ? 2 * s - 1 : 0; }  // the number of a tile's load
  JUP_HD int v_load(int s) const { return s < tiles - 1 ? 2 * s + 2 : 2 * tiles - 1; }
  JUP_HD bool is_v(int load) const { return load == 2 * tiles - 1 || (load > 0 && (load & 1) == 0); }
  JUP_HD int tile(int load) const { return load == 2 * tiles - 1 ? tiles - 1 : is_v(load) ? load / 2 - 1 : (load + 1) / 2; }
  // The thread that waits for the V tiles does not see the K tiles land.  A wait for the parity of a barrier's phase
  // says nothing before the phase in front of it is over, and that one belongs to a K tile where a V tile comes into a K tile's
  // slot: load SLOTS, behind K_0, and the last one.  K tile in front of tile s's V tile in its slot, or -1:
  JUP_HD int k_before_v(int s) const {
    const int before = v_load(s) - SLOTS;
    return before >= 0 && !is_v(before) ? tile(before) : -1;
  }
  // The other way round: does a V tile follow tile s's K tile in its slot?
  JUP_HD bool v_after_k(int s) const {
    const int next = k_load(s) + SLOTS;
    return next < loads() && is_v(next);
  }
};

}  // namespace jup
