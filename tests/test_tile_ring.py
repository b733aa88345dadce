"""The order of the K and V loads in the tensor-core branch kernel's ring (csrc/tile_ring.h), compiled for the host.  A wait for
the parity of a barrier's phase returns at once while the phase in front of it is unfinished, so whoever waits for a load has
to know that the load before it in its slot has landed: by its own earlier wait, or told by the other waiter."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_08242_b200", "csrc")
PROGRAM = r"""
#include <cstdio>
#include "tile_ring.h"
template <int SLOTS> static void print(int tiles) {
  const jup::TileRing<SLOTS> r{tiles};
  for (int s = 0; s < tiles; ++s)
    std::printf("t %d %d %d %d %d %d\n", SLOTS, tiles, r.k_load(s), r.v_load(s), r.k_before_v(s), int(r.v_after_k(s)));
  for (int i = 0; i < r.loads(); ++i)
    std::printf("l %d %d %d %d %d %d\n", SLOTS, tiles, r.slot(i), r.parity(i), int(r.is_v(i)), r.tile(i));
}
int main() {
  for (int tiles = 1; tiles <= 80; ++tiles) print<6>(tiles), print<12>(tiles);
}
"""


@pytest.fixture(scope="module")
def rings(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    src, exe = str(d / "ring.cpp"), str(d / "ring")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, src, "-o", exe], check=True, timeout=120)
    out = {}
    for line in subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout.splitlines():
        kind, slots, tiles, *rest = line.split()
        out.setdefault((int(slots), int(tiles)), {"t": [], "l": []})[kind].append([int(x) for x in rest])
    return out


def test_every_tile_is_loaded_once_in_the_order_of_use(rings):
    for (slots, tiles), ring in rings.items():
        order = [(bool(v), t) for _, _, v, t in ring["l"]]
        want = [(False, 0)] + [x for s in range(1, tiles) for x in ((False, s), (True, s - 1))] + [(True, tiles - 1)]
        assert order == want
        for s, (k, v, _, _) in enumerate(ring["t"]):
            assert order[k] == (False, s) and order[v] == (True, s)
        assert [(s, p) for s, p, _, _ in ring["l"]] == [(i % slots, i // slots % 2) for i in range(2 * tiles)]


def test_no_wait_for_a_phase_behind_one_not_seen(rings):
    for (slots, tiles), ring in rings.items():
        told = [k_before for _, _, k_before, _ in ring["t"]]
        for is_v in (False, True):
            seen = set()  # the loads that this waiter has seen land, in the order of its waits
            for s, (k, v, k_before, _) in enumerate(ring["t"]):
                if is_v and k_before >= 0:
                    seen.add(ring["t"][k_before][0])
                i = v if is_v else k
                assert i < slots or i - slots in seen, (slots, tiles, is_v, s)
                seen.add(i)
        # the K tiles that the other waiter announces are those, at most K_0 and one more: a single-phase barrier each
        announced = [s for s, (_, _, _, v_after) in enumerate(ring["t"]) if v_after]
        assert announced == sorted(t for t in told if t >= 0)
        assert len(announced) <= 2 and len([s for s in announced if s > 0]) <= 1


def test_the_announcement_is_needed(rings):
    """Without it, every list of more than half the slots' tiles has such a wait."""
    for (slots, tiles), ring in rings.items():
        seen, bad = set(), 0
        for _, v, _, _ in ring["t"]:
            bad += not (v < slots or v - slots in seen)
            seen.add(v)
        assert (bad > 0) == (tiles > slots // 2)
