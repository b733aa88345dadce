"""The tensor-core branch kernel where its units -- (layer, kv head, row tile) -- fill the machine more than once: full waves
with a CTA per unit, the rest shared by clusters; and its tile lists, in which prefix and suffix tiles take turns."""
import numpy as np
import pytest

import oracle
from tests.helpers import assert_close
from tests.test_gpu_branch_layers import make_layers, run_layers
from tests.test_gpu_branch_tc import run_case, ctx as tc_ctx  # noqa: F401 (fixture: the kernel pinned)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["plain", "fused", "tree"])
def test_one_layer_with_a_shared_rest(tc_ctx, mode):  # noqa: F811
    """64 kv heads x 3 row tiles = 192 units."""
    run_case(tc_ctx, 710, 12, 128, 64, 1300, 16, [16, 33, 140, 16, 200, 300, 144, 145, 17, 80, 128, 272], mode)


@pytest.mark.parametrize("P,lens", [
    (0, [8, 300, 9, 520, 136, 137]),             # no prefix: the list is the suffix part alone
    (128 * 4, [8, 8, 8, 8, 8, 8]),               # as many prefix tiles as lead the list, and only the step's block
    (128 * 5 + 1, [8 + 128, 9, 8, 264, 8, 400]),  # both kinds left over, odd numbers of either
    (128 * 12, [9, 8, 8, 8, 8, 8]),              # two suffix entries
])
@pytest.mark.parametrize("mode", ["plain", "fused"])
def test_mixed_tile_lists(tc_ctx, P, lens, mode):  # noqa: F811
    run_case(tc_ctx, 720, 6, 32, 8, P, 8, lens, mode)


def test_layers_with_a_shared_rest():
    """8 layers x 8 kv heads x 3 row tiles = 192 units over all layers."""
    import paper_2504_08242_b200 as J
    L, B, Hq, Hkv, D, P, n = 8, 16, 32, 8, 128, 1100, 5
    lens = [5 + 17 * i for i in range(B)]
    layers, scap = make_layers(730, L, B, Hq, Hkv, D, P, n, lens)
    scale = 1.0 / np.sqrt(D)
    c = J.Context(0)
    got, launches = run_layers(c, layers, scap, B, Hq, D, P, n, lens, scale, batched=True)
    c.close()
    assert launches == 1
    lens_np = np.asarray(lens, np.int32)
    for Lr, (out, lse, sk, sv) in zip(layers, got):
        rk, rv = Lr["sk"].copy(), Lr["sv"].copy()
        oracle.kv_append(rk, rv, Lr["kn"], Lr["vn"], pos_per_seq=(lens_np - n).astype(np.int32))
        ref, ref_lse = oracle.branch(Lr["q"], Lr["pk"], Lr["pv"], P, rk, rv, lens_np, scale,
                                     n_threads=oracle.hardware_threads(), return_lse=True)
        assert_close(out, ref, "layers with a shared rest")
        assert np.max(np.abs(lse - ref_lse)) < 2e-2
        assert np.array_equal(sk, rk) and np.array_equal(sv, rv)
