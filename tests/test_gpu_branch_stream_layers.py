"""The streaming branch kernel over more (kv head, layer) problems than there are SMs, where it takes narrow CTAs, two on an
SM, against the oracle."""
import numpy as np
import pytest

import oracle
from tests.helpers import assert_close
from tests.test_gpu_branch_layers import make_layers, run_layers

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2504_08242_b200 as J
    c = J.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("L,B,Hq,Hkv,P,n,lens,launches", [
    (5, 8, 32, 32, 300, 1, [1, 17, 64, 100, 128, 129, 200, 257], 1),   # 160 problems
    (10, 3, 16, 16, 0, 1, [1, 2, 49], 1),                              # 160 of a few chunks each, no prefix
    (16, 2, 40, 20, 1029, 2, [2, 300], 1),                             # 320, more than two per SM; grouped heads
    (19, 4, 32, 32, 70, 1, [1, 16, 17, 33], 2),                        # 512, then the rest of the layers: 96
])
def test_more_problems_than_sms(ctx, D, L, B, Hq, Hkv, P, n, lens, launches):
    layers, scap = make_layers(900 + L, L, B, Hq, Hkv, D, P, n, lens)
    scale = 1.0 / np.sqrt(D)
    got, n_launches = run_layers(ctx, layers, scap, B, Hq, D, P, n, lens, scale, batched=True)
    assert n_launches == launches
    lens_np = np.asarray(lens, np.int32)
    for l in sorted({0, 1, L // 2, L - 1}):
        Lr, (out, lse, sk, sv) = layers[l], got[l]
        rk, rv = Lr["sk"].copy(), Lr["sv"].copy()
        oracle.kv_append(rk, rv, Lr["kn"], Lr["vn"], pos_per_seq=(lens_np - n).astype(np.int32))
        ref, ref_lse = oracle.branch(Lr["q"], Lr["pk"], Lr["pv"], P, rk, rv, lens_np, scale,
                                     n_threads=oracle.hardware_threads(), return_lse=True)
        assert_close(out, ref, f"layer {l}")
        assert np.max(np.abs(lse - ref_lse)) < 2e-2
        assert np.array_equal(sk, rk) and np.array_equal(sv, rv)
