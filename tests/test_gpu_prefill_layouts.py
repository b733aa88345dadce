"""The layouts a prefill call can take (several CTAs sharing a query tile's KV walk, two query tiles per CTA, heads of a
group), against the oracle: outputs, LSE and caches, group sizes that do and do not divide a tile, chunk lengths around
multiples of a tile's tokens, walks of fewer tiles than a cluster has CTAs and of many."""
import numpy as np
import pytest

import oracle
from workloads import synth
from tests.helpers import assert_close, run_gpu_prefill, token_to_cache

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2504_08242_b200 as J
    c = J.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("B,Hq,Hkv,parts", [
    (1, 6, 2, [126, 42, 43, 300]),           # groups of 3: 42 tokens x 3 heads, K/V and query tiles do not align
    (1, 10, 2, [25, 26, 100, 420]),          # groups of 5
    (2, 8, 1, [15, 16, 17, 129]),            # groups of 8: 16 tokens per tile
    (1, 65, 1, [3, 70]),                     # a group that only packs whole or by 5 and 13
    (1, 4, 4, [1, 500, 64, 2100, 64]),       # no group: 8 CTAs share the long walks, short ones stay whole
    (1, 16, 4, [700, 60, 1400, 100]),        # clusters of several sizes as the walk grows
    (3, 32, 8, [150, 150, 333]),             # pairs of packed tiles, several waves
])
def test_layouts(ctx, D, B, Hq, Hkv, parts):
    S = sum(parts)
    w = synth.PrefillWorkload("layout", 950 + S + D, B, Hq, Hkv, D, S, S, S + 5)
    q, k, v = w.make()
    ref, ref_lse = oracle.full_causal(q, k, v, w.scale, n_threads=oracle.hardware_threads(), return_lse=True)
    for fused in (True, False):
        out, kc, vc, lse = run_gpu_prefill(ctx, q, k, v, parts, w.capacity, w.scale, want_lse=True, fused=fused)
        assert_close(out, ref, f"{w.name} fused={fused}")
        assert np.max(np.abs(lse - ref_lse)) < 2e-2
        assert np.array_equal(kc[:, :, :S], token_to_cache(k, S)) and np.array_equal(vc[:, :, :S], token_to_cache(v, S))
        assert (kc[:, :, S:] == 0x7FC0).all() and (vc[:, :, S:] == 0x7F80).all()
