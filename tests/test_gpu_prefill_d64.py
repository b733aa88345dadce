"""head_dim 64 on the tcgen05 prefill kernels, against the oracle (outputs, LSE, caches bit for bit): tile edges and
remainders of the one-tile form, the launch counts on both sides of 64 rows, the two-tile form with a ragged block, and
long walks on small grids (several CTAs share a walk)."""
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


@pytest.mark.parametrize("B,Hq,Hkv,parts", [
    (1, 2, 1, [1, 64, 65, 127, 128]),       # two launches up to 64 rows, one above; positions off the tile grid
    (2, 8, 2, [129, 300]),
    (2, 32, 8, [100, 700]),                 # enough blocks for two query tiles per CTA, the last block ragged
    (3, 32, 32, [515]),
    (1, 4, 4, [2980, 384]),                 # a long walk on a small grid
    (1, 8, 2, [3150, 100]),
])
@pytest.mark.parametrize("fused", [True, False])
def test_head_dim_64(ctx, B, Hq, Hkv, parts, fused):
    S = sum(parts)
    w = synth.PrefillWorkload("d64", 900 + S, B, Hq, Hkv, 64, S, S, S + 9)
    q, k, v = w.make()
    n0 = ctx.launch_count()
    out, kc, vc, lse = run_gpu_prefill(ctx, q, k, v, parts, w.capacity, w.scale, want_lse=True, fused=fused)
    assert ctx.launch_count() - n0 == sum(1 if fused and n > 64 else 2 for n in parts)
    ref, ref_lse = oracle.full_causal(q, k, v, w.scale, n_threads=oracle.hardware_threads(), return_lse=True)
    assert_close(out, ref, w.name)
    assert np.max(np.abs(lse - ref_lse)) < 2e-2
    assert np.array_equal(kc[:, :, :S], token_to_cache(k, S)) and np.array_equal(vc[:, :, :S], token_to_cache(v, S))
    assert (kc[:, :, S:] == 0x7FC0).all() and (vc[:, :, S:] == 0x7F80).all()
