"""What the exponentials of the prefill kernels keep: log-sum-exps to 32-bit accuracy, and NaN keys."""
import numpy as np
import pytest

import oracle
from workloads import synth
from tests.helpers import assert_close, run_gpu_prefill, to_dev

pytestmark = pytest.mark.gpu

# Scores of unit-normal inputs, |s| < 8.  A score: D / 16 <= 8 additions of partial sums below 64 / scale, half a unit in the
# last place (3.8e-6) each, times the scale 1 / sqrt(D): below 3.8e-6; its scaling to powers of two and back 1e-6; an exponential
# 2^-22; the row sum some 2^-24 for each addition of a chain that grows with every tile, below 3e-6 for 32 tiles.
LSE_TOL = 1e-5


@pytest.fixture(scope="module")
def ctx():
    import paper_2504_08242_b200 as J
    c = J.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("D,B,Hq,Hkv,parts", [
    (64, 1, 4, 4, [64, 64, 128]),           # two launches, then one
    (64, 2, 8, 2, [300, 129]),
    (64, 1, 4, 4, [2980, 384]),             # several CTAs share a long walk
    (64, 2, 32, 8, [700]),                  # two query tiles per CTA
    (128, 1, 4, 2, [100, 257, 30]),
    (128, 1, 8, 8, [2048, 256]),            # several CTAs share a long walk
    (128, 8, 32, 8, [30, 200]),             # many small query tiles
])
@pytest.mark.parametrize("fused", [True, False])
def test_log_sum_exps(ctx, D, B, Hq, Hkv, parts, fused):
    S = sum(parts)
    w = synth.PrefillWorkload("lse", 1000 + S + D, B, Hq, Hkv, D, S, S, S + 3)
    q, k, v = w.make()
    out, _, _, lse = run_gpu_prefill(ctx, q, k, v, parts, w.capacity, w.scale, want_lse=True, fused=fused)
    ref, ref_lse = oracle.full_causal(q, k, v, w.scale, n_threads=oracle.hardware_threads(), return_lse=True)
    assert_close(out, ref, w.name)
    assert np.max(np.abs(lse - ref_lse)) < LSE_TOL


def test_log_sum_exps_behind_a_shared_prefix(ctx):
    import torch
    import paper_2504_08242_b200 as J
    B, Hq, Hkv, D, P, n, seed = 11, 16, 16, 128, 700, 72, 1100
    q = synth.normal_bf16(seed, 1, (B, n, Hq, D))
    pk, pv = synth.normal_bf16(seed, 2, (1, Hkv, P, D)), synth.normal_bf16(seed, 3, (1, Hkv, P, D))
    sk, sv = synth.normal_bf16(seed, 4, (B, Hkv, n, D)), synth.normal_bf16(seed, 5, (B, Hkv, n, D))
    scale = 1.0 / np.sqrt(D)
    _, ref_lse = oracle.branch(q, pk, pv, P, sk, sv, np.full(B, n, np.int32), scale, n_threads=oracle.hardware_threads(),
                               return_lse=True)
    d = [to_dev(x) for x in (q, pk, pv, sk, sv)]
    out = torch.empty(B, n, Hq, D, dtype=torch.float32, device="cuda")
    lse = torch.empty(B, Hq, n, dtype=torch.float32, device="cuda")
    ctx.branch_prefill_attn(d[0], J.cache_desc(d[1], d[2]), P, J.cache_desc(d[3], d[4]), Hq, n, 0, scale, out, lse)
    torch.cuda.synchronize()
    assert np.max(np.abs(lse.cpu().numpy() - ref_lse)) < LSE_TOL


@pytest.mark.parametrize("D,Hq,Hkv,S", [(64, 4, 4, 90), (64, 32, 8, 1500), (128, 4, 4, 90), (128, 32, 8, 1500)])
@pytest.mark.parametrize("row", [9, 83])
def test_a_nan_key_is_not_lost(ctx, D, Hq, Hkv, S, row):
    """No value of a row from the key on is finite, every row before it is."""
    w = synth.PrefillWorkload("nan", 1200 + D + S, 1, Hq, Hkv, D, S, S, S)
    q, k, v = w.make()
    k = k.copy()
    k[:, row] = 0x7FC0
    out = run_gpu_prefill(ctx, q, k, v, [S], S, w.scale, fused=True)[0]
    assert np.isfinite(out[:, :row]).all()
    assert not np.isfinite(out[:, row:]).any()
