"""Branch attention with head_dim 64 where it takes the tensor-core kernel (many stacked rows), against the oracle: the tile
lists, in which prefix and suffix tiles take turns behind the leading prefix tiles, with few and many entries of either
kind, in CTAs that walk a unit alone and in clusters."""
import numpy as np
import pytest

import oracle
from workloads import synth
from tests.helpers import assert_close, to_dev, to_bits
from tests.test_gpu_branch_layers import make_layers, run_layers
from tests.test_gpu_branch_tc import random_tree_masks

pytestmark = pytest.mark.gpu

B, HQ, HKV, D, N = 16, 32, 8, 64, 5  # 320 stacked rows per kv head


@pytest.fixture(scope="module")
def ctx():
    import paper_2504_08242_b200 as J
    c = J.Context(0)
    yield c
    c.close()


def suffix_lengths(entries):
    """Branch lengths, the step's block included: the tiles of suffix rows before it."""
    return {"none": [N] * B,                                  # the step's block is the only suffix entry
            "one": [N] * (B - 1) + [N + 100],                 # one row tile has one more
            "many": [N + 64 + 32 * i for i in range(B)]}[entries]


@pytest.mark.parametrize("entries", ["none", "one", "many"])
@pytest.mark.parametrize("L,P", [(8, 640), (8, 641), (8, 768), (8, 1024), (8, 2048), (4, 641), (4, 4100), (3, 1281), (3, 2048)])
def test_layers(ctx, L, P, entries):
    lens = suffix_lengths(entries)
    layers, scap = make_layers(800 + L, L, B, HQ, HKV, D, P, N, lens)
    scale = 1.0 / np.sqrt(D)
    got, launches = run_layers(ctx, layers, scap, B, HQ, D, P, N, lens, scale, batched=True)
    assert launches == 1
    lens_np = np.asarray(lens, np.int32)
    for l in (0, L - 1):  # (units of all layers are numbered through: the first and the last ones)
        Lr, (out, lse, sk, sv) = layers[l], got[l]
        rk, rv = Lr["sk"].copy(), Lr["sv"].copy()
        oracle.kv_append(rk, rv, Lr["kn"], Lr["vn"], pos_per_seq=(lens_np - N).astype(np.int32))
        ref, ref_lse = oracle.branch(Lr["q"], Lr["pk"], Lr["pv"], P, rk, rv, lens_np, scale,
                                     n_threads=oracle.hardware_threads(), return_lse=True)
        assert_close(out, ref, f"layer {l}")
        assert np.max(np.abs(lse - ref_lse)) < 2e-2
        assert np.array_equal(sk, rk) and np.array_equal(sv, rv)


@pytest.mark.parametrize("P,entries", [(700, "many"), (2561, "none"), (2561, "many"), (4096, "one"), (4096, "many")])
@pytest.mark.parametrize("mode", ["plain", "fused", "tree"])
def test_one_layer(ctx, P, entries, mode):
    import torch
    import paper_2504_08242_b200 as J
    lens = np.asarray(suffix_lengths(entries), np.int32)
    (w,), scap = make_layers(850, 1, B, HQ, HKV, D, P, N, lens)
    scale = 1.0 / np.sqrt(D)
    rk, rv = w["sk"].copy(), w["sv"].copy()
    oracle.kv_append(rk, rv, w["kn"], w["vn"], pos_per_seq=(lens - N).astype(np.int32))
    if mode != "fused":
        w["sk"], w["sv"] = rk.copy(), rv.copy()
    nt = oracle.hardware_threads()
    tm = random_tree_masks(851, B, N)
    if mode == "tree":
        ref, ref_lse = oracle.branch_tree(w["q"], w["pk"], w["pv"], P, rk, rv, lens, tm, scale, n_threads=nt, return_lse=True)
    else:
        ref, ref_lse = oracle.branch(w["q"], w["pk"], w["pv"], P, rk, rv, lens, scale, n_threads=nt, return_lse=True)
    d = {k: to_dev(v) for k, v in w.items()}
    pd, sd = J.cache_desc(d["pk"], d["pv"]), J.cache_desc(d["sk"], d["sv"])
    out = torch.full((B, N, HQ, D), float("nan"), dtype=torch.float32, device="cuda")
    lse = torch.full((B, HQ, N), float("nan"), dtype=torch.float32, device="cuda")
    dl = torch.from_numpy(lens).cuda()
    if mode == "fused":
        ctx.branch_append_attn(d["q"], d["kn"], d["vn"], pd, P, sd, dl, scap, B, HQ, N, scale, out, lse)
    elif mode == "tree":
        ctx.branch_attn_tree(d["q"], pd, P, sd, dl, torch.from_numpy(tm.view(np.int32)).cuda(), scap, B, HQ, N, scale, out, lse)
    else:
        ctx.branch_attn(d["q"], pd, P, sd, dl, scap, B, HQ, N, scale, out, lse)
    torch.cuda.synchronize()
    assert ctx.poll_device_status() == 0
    assert_close(out.cpu().numpy(), ref, mode)
    assert np.max(np.abs(lse.cpu().numpy() - ref_lse)) < 2e-2
    assert np.array_equal(to_bits(d["sk"]), rk) and np.array_equal(to_bits(d["sv"]), rv)
