"""Branch calls on caches with a stride that no tensor map can carry and that no address needs: the batch stride of a cache
for one branch, the head stride of a cache with one kv head."""
import numpy as np
import pytest

import oracle
from tests.helpers import assert_close, to_dev, to_bits
from tests.test_gpu_branch_layers import make_layers

pytestmark = pytest.mark.gpu

N, UNUSED = 16, 1 << 41


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("Hkv,P", [(8, 3000), (1, 700), (8, 0)])  # 128 stacked rows per kv head
@pytest.mark.parametrize("mode", ["plain", "fused", "layers"])
def test_unused_strides(D, Hkv, P, mode):
    import torch
    import paper_2504_08242_b200 as J
    c = J.Context(0)
    L, Hq, lens = 4 if mode == "layers" else 1, 8 * Hkv, np.asarray([N + 300], np.int32)
    layers, scap = make_layers(1300 + D, L, 1, Hq, Hkv, D, P, N, lens)
    scale = 1.0 / np.sqrt(D)
    dl = torch.from_numpy(lens).cuda()
    calls, dev, refs = [], [], []
    for w in layers:
        rk, rv = w["sk"].copy(), w["sv"].copy()
        oracle.kv_append(rk, rv, w["kn"], w["vn"], pos_per_seq=lens - N)
        refs.append(oracle.branch(w["q"], w["pk"], w["pv"], P, rk, rv, lens, scale, n_threads=oracle.hardware_threads()))
        if mode == "plain":
            w = dict(w, sk=rk, sv=rv)
        t = {k: to_dev(v) for k, v in w.items()}
        t["ref_k"] = rk
        pd, sd = J.cache_desc(t["pk"], t["pv"]), J.cache_desc(t["sk"], t["sv"])
        sd.stride_batch = pd.stride_batch = UNUSED
        if Hkv == 1:
            sd.stride_head = pd.stride_head = UNUSED
        out = torch.full((1, N, Hq, D), float("nan"), dtype=torch.float32, device="cuda")
        calls.append((t["q"], t["kn"], t["vn"], pd, sd, out, None))
        dev.append(t)
    if mode == "layers":
        c.branch_append_attn_layers(calls, P, dl, scap, 1, Hq, N, scale)
    else:
        q, kn, vn, pd, sd, out, _ = calls[0]
        if mode == "plain":
            c.branch_attn(q, pd, P, sd, dl, scap, 1, Hq, N, scale, out)
        else:
            c.branch_append_attn(q, kn, vn, pd, P, sd, dl, scap, 1, Hq, N, scale, out)
    torch.cuda.synchronize()
    for call, t, ref in zip(calls, dev, refs):
        assert_close(call[5].cpu().numpy(), ref, mode)
        assert np.array_equal(to_bits(t["sk"]), t["ref_k"])
    c.close()
