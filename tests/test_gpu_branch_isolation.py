"""A branch's K rows that hold NaN or Inf stay within that branch: the outputs of the other branches are, bit for bit, what
they are with finite rows."""
import numpy as np
import pytest

from tests.helpers import to_dev
from tests.test_gpu_branch_layers import make_layers

pytestmark = pytest.mark.gpu

HQ, HKV, N = 32, 8, 5


@pytest.mark.parametrize("bad", [0x7FC0, 0x7F80, 0xFF80])  # NaN, +Inf, -Inf
@pytest.mark.parametrize("D,B,P,fused", [
    (128, 16, 600, True),
    (128, 16, 600, False),
    (128, 3, 0, True),      # no prefix: the other branches' rows first meet a tile that they see nothing of
    (64, 16, 2561, True),
    (64, 16, 2561, False),
])
def test_non_finite_keys_stay_in_their_branch(D, B, P, fused, bad):
    import torch
    import paper_2504_08242_b200 as J
    c = J.Context(0)
    if D == 128:
        c.select_branch_kernel(J.BRANCH_TENSOR_CORE)
    lens = np.asarray([N + 300] + [N + 130 + 7 * i for i in range(1, B)], np.int32)  # branch 0: two whole tiles and a rest
    (w,), scap = make_layers(950 + D, 1, B, HQ, HKV, D, P, N, lens)
    if not fused:  # the step's rows are in the cache
        for b, L in enumerate(lens):
            w["sk"][b, :, L - N:L] = w["kn"][b].transpose(1, 0, 2)
            w["sv"][b, :, L - N:L] = w["vn"][b].transpose(1, 0, 2)
    outs = []
    for poison in (False, True):
        sk = w["sk"].copy()
        if poison:
            sk[0, :, 17] = bad    # in the first and in the second tile
            sk[0, :, 200, 3] = bad
        d = {k: to_dev(v) for k, v in dict(w, sk=sk).items()}
        pd, sd = J.cache_desc(d["pk"], d["pv"]), J.cache_desc(d["sk"], d["sv"])
        out = torch.full((B, N, HQ, D), 7.0, dtype=torch.float32, device="cuda")
        lse = torch.full((B, HQ, N), 7.0, dtype=torch.float32, device="cuda")
        dl = torch.from_numpy(lens).cuda()
        if fused:
            c.branch_append_attn(d["q"], d["kn"], d["vn"], pd, P, sd, dl, scap, B, HQ, N, 1.0 / np.sqrt(D), out, lse)
        else:
            c.branch_attn(d["q"], pd, P, sd, dl, scap, B, HQ, N, 1.0 / np.sqrt(D), out, lse)
        torch.cuda.synchronize()
        assert c.poll_device_status() == 0
        outs.append((out.cpu().numpy(), lse.cpu().numpy()))
    c.close()
    (clean, clean_lse), (out, lse) = outs
    assert np.isfinite(clean).all() and np.isfinite(clean_lse).all()
    assert not np.isfinite(out[0]).all()  # the rows were read
    assert np.array_equal(out[1:], clean[1:]) and np.array_equal(lse[1:], clean_lse[1:])
