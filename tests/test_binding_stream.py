"""The stream that a call is enqueued on when none is given: torch's current one, also with a torch whose internal calls for it
have other names."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WITHOUT = """
import sys, types, torch
delattr(torch._C, sys.argv[1])
from paper_2504_08242_b200 import binding
stream = types.SimpleNamespace(cuda_stream=4096)
torch.cuda.current_stream = lambda *a: stream
assert binding._stream(None) == 4096 and binding._stream(stream) == 4096 and binding._stream(77) == 77
"""


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_without_the_internal_calls(missing):
    subprocess.run([sys.executable, "-c", WITHOUT, missing], check=True, cwd=ROOT, timeout=300)


FIRST = """
import paper_2504_08242_b200 as J
ctx = J.Context(0)  # before torch has touched the GPU
ctx.wait_probe(1000)
assert ctx.poll_device_status() == J.ERR_TIMEOUT and ctx.poll_device_status() == 0
ctx.close()
"""


@pytest.mark.gpu
def test_a_call_before_torch_has_touched_the_gpu():
    subprocess.run([sys.executable, "-c", FIRST], check=True, cwd=ROOT, timeout=300)


@pytest.mark.gpu
def test_the_current_stream():
    import torch
    from paper_2504_08242_b200 import binding
    assert binding._stream(None) == torch.cuda.current_stream().cuda_stream
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert binding._stream(None) == side.cuda_stream
