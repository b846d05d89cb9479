"""The native half of the binding turns what torch's C++ API throws into Python exceptions.  The calls run in a process of
their own, so that one that ends the process fails its test alone; none of them reaches the library, so no GPU is needed."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import torch
from paper_2501_04304_b200 import binding as b
class Stream:
    cuda_stream = 0
"""


@pytest.mark.parametrize("call", [
    # an output without a first dimension: its stride is asked for right before the library is called
    "b.native().linear(0, 0, 8, 0, 0, 0, torch.zeros(4, 32, dtype=torch.uint8), None, None, None, torch.zeros(()), None, False, Stream())",
    # a tensor without storage: its address is
    "x = torch.zeros(4, 32, dtype=torch.uint8).to_sparse()\n"
    "b.native().linear(0, 0, 8, 0, 0, 0, x, None, None, None, torch.zeros(4, 8), None, False, Stream())",
    # a CPU tensor where a buffer is to be made on the tensor's device
    "q = torch.zeros(1, 16, 1, 40, dtype=torch.float16)\nb.native().cross_attn_logq(q, q, q, 8, 0, None, None, 0, 0, None, 0, Stream())",
    # no current stream to take without a device
    "assert not torch.cuda.is_available() or 0 / 0\nb.native().self_attn_logq(*[torch.zeros(1, 16, 1, 40)] * 3, 8, None, None, 0, None)",
], ids=["stride", "storage", "allocation", "stream"])
def test_exceptions_of_the_tensor_library_reach_python(call):
    body = "\n    ".join(call.split("\n"))
    script = PRELUDE + f"b.native()\ntry:\n    {body}\n    print('no exception')\nexcept Exception as e:\n    print('raised', type(e).__name__)\n"
    from paper_2501_04304_b200 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.startswith("raised"), (r.returncode, r.stdout, r.stderr[-2000:])
