"""The package imports, and its host functions work, with a torch that has no
CUDA in it; calls then read the current stream through torch's public call."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
import torch
for name in {names!r}:
    if hasattr(torch._C, name):
        delattr(torch._C, name)
import paper_2609_17475_gb300 as jf
from paper_2609_17475_gb300 import binding
assert jf.jf_kv_page_bytes(4, 256, 256) == 294912
assert len(jf.jf_tq4_codebook(128)) == 16
class Stream:
    cuda_stream = 77
torch.cuda.current_stream = lambda: Stream()
assert binding._stream(None) == 77
assert binding._stream(Stream()) == 77 and binding._stream(5) == 5
"""


@pytest.mark.parametrize("names", [["_cuda_getCurrentRawStream", "_cuda_getDevice"],
                                   ["_cuda_getCurrentRawStream"], ["_cuda_getDevice"]])
def test_import_without_the_private_stream_functions(names):
    done = subprocess.run([sys.executable, "-c", PROGRAM.format(names=names)], cwd=ROOT,
                          capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr[-2000:]
