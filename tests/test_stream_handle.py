"""The package imports, and finds the current stream, where torch does not have
the private function that returns a stream's handle (a build without CUDA)."""
import os
import subprocess
import sys

SCRIPT = """
import torch
if hasattr(torch._C, "_cuda_getCurrentRawStream"):
    del torch._C._cuda_getCurrentRawStream
import paper_2504_01266_gb300 as giga

class Stream:
    cuda_stream = 77

torch.cuda.current_stream = lambda device=None: Stream
assert giga._stream(torch.device("cuda", 0)) == 77
assert giga._stream(torch.device("cuda")) == 77
"""


def test_import_without_the_private_function():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=root, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr
