"""The binding's stream handle without torch's private short cut."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import types
import torch
if hasattr(torch._C, "_cuda_getCurrentRawStream"):
    del torch._C._cuda_getCurrentRawStream
from paper_2605_16579_b200 import arl2
torch.cuda.current_device = lambda: 3
torch.cuda.current_stream = lambda index: types.SimpleNamespace(cuda_stream=1000 + index)
calls = []
layer = arl2.Layer.__new__(arl2.Layer)
layer.device, layer._ctx = torch.device("cuda"), None
layer._lib = types.SimpleNamespace(arl2_reset=lambda *args: calls.append(args) or 0)
layer._run("arl2_reset", -1)
assert calls == [(None, -1, 1003)], calls
"""


def test_a_call_without_the_private_stream_getter():
    subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, check=True, timeout=300)
