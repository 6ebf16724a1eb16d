"""The Python binding's own work (arguments, errors) where it needs no GPU."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_VMAP = """
import types
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2505_18573_b200 import build
build.build()
from paper_2505_18573_b200 import binding as e3

with FakeTensorMode():
    ent = torch.empty((3, 8), device="cuda")
out, stream = torch.zeros(2, dtype=torch.float64), types.SimpleNamespace(cuda_stream=0)
try:
    torch.vmap(lambda x: e3.e3_masked_mean_entropy_static(x, None, out, stream))(ent)
except RuntimeError as e:
    print("raised:", e)
"""


def test_a_tensor_without_memory_raises():
    """Found when the call's pointers are taken, with the GIL released: it has to come back as an exception."""
    r = subprocess.run([sys.executable, "-c", _VMAP], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("raised:"), r.stderr[-2000:]
