"""The package imports with a torch that was built without CUDA (the calls need a GPU, the import does not)."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import torch
for name in [n for n in dir(torch._C) if n.startswith("_cuda_")]:
    delattr(torch._C, name)
from paper_2410_05265_b200 import binding, block, inputs
assert callable(binding.Context) and callable(block.Block)
"""


def test_import_with_a_torch_without_cuda():
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
