"""How the torch side of the modules gets loaded: by the first call."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_importing_the_modules_loads_no_library():
    """Only a call needs the CUDA library; without one it says so, and a CPU tensor is refused before that."""
    code = """
import torch
from paper_2405_03133_b200 import LoryError, layer
m = layer.LoryMoE(8, 8, 2, T=4, device="cpu")
for call in (lambda: m(torch.zeros(1, 4, 8, dtype=torch.bfloat16)), layer._glue):
    try:
        call()
    except RuntimeError as e:
        print(type(e).__name__)
assert issubclass(LoryError, RuntimeError)
"""
    env = dict(os.environ, LORY_LIBRARY=os.path.join(ROOT, "no_such_library.so"))
    out = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert out.stdout.split() == ["RuntimeError", "LoryError"], out.stderr
