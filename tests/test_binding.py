"""The extension module between Python and the scoring calls, without a GPU."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CALL = r"""
import torch
from paper_2508_13231_b200 import kvp
try:
    print(kvp._native().current_stream() >= 0)
except RuntimeError as e:
    print("RuntimeError")
"""


def test_what_torch_throws_is_raised():
    """torch's C++ calls throw where there is no device; that is an exception in Python and not the end of the process."""
    import torch
    r = subprocess.run([sys.executable, "-c", CALL], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["True" if torch.cuda.is_available() else "RuntimeError"]
