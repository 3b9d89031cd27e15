"""The binding passes torch's current stream, through torch's raw-handle binding where
there is one and through the public stream object where there is none."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROG = """
import types, torch
if {without}:
    if hasattr(torch._C, "_cuda_getCurrentRawStream"):
        del torch._C._cuda_getCurrentRawStream
else:
    torch._C._cuda_getCurrentRawStream = lambda dev: 1000 + dev
torch.cuda.current_device = lambda: 3
torch.cuda.current_stream = lambda: types.SimpleNamespace(cuda_stream=77)
from paper_1905_06234_gb300 import _native
print(_native._stream())
"""


@pytest.mark.parametrize("without,handle", [(False, 1003), (True, 77)])
def test_handle(without, handle):
    r = subprocess.run([sys.executable, "-c", PROG.format(without=without)], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert int(r.stdout.split()[-1]) == handle
