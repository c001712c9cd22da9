"""The wrapper tells the caller's current stream from the solver's by its
handle; torch's private accessor of that handle may be missing."""
import subprocess
import sys
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent
CODE = """
import types, torch
if {missing}:
    vars(torch._C).pop("_cuda_getCurrentRawStream", None)
else:
    torch._C._cuda_getCurrentRawStream = lambda dev: 100 + dev
torch.cuda.current_device = lambda: 0
waits = []
stream = types.SimpleNamespace(cuda_stream=100, wait_stream=waits.append)
torch.cuda.current_stream = lambda dev=None: stream
from paper_2501_15314_gb300.api import IBMSolver
s = object.__new__(IBMSolver)
s.lib = types.SimpleNamespace(f=lambda ctx, x: x + 1)
s.ctx, s.stream, s._on = None, stream, (100, 0)
assert s._call("f", 4) == 5 and not waits        # the solver's own stream
s._on = (200, 0)
assert s._call("f", 4) == 5 and len(waits) == 2  # another one: before and after
"""


@pytest.mark.parametrize("missing", [False, True])
def test_call_waits_for_other_streams_only(missing):
    subprocess.run([sys.executable, "-c", CODE.format(missing=missing)], cwd=ROOT, check=True)
