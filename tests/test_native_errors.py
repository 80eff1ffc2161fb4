"""Errors inside the native entry points arrive as the Python exceptions they are, with the interpreter intact.
A tensor that says it is on a device but has no memory (no device is needed for one) raises on the way to the
library call, one without dimensions where it is asked for a size; in a process of its own, so that a crash is a failure and not the end of the run."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SCRIPT = """
import sys
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2608_19662_b200 import binding

binding.load_library()
with FakeTensorMode():
    t = torch.empty((4, 4, 4), device="cuda:0", dtype=torch.bfloat16)
    point = torch.empty((), device="cuda:0", dtype=torch.bfloat16)
context = [object(), None, binding.BF16]
arguments = {"dimensions": [point] * 4 + [4] + [point] * 4 + [None, point],
             "encode": [t, None, None, t, 4, None, t, None, t, None, t],
             "decode": [t, None, t, None, t, None, t, None, None, None, t, None, t]}
name = sys.argv[1]
for _ in range(3):
    try:
        getattr(binding._native, "encode" if name == "dimensions" else name)(*context, *arguments[name])
    except Exception as e:
        print("raised", "RuntimeError" if isinstance(e, RuntimeError) else type(e).__name__)
"""


@pytest.mark.parametrize("name,error", [("encode", "RuntimeError"), ("decode", "RuntimeError"), ("dimensions", "IndexError")])
def test_errors_of_tensors_arrive(name, error):
    run = subprocess.run([sys.executable, "-c", SCRIPT, name], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0 and run.stdout.split() == ["raised", error] * 3, run.stderr[-2000:]
