"""Errors inside the native entry points arrive as the Python exceptions they are, with the interpreter intact.
A tensor that says it is on a device but has no memory (no device is needed for one) raises at the point where
its address is taken; in a process of its own, so that a crash is a failure and not the end of the run."""
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
context = [object(), None, binding.BF16]
arguments = {"encode": [t, None, None, t, 4, None, t, None, t, None, t], "decode": [t, None, t, None, t, None, t, None, None, None, t, None, t]}
name = sys.argv[1]
for _ in range(3):
    try:
        getattr(binding._native, name)(*context, *arguments[name])
    except RuntimeError as e:
        print("raised", type(e).__name__)
"""


@pytest.mark.parametrize("name", ["encode", "decode"])
def test_a_tensor_without_memory(name):
    run = subprocess.run([sys.executable, "-c", SCRIPT, name], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0 and run.stdout.split() == ["raised", "RuntimeError"] * 3, run.stderr[-2000:]
