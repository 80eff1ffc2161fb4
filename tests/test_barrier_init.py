"""Every kernel that sets up mbarriers has all its threads pass a block barrier, on every path, between
the set-up and the first use.  (A missing one is a race that mostly goes well, and hangs or reads unfilled
shared memory when it does not: it is looked for in the sources, not on a device.)"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_19662_b200", "csrc")
INIT = re.compile(r"\bmbar_init\(|mbarrier\.init")
USE = re.compile(r"\b(?:rc_)?mbar_(?:wait|arrive|expect_tx)\b|\btma_load\w*\(|\bcp_async_arrive\(|\btc_commit\(")


def kernels(text):
    """(name, signature, body) of every __global__ function."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__global__", text):
        head = text[m.start():text.index("{", m.start())]
        if ";" in head:
            continue
        at, depth = text.index("{", m.start()), 0
        for end in range(at, len(text)):
            depth += (text[end] == "{") - (text[end] == "}")
            if depth == 0:
                break
        yield re.search(r"(\w+)\s*\(", re.sub(r"__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)|__global__|template\s*<[^>]*>", "", head)).group(1), head, text[at:end]


def _unguarded(body):
    """A use of a barrier that no block barrier at the kernel's top level separates from the set-up, or None."""
    start = max(m.end() for m in INIT.finditer(body))
    depth = body[:start].count("{") - body[:start].count("}")
    for m in re.finditer(r"[{}]|__syncthreads\(\);|" + USE.pattern, body[start:]):
        if m.group() == "{":
            depth += 1
        elif m.group() == "}":
            depth -= 1
        elif m.group().startswith("__syncthreads"):
            if depth == 1:
                return None
        else:
            return m.group()
    return None


FOUND = [pytest.param(body, id=f"{os.path.basename(path)}:{name}") for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")))
         for name, _, body in kernels(open(path).read()) if INIT.search(body)]


def test_the_kernels_were_found():
    assert len(FOUND) >= 3


@pytest.mark.parametrize("body", FOUND)
def test_block_barrier_between_set_up_and_use(body):
    assert _unguarded(body) is None
