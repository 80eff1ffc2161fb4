"""Kernels that come up while the kernel before them still runs (they call rc_grid_wait) declare no input
`const ... __restrict__` (but the rotary tables, which no kernel writes).  That form says that the data does not change during the kernel's life; the compiler
may then load it through the non-coherent path and ahead of the wait, while the kernel before still writes it.
Looked for in the sources: on a device it goes well until a compiler or a launch's timing changes."""
import glob
import os
import re

import pytest

from test_barrier_init import CSRC, kernels

FOUND = [pytest.param(signature, id=f"{os.path.basename(path)}:{name}") for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")))
         for name, signature, body in kernels(open(path).read()) if "rc_grid_wait()" in body]


def test_the_kernels_were_found():
    assert len(FOUND) >= 8


@pytest.mark.parametrize("signature", FOUND)
def test_no_input_is_promised_to_be_constant(signature):
    assert not re.search(r"const\s+\w+\s*\*\s*__restrict__\s+(?!cos_tab|sin_tab)", signature)
