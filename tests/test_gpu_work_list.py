"""The attention's work list where its building changes: around the block's 256 threads, on both
sides of the limit up to which the items are sorted one by one, and of the limit up to which the
launches overlap."""
import numpy as np
import pytest
import torch

from paper_2608_19662_b200 import workloads as wl

from pipeline import gpu_encode, make_ctx, max_abs, oracle_encode

pytestmark = pytest.mark.gpu


# two groups: 1024 work items (the sorting limit) are 512 one-pair resources
@pytest.mark.parametrize("n", [1, 255, 257, 511, 512, 513, 1300])
def test_items_around_the_plan_limits(n):
    sh = wl.Shape(4, 2, 128, 1e6, "bf16")        # 128 tokens per work item
    rng = np.random.default_rng(n)
    lens = rng.integers(0, 9, n).astype(np.int32)
    lens[0] = 300 if n == 1 else 129             # one resource of more than one item
    pool = wl.pack_resources(sh, n, lens, [np.ones(int(k), np.uint8) for k in lens], bulk=True)
    rc = make_ctx(sh, max_pos=512)
    o, kc, vc = gpu_encode(rc, pool)
    ref, kc_ref, vc_ref = oracle_encode(pool)
    assert max_abs(o, ref) < 1e-2
    assert torch.equal(vc.cpu().view(torch.int16), torch.from_numpy(vc_ref).to(torch.bfloat16).view(torch.int16))
    assert rc.poll_status() == 0
