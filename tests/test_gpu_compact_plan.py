"""Compaction where its counting and page tables can go wrong: resource starts at every byte offset, lengths
around the 16-byte loads, more resources than the cluster has warps, more routes than threads."""
import numpy as np
import pytest
import torch

from oracle import recache_oracle as orc
from paper_2608_19662_b200 import PAGED
from paper_2608_19662_b200 import workloads as wl

from pipeline import gpu_compact, make_ctx, oracle_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,gap,requests", [
    (list(range(0, 70)), 1, 3),                       # every length to 69 at every alignment
    ([1, 15, 16, 17, 31, 33, 511, 513], 5, 1),
    ([3] * 300, 2, 2),                                # more resources than the cluster's 256 warps
    ([40, 7], 0, 140),                                # 1120 routes: a second chunk of the plan's 1024 threads
])
def test_counts_and_tables(lens, gap, requests):
    sh = wl.Shape(8, 8, 64, 1e4, "bf16")
    rng = np.random.default_rng([len(lens), requests])
    pool = wl.pack_resources(sh, 5, lens, [rng.integers(0, 2, n).astype(np.uint8) for n in lens], slot_gap=gap, bulk=True)
    pool.keep[:] = np.where(pool.keep > 0, rng.integers(1, 256, pool.keep.shape), 0)     # any nonzero byte keeps
    lists = [[int(x) for x in rng.permutation(len(lens))] for _ in range(requests)]
    vis = [rng.integers(0, 2, (8, len(x))).astype(np.uint8) for x in lists]
    req = wl.make_requests(sh, 9, pool, lists, vis, [1] * requests)
    kc = wl.normal(1, (8, pool.pool_tokens, 64), sh.torch_dtype).cuda()
    vc = wl.normal(2, (8, pool.pool_tokens, 64), sh.torch_dtype).cuda()
    rc = make_ctx(sh, max_pos=4096)
    rows = oracle_rows(pool, req)
    flat = [r for per in rows for r in per]
    cu = orc.route_prefix(rows)
    out = gpu_compact(rc, pool, req, kc, vc, capacity=int(cu[-1]) + 1)
    assert np.array_equal(out["route_cu"].cpu().numpy(), cu)
    assert np.array_equal(out["route_idx"].cpu().numpy()[:cu[-1]], np.concatenate(flat))
    n_pages = [(len(r) + 63) // 64 for r in flat]
    free = rng.permutation(sum(n_pages) + 3).astype(np.int32)
    paged = gpu_compact(rc, pool, req, kc, vc, mode=PAGED, capacity=int(cu[-1]) + 1, n_pool_pages=len(free), free_pages=free,
                        max_pages=max(n_pages) + 1)
    table = paged["page_table"].cpu().numpy()
    at = 0
    for i, n in enumerate(n_pages):
        assert np.array_equal(table[i, :n], free[at:at + n]) and (table[i, n:] == -1).all()
        at += n
    assert np.array_equal(paged["route_len"].cpu().numpy(), [len(r) for r in flat])
    assert rc.poll_status() == 0
