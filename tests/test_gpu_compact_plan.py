"""Compaction where its three kernels change their way: the count kernel's 4096 blocks, the plan's warp per
route up to 32 routes, thread per route beyond and second round of its 1024 threads, the gather's passes of 2048
tokens and its number of blocks per pair (fewer where only indices are wanted); resource starts at every byte
offset."""
import numpy as np
import pytest
import torch

from oracle import recache_oracle as orc
from paper_2608_19662_b200 import PACKED, PAGED
from paper_2608_19662_b200 import workloads as wl

from pipeline import dev, gpu_compact, make_ctx, oracle_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,gap,requests,groups", [
    (list(range(0, 70)), 1, 3, 8),                    # every length to 69 at every alignment
    ([1, 15, 16, 17, 31, 33, 511, 513], 5, 1, 8),     # few pairs: eight blocks copy each, one where only indices are wanted
    ([3] * 300, 2, 2, 8),                             # lists of many 32-resource steps, with a remainder
    ([40, 7], 0, 140, 8),                             # 1120 routes: a second round of the plan's 1024 threads
    ([70, 3, 129], 0, 32, 1),                         # 32 routes: a warp for each
    ([70, 3, 129], 0, 33, 1),                         # 33: a thread for each; lists of one step of four, cut short
    ([2047, 2048, 2049, 4097], 3, 1, 2),              # around the gather's passes
    ([1, 2] * 2100, 0, 1, 2),                         # 4200 resources for the count's 4096 blocks
])
def test_counts_and_tables(lens, gap, requests, groups):
    sh = wl.Shape(groups, groups, 64, 1e4, "bf16")
    rng = np.random.default_rng([len(lens), requests])
    pool = wl.pack_resources(sh, 5, lens, [rng.integers(0, 2, n).astype(np.uint8) for n in lens], slot_gap=gap, bulk=True)
    pool.keep[:] = np.where(pool.keep > 0, rng.integers(1, 256, pool.keep.shape), 0)     # any nonzero byte keeps
    lists = [[int(x) for x in rng.permutation(len(lens))] for _ in range(requests)]
    vis = [rng.integers(0, 2, (groups, len(x))).astype(np.uint8) for x in lists]
    req = wl.make_requests(sh, 9, pool, lists, vis, [1] * requests)
    kc = wl.normal(1, (groups, pool.pool_tokens, 64), sh.torch_dtype).cuda()
    vc = wl.normal(2, (groups, pool.pool_tokens, 64), sh.torch_dtype).cuda()
    rc = make_ctx(sh, max_pos=4096)
    rows = oracle_rows(pool, req)
    flat = [r for per in rows for r in per]
    cu = orc.route_prefix(rows)
    out = gpu_compact(rc, pool, req, kc, vc, capacity=int(cu[-1]) + 1)
    assert np.array_equal(out["route_cu"].cpu().numpy(), cu)
    assert np.array_equal(out["route_idx"].cpu().numpy()[:cu[-1]], np.concatenate(flat))
    for name, cache in (("k_out", kc), ("v_out", vc)):
        rows_of = torch.cat([cache[i % groups][torch.from_numpy(np.asarray(r, np.int64)).cuda()] for i, r in enumerate(flat)])
        assert torch.equal(out[name][:cu[-1]].view(torch.int16), rows_of.view(torch.int16))
    only = [torch.full_like(out[name], -7) for name in ("route_cu", "route_idx")]             # the index list alone
    rc.compact_routes(kc, vc, dev(pool.keep), dev(req.res_off), dev(req.res_slot), dev(req.res_len), dev(req.vis), PACKED, *only, None, None)
    assert torch.equal(only[0], out["route_cu"]) and torch.equal(only[1][:cu[-1]], out["route_idx"][:cu[-1]])
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


@pytest.mark.parametrize("n,requests,groups", [
    (9, 8, 1), (129, 9, 1), (33, 16, 1), (17, 17, 1), (65, 32, 1), (9, 33, 1), (5, 64, 1), (9, 65, 1), (3, 128, 1), (5, 129, 1), (2, 300, 1),
    (64, 1, 8), (65, 1, 8), (100, 5, 8),
])
def test_lengths_where_lanes_share_routes(n, requests, groups):
    """A gather that plans for itself deals a route's resources to 32, 16, 8, 4, 2 or 1 lanes, four at a time, and adds up pairs
    by pair up to 512, by resource beyond."""
    test_counts_and_tables([1 + i % 3 for i in range(n)], 1, requests, groups)


@pytest.mark.parametrize("requests,visible", [(2, 0.25), (4, 1.0), (64, 1.0)])
def test_time_on_both_sides_of_the_gather_that_plans_for_itself(requests, visible):
    """4096 pairs take less than 1.3 times without a plan launch what a few pairs more take with one, indices alone.
    (Measured 0.75-1.15; with a thread to each pair and to each of 9-32 routes 1.4-1.8.)"""
    sh = wl.Shape(8, 8, 64, 1e4, "bf16")
    rc = make_ctx(sh, max_pos=4096)
    rng = np.random.default_rng(requests)
    calls = []
    for each in (512 // requests, 512 // requests + 1):
        n = each * requests
        pool = torch.zeros((8, 8 * n, 64), dtype=sh.torch_dtype, device="cuda")
        ints = lambda a, t=np.int32: dev(np.ascontiguousarray(a, dtype=t))
        args = (pool, pool, ints(np.ones(8 * n), np.uint8), ints(np.arange(requests + 1) * each), ints(np.arange(n) * 8), ints(np.full(n, 8)),
                ints(rng.random((8, n)) < visible, np.uint8), PACKED, ints(np.zeros(8 * requests + 1)), ints(np.zeros(64 * n)), None, None)
        calls.append((args, torch.empty(rc.compact_workspace_bytes(requests, n), dtype=torch.uint8, device="cuda")))
    best = [1e9, 1e9]
    start, stop = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    for _ in range(8):
        for i, (args, ws) in enumerate(calls):
            start.record()
            for _ in range(100):
                rc.compact_routes(*args, workspace=ws)
            stop.record()
            stop.synchronize()
            best[i] = min(best[i], start.elapsed_time(stop))
    assert best[0] < 1.3 * best[1], best
    assert rc.poll_status() == 0


@pytest.mark.parametrize("n,requests", [(255, 2), (256, 2), (257, 2), (1, 513)])   # eight groups: 4096 pairs are 512 listed resources
def test_offsets_around_the_gather_that_plans_for_itself(n, requests):
    test_counts_and_tables([1 + i % 3 for i in range(n)], 1, requests, 8)


@pytest.mark.parametrize("mode", [PACKED, PAGED])
@pytest.mark.parametrize("requests", [2, 200])            # three resources of each: 48 pairs, and more than a gather plans for
def test_resources_that_no_request_lists_leave_no_trace(mode, requests):
    """Lists with room before the first request and behind the last, filled with visible resources: the outputs are those of the
    requests' own lists."""
    groups, d = 8, 64
    sh = wl.Shape(groups, groups, d, 1e4, "bf16")
    rc = make_ctx(sh, max_pos=4096)
    rng = np.random.default_rng(requests)
    lens, spare = rng.integers(1, 40, 3 * requests).astype(np.int32), 5
    slot = np.concatenate([[0], np.cumsum(lens)])[:-1].astype(np.int32)
    pool = int(lens.sum())
    k, v = (wl.normal(i, (groups, pool, d), sh.torch_dtype).cuda() for i in (1, 2))
    keep, vis = rng.integers(0, 2, pool).astype(np.uint8), rng.integers(0, 2, (groups, 3 * requests)).astype(np.uint8)
    n_pages = requests * groups * 2 + 1                    # a route has at most 117 rows: two pages of 64
    got = []
    for room in (0, spare):
        wide = lambda a: np.concatenate([a[:room], a, a[-room:]]) if room else a
        ones = np.ones((groups, room), np.uint8)
        cu, idx, length = (torch.full((n,), -7, dtype=torch.int32, device="cuda") for n in (requests * groups + 1, groups * pool, requests * groups))
        rows = (groups * pool, d) if mode == PACKED else (n_pages, 64, d)
        k_out, v_out = (torch.full(rows, -7, dtype=sh.torch_dtype, device="cuda") for _ in range(2))
        table = torch.full((requests * groups, 2), -7, dtype=torch.int32, device="cuda")
        pages = dict(page_table=table, free_pages=dev(np.arange(n_pages, dtype=np.int32))) if mode == PAGED else {}
        rc.compact_routes(k, v, dev(keep), dev((np.arange(requests + 1) * 3 + room).astype(np.int32)), dev(wide(slot)), dev(wide(lens)),
                          dev(np.concatenate([ones, vis, ones], 1)), mode, cu, idx, k_out, v_out, route_len=length,
                          workspace=torch.zeros(rc.compact_workspace_bytes(requests, 3 * requests + 2 * room), dtype=torch.uint8, device="cuda"), **pages)
        got.append((cu, idx, length, k_out, v_out, table))
    assert all(torch.equal(a, b) for a, b in zip(*got)) and rc.poll_status() == 0
