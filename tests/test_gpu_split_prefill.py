"""Prefill launches whose items are cut across CTAs: few long items, items that end at a cut, parts that
begin in the route, the history or the causal range, and launches on both sides of the decision."""
import numpy as np
import pytest
import torch

from oracle import recache_oracle as orc
from paper_2608_19662_b200 import workloads as wl

from pipeline import dev, f64, make_ctx, max_abs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,g,lens,hist,route,out", [
    (8, 2, [5], [3000], [(0, 0)], torch.float32),                    # two items over all CTAs, no route
    (4, 1, [70, 1], [1900, 640], [(2500, 2500), (129, 129)], torch.bfloat16),   # parts inside the route
    (8, 1, [33, 40], [1281, 0], [(0, 700), (4000, 4000)], torch.float32),       # eight heads; an item of route tiles only
    (16, 8, [250, 17, 129], [300, 2048, 1000], [(500, 900)] * 3, torch.float32),   # two heads: pairs of 128 tokens
    (8, 2, [130, 64, 65, 3], [127, 128, 129, 0], [(0, 300)] * 4, torch.float32),   # short: below the decision
    (32, 8, [1100], [0], [(1500, 2600)], torch.bfloat16),            # more items than CTAs, two rounds
    (32, 8, [1290], [0], [(1500, 2600)], torch.float32),             # a second round of CTAs that is nearly empty
])
def test_split_items_match_oracle(hq, g, lens, hist, route, out):
    sh = wl.Shape(hq, g, 128, 1e6, "bf16")
    rng = np.random.default_rng([hq, g, len(lens)])
    B, d = len(lens), 128
    lens, hist = np.asarray(lens), np.asarray(hist)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    n_route = np.concatenate([rng.integers(a, b + 1, g) for a, b in route])
    r_cu = np.concatenate([[0], np.cumsum(n_route)]).astype(np.int32)
    room = (hist + lens + 63) // 64 * 64
    slot = np.concatenate([[0], np.cumsum(room)])
    rows = int(slot[-1])
    N = lambda i, *s: wl.normal(1000 + i, s, sh.torch_dtype)
    q, k, v = N(0, int(cu[-1]), hq, d), N(1, int(cu[-1]), g, d), N(2, int(cu[-1]), g, d)
    kr, vr, kc, vc = N(3, int(r_cu[-1]) + 1, d), N(4, int(r_cu[-1]) + 1, d), N(5, g, rows, d), N(6, g, rows, d)
    pos0 = (hist + 100).astype(np.int32)
    rc = make_ctx(sh, max_pos=8192)
    d_kc, d_vc = dev(kc), dev(vc)
    args = (dev(q), dev(k), dev(v), dev(cu), dev(pos0), int(lens.max()), dev(kr), dev(vr), dev(r_cu))
    tail = (dev(slot[:-1].astype(np.int32)), dev(hist.astype(np.int32)))
    o = rc.attend_prefill_history(*args, d_kc, d_vc, *tail, out_dtype=out)
    again = rc.attend_prefill_history(*args, d_kc, d_vc, *tail, out_dtype=out)
    assert torch.equal(o, again)                                     # the cuts and the merge have a fixed order
    # oracle: route rows by a list of indices into a pool that holds exactly them
    pool_k, pool_v = np.zeros((g, int(r_cu[-1]) + 1, d)), np.zeros((g, int(r_cu[-1]) + 1, d))
    pool_k[:], pool_v[:] = f64(kr)[None], f64(vr)[None]
    lists = [[np.arange(r_cu[b * g + kg], r_cu[b * g + kg + 1]) for kg in range(g)] for b in range(B)]
    hk = [f64(kc)[:, slot[b]:slot[b] + hist[b]] for b in range(B)]
    hv = [f64(vc)[:, slot[b]:slot[b] + hist[b]] for b in range(B)]
    ref, _ = orc.attend_prefill(f64(q), f64(k), f64(v), cu, pos0, lists, pool_k, pool_v, sh.rope_theta, storage=sh.dtype, hist_k=hk, hist_v=hv)
    tol = 1e-2 + (2.0 ** -8 * np.abs(ref) if out == torch.bfloat16 else 0)   # bf16 results: half an ulp on top
    assert (np.abs(f64(o) - ref) <= tol).all()
    assert rc.poll_status() == 0


def _padded(t, n):
    """`t` with n more rows of NaN behind it: a buffer of a larger capacity."""
    return torch.cat([t, torch.full((n, *t.shape[1:]), float("nan"), dtype=t.dtype, device=t.device)])


@pytest.mark.parametrize("hq,g,lens,route", [
    (32, 8, [512], 3000),                 # one round of CTAs, half of them idle
    (32, 8, [1100], 2600),                # two rounds, the second nearly empty
    (8, 1, [33, 40], 3000),               # two requests, items few and long
])
def test_first_turn_does_not_depend_on_capacities(hq, g, lens, route):
    """Packed and gathered rows, in tight buffers and in large ones, and the request alone: the same bits."""
    sh = wl.Shape(hq, g, 128, 1e6, "bf16")
    B, d = len(lens), 128
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    n = np.full(B * g, route)
    r_cu = np.concatenate([[0], np.cumsum(n)]).astype(np.int32)
    N = lambda i, *s: dev(wl.normal(500 + i, s, sh.torch_dtype))
    q, k, v = N(0, int(cu[-1]), hq, d), N(1, int(cu[-1]), g, d), N(2, int(cu[-1]), g, d)
    kc, vc = N(3, g, route + 50, d), N(4, g, route + 50, d)
    rng = np.random.default_rng(route)
    idx = [np.sort(rng.permutation(route + 50)[:route]) for _ in n]
    kr, vr = (torch.cat([c[r % g][dev(x)] for r, x in enumerate(idx)]) for c in (kc, vc))
    idx, pos0 = dev(np.concatenate(idx).astype(np.int32)), np.full(B, 100, np.int32)
    rc = make_ctx(sh, max_pos=8192)

    def packed(extra=0, of=slice(0, B)):
        c, r = cu[of.start:of.stop + 1], r_cu[of.start * g:of.stop * g + 1]
        tok, rows = slice(int(c[0]), int(c[-1])), slice(int(r[0]), int(r[-1]))
        return rc.attend_prefill(q[tok], k[tok], v[tok], dev(c - c[0]), dev(pos0[of]), max(lens), _padded(kr[rows], extra), _padded(vr[rows], extra),
                                 dev(r - r[0]))[0]

    def gathered(extra=0):
        more = torch.zeros(extra, dtype=torch.int32, device="cuda")
        return rc.attend_prefill_gather(q, k, v, dev(cu), dev(pos0), max(lens), kc, vc, torch.cat([idx, more]), dev(r_cu))[0]

    want = packed()
    for got in (packed(9000 * B * g), gathered(), gathered(9000 * B * g), torch.cat([packed(0, slice(b, b + 1)) for b in range(B)])):
        assert torch.equal(want, got)
    assert rc.poll_status() == 0


def test_later_turn_does_not_depend_on_capacities():
    """One long history among short ones, in a tight cache and in one with room: the same bits."""
    sh = wl.Shape(8, 2, 128, 1e6, "bf16")
    hist, new = np.array([3000, 0, 0, 0], np.int32), 5
    N = lambda i, *s: dev(wl.normal(600 + i, s, sh.torch_dtype))
    q, k, v = N(0, 4 * new, 8, 128), N(1, 4 * new, 2, 128), N(2, 4 * new, 2, 128)
    slot = np.concatenate([[0], np.cumsum((hist + new + 63) // 64 * 64)]).astype(np.int32)
    kc, vc, rows = N(3, 2, int(slot[-1]), 128), N(4, 2, int(slot[-1]), 128), N(5, 1, 128)
    cu = dev(np.arange(5, dtype=np.int32) * new)
    rc = make_ctx(sh, max_pos=8192)
    got = []
    for extra in (0, 20000):
        caches = [torch.cat([c, torch.full((2, extra, 128), float("nan"), dtype=c.dtype, device="cuda")], 1) for c in (kc, vc)]
        got.append(rc.attend_prefill_history(q, k, v, cu, dev(hist + 9), new, _padded(rows, extra), _padded(rows, extra),
                                             torch.zeros(9, dtype=torch.int32, device="cuda"), *caches, dev(slot[:-1]), dev(hist)))
    assert torch.equal(*got)
    assert rc.poll_status() == 0


def test_one_workspace_serves_the_largest_call_and_all_smaller_ones():
    sh = wl.Shape(32, 8, 128, 1e6, "bf16")
    rc = make_ctx(sh, max_pos=8192)
    sizes = [(b, t, t) for b in (1, 3, 40, 300) for t in (1, 64, 777, 40000) if t >= b]
    for query in (rc.prefill_workspace_bytes, rc.prefill_history_workspace_bytes, rc.encode_workspace_bytes):
        need = {size: query(*size) for size in sizes}
        assert all(need[a] <= need[b] for a in sizes for b in sizes if all(x <= y for x, y in zip(a, b)))
    ws = torch.empty(rc.prefill_workspace_bytes(300, 40000, 40000), dtype=torch.uint8, device="cuda")
    assert rc.prefill_workspace_bytes(1, 512, 512) < 1 << 16 and ws.numel() < 1 << 18      # nothing set aside for parts
    N = lambda i, *s: dev(wl.normal(700 + i, s, sh.torch_dtype))
    new, hist = 40, 2500
    q, k, v, kc, vc = N(0, new, 32, 128), N(1, new, 8, 128), N(2, new, 8, 128), N(3, 8, hist + new, 128), N(4, 8, hist + new, 128)
    rows, cu, pos, none = N(5, 1, 128), dev(np.array([0, new], np.int32)), dev(np.array([hist], np.int32)), torch.zeros(9, dtype=torch.int32, device="cuda")
    turn = lambda **kw: rc.attend_prefill(q, k, v, cu, pos, new, rows, rows, none, **kw)[0]
    later = lambda **kw: rc.attend_prefill_history(q, k, v, cu, pos, new, rows, rows, none, kc, vc, none[:1], pos, out_dtype=torch.float32, **kw)
    assert torch.equal(turn(), turn(workspace=ws))
    whole, parts = later(workspace=ws), later()
    assert rc.poll_status() == 0
    # two orders of summation of the same rows, probabilities in bf16: 2^-9 of each, signs at random over 2500 rows
    assert not torch.equal(whole, parts) and (whole - parts).abs().max().item() < 2e-3


@pytest.mark.parametrize("new,hist,split", [
    ([16], 1904, False),          # eight items of 15 K/V tiles: the merge would take longer than what the parts save
    ([16], 1905, True),           # of 16
    ([16] * 4, 1500, False),
    ([16] * 4, 2500, True),
    ([16] * 19, 1800, False),     # a second round of 4 CTAs; the merge would take as long
    ([1216], 700, False),         # 152 items of 6-15 tiles, short ones last
    ([1216], 3000, True),         # of 24-33
])
def test_split_only_where_it_pays(new, hist, split):
    """With room for parts the bits are those of the undivided call exactly where the call stays undivided (8 groups, 148 SMs)."""
    sh = wl.Shape(16, 8, 128, 1e6, "bf16")
    rc = make_ctx(sh, max_pos=8192)
    B, cu = len(new), np.concatenate([[0], np.cumsum(new)]).astype(np.int32)
    room, n = (hist + max(new) + 63) // 64 * 64, sum(new)
    N = lambda i, *s: dev(wl.normal(900 + i, s, sh.torch_dtype))
    q, k, v, kc, vc, rows = N(0, n, 16, 128), N(1, n, 8, 128), N(2, n, 8, 128), N(3, 8, B * room, 128), N(4, 8, B * room, 128), N(5, 1, 128)
    slot, hists = dev(np.arange(B, dtype=np.int32) * room), dev(np.full(B, hist, np.int32))
    none = torch.zeros(8 * B + 1, dtype=torch.int32, device="cuda")
    later = lambda ws: rc.attend_prefill_history(q, k, v, dev(cu), hists, max(new), rows, rows, none, kc, vc, slot, hists, out_dtype=torch.float32, workspace=ws)
    whole, got = (later(torch.empty(need(B, n, max(new)), dtype=torch.uint8, device="cuda"))
                  for need in (rc.prefill_workspace_bytes, rc.prefill_history_workspace_bytes))
    assert torch.equal(whole, got) != split
    assert (whole - got).abs().max().item() < 2e-3      # two orders of summation, see above
    assert rc.poll_status() == 0
