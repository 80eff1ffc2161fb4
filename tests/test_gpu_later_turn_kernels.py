"""Which attention a later turn runs: items of one query tile (attn_tile.cu) where it has few or where no request has a
second tile, pairs of tiles (attn_tc.cu) where it has many, or many keys each; and that the result is the same bits
whichever it is, as the choice may follow from the room of a cache."""
import numpy as np
import pytest
import torch

from paper_2608_19662_b200 import workloads as wl

from pipeline import dev, kernels_of, make_ctx

pytestmark = pytest.mark.gpu

ROOM = 40 * 128       # rows of a cache with room for 40 K/V tiles a request


def _turn(hq, batch, new, hist, room):
    """A later turn of `batch` requests, in a cache of `room` rows for each; the result and the kernel that computed it."""
    g, d = 8, 128
    sh = wl.Shape(hq, g, d, 1e6, "bf16")
    rc = make_ctx(sh, max_pos=8192)
    N = lambda i, *s: dev(wl.normal(800 + i, s, sh.torch_dtype))
    n = batch * new
    q, k, v = (N(0, n, hq, d).float() * 8).to(sh.torch_dtype), N(1, n, g, d), N(2, n, g, d)     # (a spread that makes rows rescale their sums)
    kc, vc = (torch.full((g, batch * room, d), float("nan"), dtype=sh.torch_dtype, device="cuda") for _ in range(2))
    for i, c in ((3, kc), (4, vc)):
        c.view(g, batch, room, d)[:, :, :hist] = N(i, g, batch, hist, d)
    step = dev(np.arange(batch + 1, dtype=np.int32))
    hist_len = torch.full((batch,), hist, dtype=torch.int32, device="cuda")
    none = torch.zeros(batch * g + 1, dtype=torch.int32, device="cuda")
    rows = N(5, 1, d)
    run = lambda: rc.attend_prefill_history(q, k, v, step * new, hist_len, new, rows, rows, none, kc, vc, step[:-1] * room, hist_len)
    o, names = kernels_of(run)
    assert ("attn_tile_kernel" in names) != ("attn_tc_kernel" in names)
    assert rc.poll_status() == 0
    return o, "tile" if "attn_tile_kernel" in names else "pair"


# eight groups: three rounds of CTAs are 444 work items of 128 rows on 148 SMs, eight are 1184
@pytest.mark.parametrize("hq,batch,new,hist,tight,roomy", [
    (16, 6, 512, 200, "tile", "tile"),       # 2 heads: 432 items, three rounds
    (16, 7, 512, 200, "tile", "pair"),       # 504: by the room, which only the time follows from
    (32, 7, 256, 4000, "pair", "pair"),      # 504 of 33 K/V tiles
    (32, 16, 256, 100, "tile", "pair"),      # 1152
    (64, 17, 128, 100, "pair", "pair"),      # 1224: more than eight rounds
    (16, 80, 64, 100, "tile", "tile"),       # 1280, but no request has a second query tile
    (32, 50, 64, 100, "pair", "pair"),       # 1200, of requests that have one
])
def test_kernel_and_bits_on_both_sides(hq, batch, new, hist, tight, roomy):
    rooms = ((hist + new + 63) // 64 * 64, max(ROOM, hist + new))
    (a, ka), (b, kb) = (_turn(hq, batch, new, hist, r) for r in rooms)
    assert (ka, kb) == (tight, roomy)
    assert torch.equal(a, b) and torch.isfinite(a).all()
