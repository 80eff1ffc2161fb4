"""Split-KV decode at the edges of its page list: items that end exactly on a CTA's
range or span many CTAs, fewer pages than CTAs, one page in all, more items than
threads, empty routes, and the appended token on the first and last row of a page."""
import numpy as np
import pytest
import torch

from oracle import recache_oracle as orc
from paper_2608_19662_b200 import workloads as wl

from pipeline import dev, f64, make_ctx, max_abs

pytestmark = pytest.mark.gpu

PT = wl.PAGE_TOKENS


def _batch(rng, sh, res_rows, hist_rows):
    """Paged decode inputs with the given rows per item: pages shuffled, tables padded with -1."""
    rp, hp = (res_rows + PT - 1) // PT, (hist_rows + PT - 1) // PT
    ids = rng.permutation(int(rp.sum() + hp.sum())).astype(np.int32)
    rt = np.full((len(rp), max(1, int(rp.max()))), -1, np.int32)
    ht = np.full((len(hp), max(1, int(hp.max()))), -1, np.int32)
    c = 0
    for it in range(len(rp)):
        rt[it, :rp[it]] = ids[c:c + rp[it]]; c += int(rp[it])
        ht[it, :hp[it]] = ids[c:c + hp[it]]; c += int(hp[it])
    seed = int(rng.integers(1 << 30))
    kp = wl.normal(seed, (len(ids), PT, sh.head_dim), sh.torch_dtype)
    vp = wl.normal(seed + 1, (len(ids), PT, sh.head_dim), sh.torch_dtype)
    return kp, vp, rt, ht


@pytest.mark.parametrize("hq,groups,batch,res,hist", [
    (32, 8, 1, (0, 0), (1, 1)),          # one page per item, empty routes: 8 pages for 148 CTAs
    (8, 1, 1, (0, 0), (1, 1)),           # one page in all
    (4, 1, 1, (700, 700), (64 * 140, 64 * 140)),   # one item spread over every CTA
    (8, 1, 3, (63, 65), (64, 65)),       # page edges, eight heads per group
    (2, 2, 5, (1, 130), (127, 129)),     # one head per group
    (16, 8, 40, (0, 200), (1, 700)),     # ragged: 320 items, ranges that begin and end inside items
    (8, 8, 70, (0, 64), (1, 64)),        # more items than CTAs and threads, one or two pages each
    (8, 8, 80, (0, 64), (1, 130)),       # 640 items: more than four a CTA, appended by a launch of their own
])
def test_ragged_pages_match_oracle_and_append(hq, groups, batch, res, hist):
    sh = wl.Shape(hq, groups, 128, 1e6, "bf16")
    rng = np.random.default_rng([hq, batch, res[1]])
    items = batch * groups
    res_rows = rng.integers(res[0], res[1] + 1, items).astype(np.int32)
    hist_rows = np.repeat(rng.integers(hist[0], hist[1] + 1, batch), groups).astype(np.int32)
    kp, vp, rt, ht = _batch(rng, sh, res_rows, hist_rows)
    rc = make_ctx(sh, max_pos=16384)
    q, kn, vn = (wl.normal(900 + i, (batch, h, 128), sh.torch_dtype) for i, h in enumerate((hq, groups, groups)))
    q_pos = (np.arange(batch) * 7 + 3).astype(np.int32)
    d_kp, d_vp = dev(kp), dev(vp)
    o = rc.attend_decode(dev(q), dev(q_pos), d_kp, d_vp, dev(rt), dev(res_rows), dev(ht), dev(hist_rows), k_new=dev(kn),
                         v_new=dev(vn), out_dtype=torch.float32)
    kr, vr = f64(kp), f64(vp)
    orc.append_decode_kv(kr, vr, ht, hist_rows, f64(kn), f64(vn), q_pos, sh.rope_theta, PT, storage=sh.dtype)
    ref = orc.attend_decode(f64(q), q_pos, kr, vr, rt, res_rows, ht, hist_rows, sh.rope_theta, PT, storage=sh.dtype)
    assert max_abs(o, ref) < 1e-2
    # the append writes one row per item and nothing else
    assert torch.equal(d_vp.cpu().view(torch.int16), torch.from_numpy(vr).to(torch.bfloat16).view(torch.int16))
    changed = (d_kp.cpu().view(torch.int16) != kp.view(torch.int16)).any(-1).sum().item()
    assert changed == items
    assert max_abs(d_kp, kr) < 4e-2          # 1 bf16 ulp of a key in [4, 8): 3.1e-2
    many = items > 4 * torch.cuda.get_device_properties(0).multi_processor_count
    assert rc.kernel_times()["decode_append"][1] == int(many)
    assert rc.poll_status() == 0


@pytest.mark.parametrize("hq,groups,batch,res,hist", [
    (32, 8, 1, (500, 900), (2000, 2000)),     # one sequence: CTAs of its own for every item
    (8, 1, 1, (0, 0), (64 * 200, 64 * 200)),  # more pages than CTAs in one item
    (8, 2, 1, (1, 70), (1, 1)),               # fewer pages than an item has CTAs
    (16, 8, 4, (100, 400), (64, 3000)),       # few items of very different length
    (16, 8, 16, (0, 900), (1, 2000)),         # gathered and paged pages mixed in a CTA's range
])
def test_gathered_rows_match_paged(hq, groups, batch, res, hist):
    """The zero-copy decode over the rows of a pool equals the paged one over the same rows in pages, bit for bit:
    with tables of the same width both deal their pages out alike."""
    sh = wl.Shape(hq, groups, 128, 1e6, "bf16")
    rng = np.random.default_rng([hq, batch, res[1], 7])
    items = batch * groups
    res_rows = rng.integers(res[0], res[1] + 1, items).astype(np.int32)
    hist_rows = np.repeat(rng.integers(hist[0], hist[1] + 1, batch), groups).astype(np.int32)
    kp, vp, rt, ht = _batch(rng, sh, res_rows, hist_rows)
    pool = max(1, int(res_rows.max()) * 3)
    kc, vc = wl.normal(11, (groups, pool, 128), sh.torch_dtype), wl.normal(12, (groups, pool, 128), sh.torch_dtype)
    cu = np.concatenate([[0], np.cumsum(res_rows)]).astype(np.int32)
    idx = np.concatenate([rng.permutation(pool)[:n] for n in res_rows] + [np.zeros(1, np.int64)]).astype(np.int32)
    for it in range(items):                   # the same rows, in the item's pages
        for n in range(int(res_rows[it])):
            page, r = rt[it, n // PT], n % PT
            kp[page, r], vp[page, r] = kc[it % groups, idx[cu[it] + n]], vc[it % groups, idx[cu[it] + n]]
    rc = make_ctx(sh, max_pos=16384)
    q = wl.normal(900, (batch, hq, 128), sh.torch_dtype)
    q_pos = (np.arange(batch) * 7 + 3).astype(np.int32)
    paged = rc.attend_decode(dev(q), dev(q_pos), dev(kp), dev(vp), dev(rt), dev(res_rows), dev(ht), dev(hist_rows), out_dtype=torch.float32)
    gathered = rc.attend_decode_gather(dev(q), dev(q_pos), dev(kc), dev(vc), dev(idx), dev(cu), rt.shape[1], dev(kp), dev(vp), dev(ht),
                                       dev(hist_rows), out_dtype=torch.float32)
    ref = orc.attend_decode(f64(q), q_pos, f64(kp), f64(vp), rt, res_rows, ht, hist_rows, sh.rope_theta, PT, storage=sh.dtype)
    assert max_abs(paged, ref) < 1e-2 and torch.equal(paged, gathered)
    assert rc.poll_status() == 0


@pytest.mark.parametrize("gather", [False, True])
def test_one_sequence_right_behind_other_kernels(gather):
    """A step of one sequence (whose blocks go straight to their roles) gives the same bits every time, whatever
    the kernels before it left in shared memory, where its barriers are set up."""
    sh = wl.Shape(8, 2, 128, 1e6, "bf16")
    rng = np.random.default_rng(31)
    rows = lambda n, lo, hi: rng.integers(lo, hi + 1, n).astype(np.int32)
    rc = make_ctx(sh, max_pos=4096)
    steps = []
    for batch in (1, 12):
        res, hist = rows(2 * batch, 100, 900), np.repeat(rows(batch, 1, 1500), 2)
        kp, vp, rt, ht = _batch(rng, sh, res, hist)
        q, pos = dev(wl.normal(batch, (batch, 8, 128), sh.torch_dtype)), dev(np.arange(batch, dtype=np.int32) + 9)
        pages, tail = (dev(kp), dev(vp)), (dev(ht), dev(hist))
        if gather:
            cu = np.concatenate([[0], np.cumsum(res)]).astype(np.int32)
            cache = [dev(wl.normal(40 + i, (2, 900, 128), sh.torch_dtype)) for i in range(2)]
            idx = dev(np.concatenate([rng.permutation(900)[:n] for n in res]).astype(np.int32))
            steps.append(lambda a=(q, pos, *cache, idx, dev(cu), rt.shape[1], *pages, *tail): rc.attend_decode_gather(*a))
        else:
            steps.append(lambda a=(q, pos, *pages, dev(rt), dev(res), *tail): rc.attend_decode(*a))
    first = steps[0]()
    got = [(steps[1](), steps[0]())[1] for _ in range(30)]
    assert all(torch.equal(first, x) for x in got)
    assert rc.poll_status() == 0
