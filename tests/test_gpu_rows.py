"""The exact-arithmetic attention at the edges of its blocks: sequences one token around a block of
query rows and around the key tiles of a full round of warps, every number of heads per group."""
import numpy as np
import pytest
import torch

from paper_2608_19662_b200 import workloads as wl

from pipeline import dev, gpu_compact, gpu_encode, gpu_prefill, make_ctx, max_abs, oracle_encode, oracle_prefill, oracle_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,g,d,dtype,tol", [
    (2, 2, 64, "f32", 1e-5), (4, 2, 64, "f32", 1e-5), (6, 2, 64, "f32", 1e-5), (5, 1, 64, "f32", 1e-5), (8, 1, 64, "f32", 1e-5),
    (2, 2, 128, "f32", 1e-5), (3, 1, 128, "f32", 1e-5), (7, 1, 128, "f32", 1e-5), (8, 1, 128, "f32", 1e-5),
    (4, 2, 64, "bf16", 1e-2), (3, 3, 128, "bf16", 1e-2),
])
def test_block_edges(hq, g, d, dtype, tol):
    sh = wl.Shape(hq, g, d, 1e4, dtype)
    rng = np.random.default_rng([hq, g, d])
    lens = [1, 15, 16, 17, 0, 31, 33, 255, 257, 290]
    pool = wl.pack_resources(sh, hq * 100 + d, lens, [rng.integers(0, 2, n).astype(np.uint8) for n in lens])
    rc = make_ctx(sh, max_pos=1024)
    o, kc, vc = gpu_encode(rc, pool)
    ref, kc_ref, vc_ref = oracle_encode(pool)
    assert max_abs(o, ref) < tol
    lists = [[9, 1], [], [3, 4, 7, 8]]
    vis = [rng.integers(0, 2, (g, len(x))).astype(np.uint8) for x in lists]
    req = wl.make_requests(sh, 7, pool, lists, vis, [17, 40, 3])
    rows = oracle_rows(pool, req)
    out = gpu_compact(rc, pool, req, kc, vc)
    p, _, _ = gpu_prefill(rc, req, out["k_out"], out["v_out"], out["route_cu"])
    p_ref, _ = oracle_prefill(req, rows, kc_ref, vc_ref)
    assert max_abs(p, p_ref) < tol
    assert rc.poll_status() == 0


@pytest.mark.parametrize("hq,g,d,dtype", [(4, 2, 64, "f32"), (8, 1, 128, "f32"), (2, 2, 64, "bf16"), (3, 3, 128, "bf16")])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_values_that_are_not_finite_reach_only_the_rows_that_see_them(hq, g, d, dtype, value):
    sh = wl.Shape(hq, g, d, 1e4, dtype)
    lens, at, col = [290, 45, 9], (100, 44, 2), 5           # the middle of a block, a last token, a short sequence
    pool = wl.pack_resources(sh, 3, lens, [np.ones(n, np.uint8) for n in lens])
    rc = make_ctx(sh, max_pos=1024)
    clean, kc, vc = gpu_encode(rc, pool)
    for i, j in enumerate(at):
        pool.v[int(pool.cu_seqlens[i]) + j, :, col] = value
    o, kc, vc = gpu_encode(rc, pool)
    for i, j in enumerate(at):
        own, want = (x[int(pool.cu_seqlens[i]):int(pool.cu_seqlens[i + 1])] for x in (o, clean))
        assert torch.equal(own[:j], want[:j])                # earlier tokens: as if it were not there
        assert not torch.isfinite(own[j:, :, col]).any() and (value != value or (own[j, :, col] == value).all())
        own[j:, :, col] = want[j:, :, col]
        assert torch.equal(own, want)                        # later ones: that column and no other
    # a route whose last rows (45 of them, not a multiple of the key tile) are the one with that value, then none
    req = wl.make_requests(sh, 7, pool, [[1], []], [np.ones((g, 1), np.uint8), np.ones((g, 0), np.uint8)], [40, 20])
    out = gpu_compact(rc, pool, req, kc, vc)
    p, _, _ = gpu_prefill(rc, req, out["k_out"], out["v_out"], out["route_cu"])
    assert torch.isfinite(p[40:]).all() and not torch.isfinite(p[:40, :, col]).any()
    assert value != value or (p[:40, :, col] == value).all()
    p[:40, :, col] = 0
    assert torch.isfinite(p).all() and rc.poll_status() == 0


@pytest.mark.parametrize("hq,g,d,dtype,tol", [(4, 2, 64, "f32", 1e-5), (32, 8, 128, "f32", 1e-5), (8, 8, 64, "bf16", 1e-2), (5, 1, 128, "bf16", 1e-2)])
def test_many_short_sequences(hq, g, d, dtype, tol):
    """A launch with blocks enough for two warps each: the oracle's results, and for a resource the same bits as
    encoded alone, by eight warps (one of them has more key tiles than there are parts)."""
    sh = wl.Shape(hq, g, d, 1e4, dtype)
    rng = np.random.default_rng(hq)
    lens = rng.integers(0, 40, 700).astype(np.int32)
    lens[[3, 350]] = 290, 65
    pool = wl.pack_resources(sh, 11, lens, [np.ones(int(n), np.uint8) for n in lens], bulk=True)
    rc = make_ctx(sh, max_pos=1024)
    o, kc, vc = gpu_encode(rc, pool)
    ref, _, _ = oracle_encode(pool)
    assert max_abs(o, ref) < tol
    for i in (3, 350, 351):
        a, b = int(pool.cu_seqlens[i]), int(pool.cu_seqlens[i + 1])
        one = torch.zeros((g, max(b - a, 1), d), dtype=sh.torch_dtype, device="cuda")
        alone = rc.encode_resources(dev(pool.q[a:b]), dev(pool.k[a:b]), dev(pool.v[a:b]), dev(np.array([0, b - a], np.int32)), max(b - a, 1),
                                    dev(np.zeros(1, np.int32)), one, one.clone(), out_dtype=torch.float32)
        assert torch.equal(alone, o[a:b])
    assert rc.poll_status() == 0
