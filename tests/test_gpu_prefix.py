"""Encoding behind a shared prefix and with global position offsets (the
"Block" ablation) on the GPU against the oracle, fp32 and bf16 paths."""
import numpy as np
import pytest
import torch

from oracle import recache_oracle as orc
from paper_2608_19662_b200 import workloads as wl

from pipeline import dev, f64, kernels_of, make_ctx, max_abs
from test_gpu_parity import assert_rotated_close

pytestmark = pytest.mark.gpu


def _case(sh, lens, P, seed):
    rng = np.random.default_rng(seed)
    pool = wl.pack_resources(sh, seed, lens, wl.keep_mask_spans(rng, lens), slot_gap=3)
    _, kp, vp = wl.resource_tensors(seed, 900, P, sh)
    return pool, kp, vp


@pytest.mark.parametrize("shape,tol,lens,P", [
    (wl.TINY_F32, 1e-5, [17, 40, 23], 9),
    (wl.QWEN3_4B, 1e-2, [130, 64, 257, 33, 200], 150),      # prefix longer than one key tile
    (wl.Shape(16, 8, 128, 1e6, "bf16"), 1e-2, [70, 190], 37),
])
def test_prefixed_and_block_encode(shape, tol, lens, P):
    sh = shape
    pool, kp, vp = _case(sh, lens, P, 41)
    rc = make_ctx(sh, max_pos=4096)
    g, d = sh.n_kv_heads, sh.head_dim
    # the prefix as a cache holds it: keys rotated at 0..P-1 in the storage dtype (from the oracle)
    pk = orc.round_storage(np.transpose(orc.rope(f64(kp), np.arange(P), sh.rope_theta), (1, 0, 2)), sh.dtype)
    pv = np.transpose(f64(vp), (1, 0, 2))
    pk_d, pv_d = dev(pk).to(sh.torch_dtype).contiguous(), dev(pv).to(sh.torch_dtype).contiguous()
    for name, offs in (("local", [P] * len(lens)), ("block", [P + int(c) for c in pool.cu_seqlens[:-1]])):
        ref_o, ref_k, ref_v = orc.encode_resources(f64(pool.q), f64(pool.k), f64(pool.v), pool.cu_seqlens, sh.rope_theta,
                                                   storage=sh.dtype, pos_offset=offs, prefix_k=pk, prefix_v=pv)
        kc = torch.full((g, pool.pool_tokens, d), float("nan"), dtype=sh.torch_dtype, device="cuda")
        vc = torch.full_like(kc, float("nan"))
        o = rc.encode_resources_prefixed(dev(pool.q), dev(pool.k), dev(pool.v), dev(pool.cu_seqlens), pool.max_len,
                                         dev(pool.dst_slot), kc, vc, k_prefix=pk_d, v_prefix=pv_d,
                                         pos_offset=dev(np.asarray(offs, np.int32)), out_dtype=torch.float32)
        assert max_abs(o, ref_o) < tol, name
        kc_ref = np.full((g, pool.pool_tokens, d), np.nan); vc_ref = np.full_like(kc_ref, np.nan)
        orc.write_cache(kc_ref, vc_ref, ref_k, ref_v, pool.cu_seqlens, pool.dst_slot)
        written = ~np.isnan(kc_ref)
        assert np.array_equal(np.isnan(f64(kc)), ~written)
        assert_rotated_close(sh, kc, np.where(written, kc_ref, 0.0), written)
    # no prefix, no offsets: the extended call is the plain one, bit for bit
    kc1 = torch.zeros((g, pool.pool_tokens, d), dtype=sh.torch_dtype, device="cuda"); vc1 = torch.zeros_like(kc1)
    kc2, vc2 = torch.zeros_like(kc1), torch.zeros_like(kc1)
    a = rc.encode_resources(dev(pool.q), dev(pool.k), dev(pool.v), dev(pool.cu_seqlens), pool.max_len, dev(pool.dst_slot), kc1, vc1)
    b = rc.encode_resources_prefixed(dev(pool.q), dev(pool.k), dev(pool.v), dev(pool.cu_seqlens), pool.max_len,
                                     dev(pool.dst_slot), kc2, vc2)
    assert torch.equal(a, b) and torch.equal(kc1, kc2)
    assert rc.poll_status() == 0


# 148 SMs, eight groups: up to 8 K/V tiles of prefix 888 work items of 128 rows are encoded one by one, up to 32 tiles 444, beyond 148
@pytest.mark.parametrize("hq,prefix,most", [(16, 150, 888), (32, 1024, 888), (64, 1025, 444), (16, 4096, 444), (32, 4097, 148), (64, 6000, 148)])
def test_kernel_and_bits_on_both_sides(hq, prefix, most):
    """A resource encoded with as many others as fit under the limit, and with one more: by the kernel with a tile to an item and by the
    one with pairs, to the same bits.  Queries times eight: rows rescale their sums several times on the way."""
    g, d = 8, 128
    sh = wl.Shape(hq, g, d, 1e6, "bf16")
    rc = make_ctx(sh, max_pos=16384)
    N = lambda i, *s: dev(wl.normal(60 + i, s, sh.torch_dtype))
    kp, vp = N(3, g, prefix, d), N(4, g, prefix, d)
    tile = 128 // (hq // g)
    first, fit = 2 * tile + 5, (most // g - 2) * tile      # two resources: items = tokens / tile + 2, for each group
    all_q, all_k, all_v = ((N(i, fit + tile, h, d).float() * f).to(sh.torch_dtype) for i, h, f in ((0, hq, 8), (1, g, 1), (2, g, 1)))
    got = []
    for n in (fit, fit + tile):
        cu, q, k, v = dev(np.array([0, first, n], np.int32)), all_q[:n], all_k[:n], all_v[:n]
        kc, vc = (torch.zeros((g, n, d), dtype=sh.torch_dtype, device="cuda") for _ in range(2))
        run = lambda: rc.encode_resources_prefixed(q, k, v, cu, n, cu[:2], kc, vc, k_prefix=kp, v_prefix=vp,
                                                   pos_offset=torch.full((2,), prefix, dtype=torch.int32, device="cuda"))
        o, names = kernels_of(run)
        got.append((o[:first], names))
    assert "attn_tile_kernel" in got[0][1] and "attn_tc_kernel" in got[1][1]
    assert torch.equal(got[0][0], got[1][0]) and torch.isfinite(got[0][0]).all()
    assert rc.poll_status() == 0
