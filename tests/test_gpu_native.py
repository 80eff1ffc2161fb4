"""The native entry points take the same arguments as ever: optional outputs and workspaces, positional
and keyword forms, and the same errors for what they cannot take."""
import numpy as np
import pytest
import torch

from paper_2608_19662_b200 import ReCacheError
from paper_2608_19662_b200 import workloads as wl

from pipeline import dev, make_ctx

pytestmark = pytest.mark.gpu


def test_arguments_and_errors():
    sh = wl.QWEN3_4B
    pool = wl.pack_resources(sh, 3, [70, 9], [np.ones(70, np.uint8), np.ones(9, np.uint8)])
    rc = make_ctx(sh, max_pos=256)
    q, k, v, cu, slot = (dev(x) for x in (pool.q, pool.k, pool.v, pool.cu_seqlens, pool.dst_slot))
    kc = torch.zeros((sh.n_kv_heads, pool.pool_tokens, sh.head_dim), dtype=sh.torch_dtype, device="cuda")
    vc = torch.zeros_like(kc)
    a = rc.encode_resources(q, k, v, cu, np.int64(70), slot, kc, vc)              # numpy sizes
    assert a.dtype == torch.bfloat16 and a.shape == q.shape
    out = torch.empty_like(q)
    ws = torch.empty(rc.encode_workspace_bytes(2, 79, 70), dtype=torch.uint8, device="cuda")
    b = rc.encode_resources(q, k, v, cu, 70, dst_slot=slot, k_cache=kc, v_cache=vc, out=out, workspace=ws)
    assert b is out and torch.equal(a, b)                                         # the given tensor itself comes back
    assert rc.encode_resources(q, k, v, cu, 70, slot, kc, vc, out_dtype=torch.float32).dtype == torch.float32
    with pytest.raises(AssertionError):
        rc.encode_resources(q.cpu(), k, v, cu, 70, slot, kc, vc)
    with pytest.raises(AssertionError):
        rc.encode_resources(q.transpose(0, 1), k, v, cu, 70, slot, kc, vc)
    with pytest.raises(TypeError):
        rc.encode_resources(None, k, v, cu, 70, slot, kc, vc)
    with pytest.raises(ReCacheError, match="workspace too small"):
        rc.encode_resources(q, k, v, cu, 70, slot, kc, vc, workspace=ws[:16])
    with pytest.raises(ReCacheError, match="max_pos"):
        rc.encode_resources(q, k, v, cu, 300, slot, kc, vc)
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(other):                                                # the current stream is the one used
        c = rc.encode_resources(q, k, v, cu, 70, slot, kc, vc)
    other.synchronize()
    assert torch.equal(a, c) and rc.poll_status() == 0
    rc.close()
    with pytest.raises(Exception):
        rc.encode_resources(q, k, v, cu, 70, slot, kc, vc)


def test_out_of_memory_is_torchs_own_error():
    """The output's allocation fails with the error type that a program catches to free memory and try again."""
    sh = wl.QWEN3_4B
    rc = make_ctx(sh, max_pos=8192)
    q = torch.zeros((8192, sh.n_q_heads, sh.head_dim), dtype=sh.torch_dtype, device="cuda")
    k = torch.zeros((8192, sh.n_kv_heads, sh.head_dim), dtype=sh.torch_dtype, device="cuda")
    cache, cu, slot = k.transpose(0, 1).contiguous(), dev(np.array([0, 8192], np.int32)), dev(np.zeros(1, np.int32))
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    try:
        torch.cuda.set_per_process_memory_fraction(torch.cuda.memory_reserved() / torch.cuda.get_device_properties(0).total_memory)
        with pytest.raises(torch.OutOfMemoryError):
            rc.encode_resources(q, k, k, cu, 8192, slot, cache, cache)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert rc.encode_resources(q, k, k, cu, 8192, slot, cache, cache.clone()).shape == q.shape and rc.poll_status() == 0
