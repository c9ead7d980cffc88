"""Scratch of a sparse call: what the decode needs, and the gathered cache only where a kernel gathers into it (SPLASH_FLAG_SIMT).  The call
stays inside what the size function names: the bytes behind it keep their pattern."""
import numpy as np
import pytest

import oracle
from paper_2609_37626_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [16, 128])
@pytest.mark.parametrize("simt", [False, True])
def test_size_and_bounds(H, simt):
    import torch
    from paper_2609_37626_b200 import binding
    B, K = 40, 300
    w = W.make_workload("scratch", 8800 + H, [500] * B, H=H, kv_dtype=2)
    sel, cnt = W.select_tokens(8800 + H, w.seq_lens, K)
    dw = binding.DeviceWorkload(w)
    out, lse = torch.empty((B, H, 512), device="cuda"), torch.empty((B, H), device="cuda")
    flags = binding.SPLASH_FLAG_SIMT if simt else 0
    size = lambda f: binding.splash_mla_decode_sparse_workspace_bytes(binding.make_shape(dw.q, dw.kv_pool, dw.block_table, out, lse, w.softmax_scale, f), K, 0, H)
    need = size(flags)
    assert size(binding.SPLASH_FLAG_SIMT) - size(0) >= B * ((K + 63) // 64) * 64 * 1152
    guard = torch.full((need + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    call = lambda ws: binding.splash_mla_decode_sparse(dw.q, dw.kv_pool, dw.block_table, dw.seq_lens, torch.from_numpy(sel).cuda(), torch.from_numpy(cnt).cuda(),
                                                       softmax_scale=w.softmax_scale, flags=flags, workspace=ws)
    o, l = call(guard[:need])
    torch.cuda.synchronize()
    assert (guard[need:] == 0xA5).all()
    ref = oracle.mla_decode_sparse(w.q, w.kv_pool, w.block_table, w.seq_lens, sel, cnt, softmax_scale=w.softmax_scale)
    assert np.abs(o.cpu().numpy() - ref[0]).max() <= 5e-2 and np.abs(l.cpu().numpy() - ref[1]).max() <= 2e-2
    with pytest.raises(binding.SplashError):
        call(guard[:need - 256])


def test_size_does_not_grow_with_the_lists():
    import torch
    from paper_2609_37626_b200 import binding
    q, kv = torch.empty((64, 128, 576), dtype=torch.bfloat16, device="cuda"), torch.empty((4, 64, 656), dtype=torch.uint8, device="cuda")
    out, lse, table = torch.empty((64, 128, 512), device="cuda"), torch.empty((64, 128), device="cuda"), torch.zeros((64, 4), dtype=torch.int32, device="cuda")
    shape = binding.make_shape(q, kv, table, out, lse, 0.07)
    assert binding.splash_mla_decode_sparse_workspace_bytes(shape, 64, 0, 128) == binding.splash_mla_decode_sparse_workspace_bytes(shape, 2048, 0, 128)
