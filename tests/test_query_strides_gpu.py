"""The query rows of the e4m3 pair kernel (33 heads and more, or several rows per request) arrive by TMA, or are copied by its warps where
the strides are none that a tensor map can state (one query for all requests, a stride of 0): the same bits either way, for slices that end
inside a group of eight heads, rows of zeros and rows whose largest value is in any chunk.  (Up to 32 heads there is one way only.)"""
import numpy as np
import pytest

from paper_2609_37626_b200 import workloads as W
from _util import compare, oracle_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,hb,he", [(16, 0, 16), (16, 3, 12), (32, 0, 32), (40, 9, 38), (64, 0, 64), (100, 30, 73), (128, 0, 128), (128, 5, 94)])
def test_one_query_for_all_requests(H, hb, he):
    import torch
    from paper_2609_37626_b200 import binding as B
    lens = [70, 1, 700, 64 * 9]
    w = W.make_workload("qs", 9500 + H + he, lens, H=H, head_begin=hb, head_end=he, kv_dtype=1)
    dw = B.DeviceWorkload(w)
    one = dw.q[1].clone()
    for r in range(hb, he):                     # the largest value of a row in every chunk in turn
        one[r, (r % 9) * 64 + r % 64] = 9.0 if r % 2 else -9.0
    one[hb] = 0
    apart = one[None].expand(len(lens), H, 576)
    assert apart.stride(0) == 0
    args = (dw.kv_pool, dw.block_table, dw.seq_lens)
    kw = dict(softmax_scale=w.softmax_scale, kv_scales=dw.kv_scales, head_begin=hb, head_end=he)
    whole = B.splash_mla_decode(apart.contiguous(), *args, **kw)
    whole = (whole[0][:, hb:he].clone(), whole[1][:, hb:he].clone())
    shared = B.splash_mla_decode(apart, *args, **kw)
    assert torch.equal(whole[0], shared[0][:, hb:he]) and torch.equal(whole[1], shared[1][:, hb:he])
    w.q = apart.contiguous().view(torch.uint16).cpu().numpy()
    compare(np.pad(whole[0].cpu().numpy(), ((0, 0), (hb, H - he), (0, 0))), np.pad(whole[1].cpu().numpy(), ((0, 0), (hb, H - he))), *oracle_run(w),
            kv_dtype=1, rows=[(i, g) for i in range(len(lens)) for g in range(hb, he)])


@pytest.mark.parametrize("H,hb,he,R", [(16, 0, 16, 3), (24, 5, 16, 5), (48, 0, 48, 8), (128, 0, 128, 2), (128, 3, 100, 5)])
def test_several_rows_per_request(H, hb, he, R):
    """Virtual heads, up to five CTA pairs a worker, the last of them with few heads or none in its second CTA."""
    import torch
    from paper_2609_37626_b200 import binding as B
    lens = [70, R, 700, 64 * 9]
    w = W.make_workload("qs_rows", 9600 + H + he, lens, H=H, head_begin=hb, head_end=he, kv_dtype=1)
    dw = B.DeviceWorkload(w)
    one = torch.randn((1, H, R, 576), generator=torch.Generator("cuda").manual_seed(he), device="cuda").to(torch.bfloat16)
    apart = one.expand(len(lens), H, R, 576)
    args = (dw.kv_pool, dw.block_table, dw.seq_lens)
    kw = dict(softmax_scale=w.softmax_scale, kv_scales=dw.kv_scales, head_begin=hb, head_end=he)
    whole = B.splash_mla_decode(apart.contiguous(), *args, **kw)
    whole = (whole[0][:, hb:he].clone(), whole[1][:, hb:he].clone())
    shared = B.splash_mla_decode(apart, *args, **kw)
    assert torch.equal(whole[0], shared[0][:, hb:he]) and torch.equal(whole[1], shared[1][:, hb:he])
