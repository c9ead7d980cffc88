"""The 64-head group of the one-CTA bf16 kernel turns its output over in blocks of sixteen heads by 32 columns: head counts at the
edges of a block and of the four rows a store writes, slices inside wider buffers, whole requests and pieces, dense and sparse."""
import numpy as np
import pytest

import oracle
from paper_2609_37626_b200 import workloads as W
from _util import TOL, compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,hb,he", [(33, 0, 33), (48, 0, 48), (49, 0, 49), (64, 0, 64), (128, 3, 66), (128, 65, 128)])
@pytest.mark.parametrize("lens", [[1, 64, 65, 0], [1500, 3]])
def test_head_counts(H, hb, he, lens):
    w = W.make_workload("wide", 9100 + H + he + len(lens), lens, H=H, head_begin=hb, head_end=he)
    out, lse = gpu_run(w, sentinel=7.0)
    compare(out, lse, *oracle_run(w), kv_dtype=0, rows=[(i, g) for i in range(len(lens)) for g in range(hb, he)])
    mask = np.ones(H, bool)
    mask[hb:he] = False
    assert np.all(out[:, mask] == 7.0) and np.all(lse[:, mask] == 7.0)


@pytest.mark.parametrize("H", [35, 64])
def test_sparse(H):
    import torch
    from paper_2609_37626_b200 import binding
    w = W.make_workload("wide_sparse", 9200 + H, [300, 40, 130], H=H, kv_dtype=2)
    sel, cnt = W.select_tokens(9200 + H, w.seq_lens, 200)
    dw = binding.DeviceWorkload(w, "cuda:0")
    out, lse = binding.splash_mla_decode_sparse(dw.q, dw.kv_pool, dw.block_table, dw.seq_lens, torch.from_numpy(sel).cuda(),
                                                torch.from_numpy(cnt).cuda(), softmax_scale=w.softmax_scale)
    ref_o, ref_l = oracle.mla_decode_sparse(w.q, w.kv_pool, w.block_table, w.seq_lens, sel, cnt, softmax_scale=w.softmax_scale)
    assert np.abs(out.cpu().numpy() - ref_o).max() <= TOL[1]["abs_o"]
    assert np.abs(lse.cpu().numpy() - ref_l).max() <= TOL[1]["lse"]
