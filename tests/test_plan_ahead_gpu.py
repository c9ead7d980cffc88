"""The CTAs of a small batch plan and prefetch before the work in front of them on the stream is done, from the lengths, ranges and
tables as they lie there then.  Work queued in front changes all three, with no synchronisation: the results are those of the new
ones, bit for bit; and the combine kernel of such calls, at part counts around its groups and its limit of one row per SM."""
import numpy as np
import pytest

from paper_2609_37626_b200 import workloads as W
from _util import compare, oracle_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kv_dtype,H,lens", [(0, 16, [200, 3, 256, 70]), (0, 16, [5000, 64, 900]), (0, 32, [3000, 1, 40]), (1, 16, [9000, 130, 65]),
                                             (1, 16, [17, 256]), (1, 128, [1, 255, 64])])
def test_lengths_ranges_and_table_change_under_the_call_before(kv_dtype, H, lens):
    import torch
    from paper_2609_37626_b200 import binding
    from test_inputs_written_in_front_gpu import Arena, ints
    w = W.make_workload("ahead", 8300 + H + len(lens), lens, H=H, kv_dtype=kv_dtype)
    dw = binding.DeviceWorkload(w)
    rng = np.random.default_rng(7)
    versions = []
    for v in range(4):
        keep = np.array([rng.integers(0, n + 1) for n in lens], np.int32) if v else np.array(lens, np.int32)
        begin = np.array([rng.integers(0, max(1, k // 2)) for k in keep], np.int32) if v else np.zeros(len(lens), np.int32)
        versions.append(dict(lens=ints(keep), begin=ints(begin), table=dw.block_table))
    versions.append(dict(versions[0], table=torch.full_like(dw.block_table, -1)))       # what a call that plans ahead may find
    a = Arena(versions)
    call = lambda: binding.splash_mla_decode(dw.q, dw.kv_pool, a.view("table"), a.view("lens"), softmax_scale=w.softmax_scale,
                                             kv_scales=dw.kv_scales, kv_begin=a.view("begin"))
    want = []
    for v in range(4):
        a.put(v)
        torch.cuda.synchronize()
        want.append([t.clone() for t in call()])
    torch.cuda.synchronize()
    got = []
    for r in range(12):
        a.put(4)
        call()
        a.put(r % 4)            # the library's own move: it lets the next call in before its last stores, which are these
        got.append([t.clone() for t in call()])
    torch.cuda.synchronize()
    for r, (o, l) in enumerate(got):
        assert torch.equal(o, want[r % 4][0]) and torch.equal(l, want[r % 4][1]), r


@pytest.mark.parametrize("kv_dtype,H", [(0, 16), (1, 16), (0, 128), (1, 74), (0, 74)])      # one row per SM is 148
@pytest.mark.parametrize("lens", [[64 * 5], [64 * 16, 64], [64 * 17], [64 * 400 + 1]])
def test_combine_of_few_rows(kv_dtype, H, lens):
    import torch
    from paper_2609_37626_b200 import binding
    w = W.make_workload("few", 8400 + H + lens[0], lens, H=H, kv_dtype=kv_dtype)
    out, lse = binding.DeviceWorkload(w).decode()
    torch.cuda.synchronize()
    compare(out.cpu().numpy(), lse.cpu().numpy(), *oracle_run(w), kv_dtype=kv_dtype)
