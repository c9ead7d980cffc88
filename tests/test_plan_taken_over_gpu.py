"""SPLASH_FLAG_REUSE_PLAN does not ask for block tables of one width: the partition that a later layer takes over may have been made by the
plan kernel, or by the decode kernel itself (cut, or a request per worker) behind a narrower table.  e4m3 slices of more than 32
heads read it from the workspace where their own table is wide; every way of making it must have left it there."""
import numpy as np
import pytest

from paper_2609_37626_b200 import workloads as W
from _util import compare, oracle_run

pytestmark = pytest.mark.gpu

NARROW, MEDIUM, WIDE = 0, 300, 9000        # extra columns: none, few, more than 8,192 pages for any batch


@pytest.mark.parametrize("kv_dtype,H", [(1, 48), (1, 128), (0, 128), (1, 16)])
@pytest.mark.parametrize("lens", [[200], [1, 0, 256, 64, 130], [3000, 70, 0, 129, 5000], [250] * 32, [400, 9] * 16])
@pytest.mark.parametrize("first", [NARROW, MEDIUM, WIDE])
def test_tables_of_other_widths(kv_dtype, H, lens, first):
    import torch
    from paper_2609_37626_b200 import binding
    # nothing that earlier calls have left in the shared workspace may help (a partition of zeros has no work in it)
    ws = binding.decode_workspace(torch.device("cuda", 0))
    if ws is not None:
        ws.zero_()
    tight = (max(lens) + 63) // 64
    order = [first] + [x for x in (NARROW, MEDIUM, WIDE) if x != first] + [first]
    begin = np.array([n // 5 for n in lens], np.int32)
    for k, extra in enumerate(order):
        w = W.make_workload("over%d" % k, 8700 + 13 * k + H, lens, H=H, kv_dtype=kv_dtype, table_stride=tight + extra)
        dw = binding.DeviceWorkload(w)
        out, lse = dw.decode(kv_begin=torch.from_numpy(begin).cuda(), flags=binding.SPLASH_FLAG_REUSE_PLAN if k else 0)
        torch.cuda.synchronize()
        rc, detail = binding.splash_workspace_status(binding.decode_workspace(out.device))
        assert rc == 0, (rc, detail)
        compare(out.cpu().numpy(), lse.cpu().numpy(), *oracle_run(w, kv_begin=begin), kv_dtype=kv_dtype, what=f"layer {k}, {extra} more columns")
