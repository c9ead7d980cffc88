"""SPLASH_FLAG_REUSE_PLAN does not ask for block tables of one width.  A batch of more than 32 requests has its partition from the plan
kernel of the first layer's call, and a later layer takes it over whatever the width of its own table; a smaller one is planned by every
call for itself, cut or a request per worker by the width of the call's table, and the flag makes no difference."""
import numpy as np
import pytest

from paper_2609_37626_b200 import workloads as W
from _util import compare, oracle_run

pytestmark = pytest.mark.gpu

NARROW, MEDIUM, WIDE = 0, 300, 9000        # extra columns


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


@pytest.mark.parametrize("kv_dtype,H", [(1, 48), (1, 128), (0, 128), (1, 16), (0, 16)])
@pytest.mark.parametrize("lens", [[200] * 33, [1, 0, 256, 64, 130, 3000, 70] * 7, [5000] + [129] * 63 + [0]])
@pytest.mark.parametrize("first", [NARROW, WIDE])
def test_a_partition_is_taken_over(kv_dtype, H, lens, first):
    """The bits of a call that plans, on a workspace of its own, and one kernel less."""
    import torch
    from paper_2609_37626_b200 import binding
    tight = (max(lens) + 63) // 64
    begin = torch.tensor([n // 5 for n in lens], dtype=torch.int32, device="cuda")
    ws = None
    for k, extra in enumerate([first] + [x for x in (NARROW, MEDIUM, WIDE) if x != first] + [first]):
        w = W.make_workload("taken%d" % k, 8800 + 13 * k + H, lens, H=H, kv_dtype=kv_dtype, table_stride=tight + extra)
        dw = binding.DeviceWorkload(w)
        if ws is None:
            shape = binding.make_shape(dw.q, dw.kv_pool, dw.block_table, torch.empty((w.B, H, W.D_V), device="cuda"), torch.empty((w.B, H), device="cuda"),
                                       w.softmax_scale)
            ws = [torch.zeros(binding.splash_mla_decode_workspace_bytes(shape, 0, H), dtype=torch.uint8, device="cuda") for _ in range(2)]
        planned = dw.decode(kv_begin=begin, workspace=ws[1])
        planning = binding.splash_last_launch_count()
        taken = dw.decode(kv_begin=begin, workspace=ws[0], flags=binding.SPLASH_FLAG_REUSE_PLAN if k else 0)
        assert binding.splash_last_launch_count() == planning - (1 if k else 0)
        assert torch.equal(planned[0], taken[0]) and torch.equal(planned[1], taken[1])
        rc, detail = binding.splash_workspace_status(ws[0])
        assert rc == 0, (rc, detail)
