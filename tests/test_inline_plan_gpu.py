"""Batches of up to 32 requests are planned by the decode kernel itself (and, with short contexts, no request is cut);
larger ones by the plan kernel.  The oracle does not know the difference: batch sizes on both sides of the line, table
widths on both sides of the other, on every kernel family, with empty requests, ranges and a second call that takes the
partition over."""
import numpy as np
import pytest

from paper_2609_37626_b200 import workloads as W
from _util import oracle_run, compare

pytestmark = pytest.mark.gpu

FAMILIES = [(0, 16), (0, 32), (0, 64), (0, 100), (1, 16), (1, 32), (1, 50), (1, 128)]      # kv_dtype, heads


@pytest.mark.parametrize("kv_dtype,H", FAMILIES)
@pytest.mark.parametrize("B,top", [(1, 256), (1, 40000), (3, 4 * 64), (3, 4 * 64 + 1), (31, 900), (32, 200), (32, 3000), (33, 200)])
def test_batches_around_the_inline_limits(kv_dtype, H, B, top):
    import torch
    from paper_2609_37626_b200 import binding
    rng = np.random.default_rng(B * 1000 + top + H)
    lens = rng.integers(0, top + 1, size=B).astype(np.int32)
    lens[rng.integers(0, B)] = top
    if B > 2:
        lens[rng.integers(0, B - 1)] = 0
    lens[-1] = top
    w = W.make_workload("inline", 7300 + B + top, lens, H=H, kv_dtype=kv_dtype)
    dw = binding.DeviceWorkload(w)
    kb = np.where(rng.random(B) < 0.5, rng.integers(0, max(2, top // 2), size=B), 0).astype(np.int32)
    for begin in (None, kb):
        args = {} if begin is None else dict(kv_begin=torch.from_numpy(kb).cuda())
        ref = oracle_run(w, kv_begin=begin)
        first = None
        for flags in (0, binding.SPLASH_FLAG_REUSE_PLAN):
            out, lse = dw.decode(flags=flags, **args)
            torch.cuda.synchronize()
            rc, detail = binding.splash_workspace_status(binding.decode_workspace(out.device))
            assert rc == 0, (rc, detail)
            compare(out.cpu().numpy(), lse.cpu().numpy(), *ref, kv_dtype=kv_dtype, what=f"begin {begin is not None} flags {flags}")
            first = (out.clone(), lse.clone()) if first is None else first
            assert torch.equal(first[0], out) and torch.equal(first[1], lse)      # the same partition: the same bits


def test_a_stale_partition_is_not_taken_for_a_small_batch():
    """A call that plans for itself between two layers of another batch on the same workspace leaves its own records; the
    next call plans anew."""
    import torch
    from paper_2609_37626_b200 import binding
    for seed, lens in ((1, [5000, 3]), (2, [70] * 40), (3, [64, 9000, 0])):
        w = W.make_workload("stale", 7400 + seed, lens, H=16)
        out, lse = binding.DeviceWorkload(w).decode()
        torch.cuda.synchronize()
        compare(out.cpu().numpy(), lse.cpu().numpy(), *oracle_run(w), kv_dtype=0)
