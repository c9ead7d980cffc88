"""Calls whose cost must follow from their parts or their bytes, whatever their shape: limits that lie far from what is measured (half
as much again and more) and far from what went wrong (ten times and more)."""
import pytest

from paper_2609_37626_b200 import workloads as W

pytestmark = pytest.mark.gpu


def device_us(call, repeat=10):
    """The best of five: one call on the device, out of `repeat` queued behind work that covers their launches."""
    import torch
    call()
    best = float("inf")
    cover = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        for _ in range(4):
            cover.zero_()
        a.record()
        for _ in range(repeat):
            call()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / repeat)
    return best


@pytest.mark.parametrize("kv_dtype", [0, 1])
@pytest.mark.parametrize("lens", [[200], [200] * 4, [4000] * 8, [64] * 40])
def test_a_migration_job_costs_what_its_parts_cost(kv_dtype, lens):
    import torch
    from paper_2609_37626_b200 import binding
    w = W.make_workload("cost", 9500 + len(lens), lens, H=128, kv_dtype=kv_dtype)
    dw = binding.DeviceWorkload(w)
    n = 800
    shape = (n, 64, 576)
    src = torch.zeros(shape, dtype=torch.uint8 if kv_dtype else torch.bfloat16, device="cuda")
    dst = torch.empty_like(src)
    sc = [torch.zeros((n, 64), device="cuda") for _ in range(2)] if kv_dtype else [None, None]
    ids = torch.randperm(n, device="cuda").to(torch.int32)
    table = torch.arange(n, dtype=torch.int32, device="cuda")
    ws = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    args = dict(src_scales=sc[0], dst_scales=sc[1], dst_id_base=n, workspace=ws)
    job = binding.make_migrate_job(src, dst, ids, ids, table, **args)
    parts = device_us(dw.decode) + device_us(lambda: binding.splash_kv_page_migrate(src, dst, ids, ids, table, **args))
    both = device_us(lambda: dw.decode(migrate_job=job))
    assert both <= 1.5 * parts + 10, (both, parts)


@pytest.mark.parametrize("n,h,d", [(16384, 1, 576), (65536, 1, 144), (24, 1, 393216)])
def test_rows_of_any_length_move_at_one_rate(n, h, d):
    """The same 19 MB as 1,024 positions of 16 heads."""
    import torch
    from paper_2609_37626_b200 import binding

    def us(n, h, d):
        a = torch.zeros((n, h, d), dtype=torch.bfloat16, device="cuda")
        out = torch.empty_like(a)
        row = torch.randperm(n, device="cuda").to(torch.int32)
        return (device_us(lambda: binding.splash_dop_pack_rows(a, None, row, out)), device_us(lambda: binding.splash_dop_unpack_rows(a, row, out)),
                device_us(lambda: binding.splash_dop_swap_outer(a.view(8, n // 8, h, d), out.view(n // 8, 8, h, d))))

    for got, usual in zip(us(n, h, d), us(1024, 16, 576)):
        assert got <= 2 * usual + 3, (got, usual)


def test_large_pages_move_at_the_rate_of_many_small_ones():
    import torch
    from paper_2609_37626_b200 import binding

    def us(n, page):
        src = torch.zeros((n, 16, page // 16), dtype=torch.uint8, device="cuda")
        dst, ids, table = torch.empty_like(src), torch.randperm(n, device="cuda").to(torch.int32), torch.arange(n, dtype=torch.int32, device="cuda")
        return device_us(lambda: binding.splash_kv_page_migrate(src, dst, ids, ids, table, dst_id_base=n))

    large, small = us(8, 1 << 20), us(228, 36864)
    assert large <= 2 * small + 3, (large, small)


def test_wide_rows_merge_at_the_rate_of_usual_ones():
    """64 rows of four parts, 8,192 wide, against 1,024 rows of 512."""
    import torch
    from paper_2609_37626_b200 import binding

    def us(rows, d_v):
        o, l = torch.zeros((4, rows, d_v), device="cuda"), torch.zeros((4, rows), device="cuda")
        out, lse = torch.empty((rows, d_v), device="cuda"), torch.empty(rows, device="cuda")
        return device_us(lambda: binding.splash_lse_merge(o, l, out, lse))

    wide, usual = us(64, 8192), us(1024, 512)
    assert wide <= 1.5 * usual + 2, (wide, usual)


@pytest.mark.parametrize("H", [64, 128])
def test_one_query_for_all_costs_what_a_query_each_costs(H):
    """e4m3 over CTA pairs: query rows at a request stride of 0 come by other loads than those that a tensor map can state."""
    import numpy as np
    import torch
    from paper_2609_37626_b200 import binding
    w = W.make_workload("query", 9510 + H, np.random.default_rng(H).integers(200, 1500, size=512), H=H, kv_dtype=1)
    dw = binding.DeviceWorkload(w)
    apart = device_us(dw.decode)
    dw.q = dw.q[:1].expand(512, H, 576)
    shared = device_us(dw.decode)
    assert shared <= 1.1 * apart, (shared, apart)
