"""The layout changes deal out their work by the vector: a block's share may begin and end inside a row, hold part of one row or thousands
of them, and go on into the next position, head or rank.  Rows from one vector to more than a block's share, counts that make
shares of every size, against torch's own indexing; pages that take several blocks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# (positions, heads, a's elements, b's elements) of int16, at even and odd addresses
SHAPES = [(1, 1, 1, 0), (3000, 1, 1, 0), (3000, 2, 1, 1), (700, 3, 16, 8), (5000, 1, 16, 0), (5000, 7, 16, 16), (900, 40, 24, 0), (77, 128, 512, 64), (300, 16, 512, 64),
          (2, 3, 20479, 0), (2, 3, 20480, 1), (3, 2, 20000, 481), (5, 1, 70000, 16), (1, 300, 2064, 0), (2, 20500, 1, 0), (2, 20500, 2, 1), (1, 41000, 16, 0)]


@pytest.mark.parametrize("n,h,da,db", SHAPES)
@pytest.mark.parametrize("odd", [0, 1])
def test_moves(n, h, da, db, odd):
    import torch
    from paper_2609_37626_b200 import binding
    g = torch.Generator(device="cuda").manual_seed(n * 7 + h + da)

    def rand(*shape):                   # at an even or odd element of its storage
        size = int(np.prod(shape))
        return torch.randint(-30000, 30000, (size + odd,), generator=g, device="cuda", dtype=torch.int16)[odd:].view(shape)

    N = n + 5
    rows = torch.randperm(N, generator=g, device="cuda")[:n].to(torch.int32)
    a, b = rand(N, h, da), rand(N, h, db) if db else None
    want = (torch.cat([a, b], -1) if db else a)[rows.long()]
    assert torch.equal(binding.splash_dop_pack_rows(a, b, rows), want)
    recv, out = rand(n, h, da), rand(N, h, da)
    want = out.clone()
    want[rows.long()] = recv
    assert torch.equal(binding.splash_dop_unpack_rows(recv, rows, out), want)
    for x in (rand(n, h, da), rand(h, n, da)):
        assert torch.equal(binding.splash_dop_swap_outer(x), x.transpose(0, 1).contiguous())


@pytest.mark.parametrize("page_bytes", [81904, 81920, 81936, 163840, 163856, 1 << 20])        # around one and two blocks' share
@pytest.mark.parametrize("entries", [0, 3, 5000])
@pytest.mark.parametrize("scales", [False, True])
def test_pages_in_several_blocks(page_bytes, entries, scales):
    import torch
    from paper_2609_37626_b200 import binding
    P, n = 9, 6
    g = torch.Generator(device="cuda").manual_seed(page_bytes + entries)
    src = torch.randint(0, 255, (P, 16, page_bytes // 16), generator=g, device="cuda", dtype=torch.uint8)
    dst = torch.zeros_like(src[:n])
    ss, ds = (torch.randn((P, 64), generator=g, device="cuda"), torch.zeros((n, 64), device="cuda")) if scales else (None, None)
    sid, did = torch.randperm(P, generator=g, device="cuda")[:n], torch.randperm(n, generator=g, device="cuda")
    table = torch.randint(-1, P, (entries,), generator=g, device="cuda", dtype=torch.int32)
    moved = torch.arange(-1, P, dtype=torch.int32, device="cuda")          # [id + 1] -> new id
    moved[sid + 1] = (P + did).to(torch.int32)
    want = moved[(table + 1).long()]
    binding.splash_kv_page_migrate(src, dst, sid.to(torch.int32), did.to(torch.int32), table, src_scales=ss, dst_scales=ds, dst_id_base=P)
    assert torch.equal(dst[did], src[sid]) and torch.equal(table, want)
    if scales:
        assert torch.equal(ds[did], ss[sid])
