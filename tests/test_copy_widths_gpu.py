"""The row copies behind page migration and the DOP layout changes take the widest vector that divides every address, pitch
and length: rows at, below and above one round of a block (256 threads x 5 vectors), for 32-, 16- and 2-byte vectors, against
torch's own indexing; and a table rewrite whose remap table holds anything at first."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROUND = 256 * 5


@pytest.mark.parametrize("width", [32, 16, 2])
@pytest.mark.parametrize("vecs", [1, 255, 256, 257, ROUND - 1, ROUND, ROUND + 1, 3 * ROUND + 7])
def test_dop_rows_of_every_width(width, vecs):
    import torch
    from paper_2609_37626_b200 import binding
    n, N, el = 5, 7, width * vecs // 2
    g = torch.Generator(device="cuda"); g.manual_seed(vecs * 64 + width)
    rand = lambda *s: torch.randint(-30000, 30000, s, generator=g, device="cuda", dtype=torch.int16)
    rows = torch.tensor([6, 0, 3, 2, 5], dtype=torch.int32, device="cuda")
    x = rand(3, n, el)
    assert torch.equal(binding.splash_dop_swap_outer(x), x.transpose(0, 1).contiguous())
    recv, out = rand(n, el), rand(N, el)
    want = out.clone(); want[rows.long()] = recv
    assert torch.equal(binding.splash_dop_unpack_rows(recv, rows, out), want)
    a, b = rand(N, 2, el), rand(N, 2, width // 2)
    assert torch.equal(binding.splash_dop_pack_rows(a, b, rows), torch.cat([a, b], -1)[rows.long()])


@pytest.mark.parametrize("page_bytes", [16, 32 * ROUND, 48 * 101, 36864])
@pytest.mark.parametrize("entries", [1, 4 * 256 - 1, 4 * 256 + 1, 20000])
def test_migrate_pages_and_table(page_bytes, entries):
    import torch
    from paper_2609_37626_b200 import binding
    lib = binding.load()
    n_src, n_dst, n = 40, 30, 17
    rng = np.random.default_rng(page_bytes + entries)
    src_ids = rng.permutation(n_src)[:n].astype(np.int32)
    dst_ids = rng.permutation(n_dst)[:n].astype(np.int32)
    table = rng.integers(-3, n_src + n_dst + 3, size=entries).astype(np.int32)
    src = torch.from_numpy(rng.integers(0, 256, size=(n_src, page_bytes), dtype=np.uint8)).cuda()
    dst = torch.zeros((n_dst, page_bytes), dtype=torch.uint8, device="cuda")
    need = lib.splash_kv_page_migrate_workspace_bytes(n_src + n_dst)
    # whatever a workspace may hold: indexes of pages listed under other ids, negative and huge ones
    ws = torch.from_numpy(rng.integers(-2, n + 2, size=need // 4).astype(np.int32)).cuda()
    s, d, t = torch.from_numpy(src_ids).cuda(), torch.from_numpy(dst_ids).cuda(), torch.from_numpy(table).cuda()
    p = lambda x: ctypes.c_void_p(x.data_ptr())
    rc = lib.splash_kv_page_migrate(p(src), None, p(dst), None, page_bytes, p(s), p(d), n, 0, n_src, n_src + n_dst, p(t), entries, p(ws), need,
                                    ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, lib.splash_last_error()
    want = np.zeros((n_dst, page_bytes), np.uint8)
    want[dst_ids] = src.cpu().numpy()[src_ids]
    assert np.array_equal(dst.cpu().numpy(), want)
    move = {int(a): n_src + int(b) for a, b in zip(src_ids, dst_ids)}
    assert np.array_equal(t.cpu().numpy(), np.array([move.get(int(e), int(e)) for e in table], np.int32))


def test_a_position_of_more_vectors_than_an_int_counts():
    """2^31 and some 2-byte vectors in one position (odd addresses: no wider path), 4 GiB in and as much out."""
    import torch
    from paper_2609_37626_b200 import binding
    d, h = (1 << 20) + 1, 2049                     # h * d = 2^31 + 2^20 + 2049
    a = torch.empty((1, h, d), dtype=torch.int16, device="cuda")
    a.view(-1)[:1 << 20] = torch.arange(1 << 20, device="cuda").to(torch.int16)
    a.view(-1)[1 << 20:] = 17
    a[0, :, 0] = torch.arange(h, device="cuda").to(torch.int16)
    a[0, :, -1] = -torch.arange(h, device="cuda").to(torch.int16)
    out = torch.zeros_like(a)
    binding.splash_dop_pack_rows(a, None, torch.zeros(1, dtype=torch.int32, device="cuda"), out)
    assert torch.equal(out, a)
