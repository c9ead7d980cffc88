"""A call may start while the kernel in front of it on the stream still runs, and waits for it on the device.  What it reads must be what that
kernel has written, although other values lay there when it came in.  The kernel in front is one of the library's own, which let the next
one in before they store: a move of 256 MB at whose very end the inputs lie.  Inputs of two versions in turn, no synchronisation in
between, results equal to those of the same inputs left alone, bit for bit."""
import numpy as np
import pytest

from paper_2609_37626_b200 import workloads as W

pytestmark = pytest.mark.gpu

FRONT = 1 << 26                      # int32 of padding in front of the inputs


class Arena:
    """Tensors at the end of one buffer that a single move of the library fills."""

    def __init__(self, versions):
        import torch
        self.at, end = {}, FRONT
        for name, t in versions[0].items():
            n = (t.numel() * t.element_size() + 3) // 4
            self.at[name] = (end, t.dtype, t.shape)
            end += (n + 63) // 64 * 64
        self.size = (end + 1023) // 1024 * 1024
        self.buffer = torch.zeros(self.size, dtype=torch.int32, device="cuda")
        self.filled = []
        for v in versions:
            b = torch.zeros(self.size, dtype=torch.int32, device="cuda")
            for name, t in v.items():
                self.view(name, b).copy_(t)
            self.filled.append(b)

    def view(self, name, buffer=None):
        import torch
        at, dtype, shape = self.at[name]
        buffer = self.buffer if buffer is None else buffer
        n = int(np.prod(shape))
        return buffer[at:].view(torch.uint8)[:n * torch.empty((), dtype=dtype).element_size()].view(dtype).view(shape)

    def put(self, v):                # [1][n][1024] -> [n][1][1024]: a plain copy, by the library's own kernel
        from paper_2609_37626_b200 import binding
        binding.splash_dop_swap_outer(self.filled[v].view(1, -1, 1024), self.buffer.view(-1, 1, 1024))

    def check(self, call, rounds=8):
        import torch
        want = []
        for v in range(len(self.filled)):
            self.put(v)
            torch.cuda.synchronize()
            want.append([t.clone() for t in call()])
            torch.cuda.synchronize()
        got = []
        for r in range(rounds):
            self.put(r % len(self.filled))
            got.append([t.clone() for t in call()])
        torch.cuda.synchronize()
        for r, ts in enumerate(got):
            for a, b in zip(ts, want[r % len(want)]):
                assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), r


def ints(x):
    import torch
    return torch.from_numpy(np.asarray(x, dtype=np.int32)).cuda()


# planned by the decode kernel, ahead (16 and 32 heads) or not, cut and uncut; and by the plan kernel
@pytest.mark.parametrize("kv_dtype,H", [(0, 16), (0, 32), (0, 64), (0, 128), (1, 16), (1, 32), (1, 48), (1, 128)])
@pytest.mark.parametrize("lens", [[200, 3, 256, 70], [9000, 130, 65], [300, 5] * 20])
def test_lengths_ranges_table_and_queries(kv_dtype, H, lens):
    import torch
    from paper_2609_37626_b200 import binding
    w = W.make_workload("front", 8500 + H + len(lens), lens, H=H, kv_dtype=kv_dtype)
    dw = binding.DeviceWorkload(w)
    rng = np.random.default_rng(H)
    versions = []
    for v in range(3):
        keep = np.array([rng.integers(0, n + 1) for n in lens]) if v else np.array(lens)
        begin = np.array([rng.integers(0, max(1, k // 2)) for k in keep]) if v else np.zeros(len(lens))
        table = w.block_table.copy()
        if v == 2:                   # other pages: every request's in reverse
            for i, n in enumerate(lens):
                p = (n + 63) // 64
                table[i, :p] = table[i, :p][::-1]
        q = torch.randn(dw.q.shape, generator=torch.Generator().manual_seed(v)).to(torch.bfloat16).cuda()
        versions.append(dict(lens=ints(keep), begin=ints(begin), table=ints(table), q=q))
    a = Arena(versions)
    a.check(lambda: binding.splash_mla_decode(a.view("q"), dw.kv_pool, a.view("table"), a.view("lens"), softmax_scale=w.softmax_scale,
                                              kv_scales=dw.kv_scales, kv_begin=a.view("begin")))


@pytest.mark.parametrize("H", [16, 128])
@pytest.mark.parametrize("B", [3, 40])
def test_token_lists_and_rows(H, B):
    import torch
    from paper_2609_37626_b200 import binding
    versions = []
    for v in range(2):
        w = W.make_workload("fronts", 8600 + v, [700] * B, H=H, kv_dtype=2)
        sel, cnt = W.select_tokens(8600 + v, w.seq_lens, 150)
        cnt = np.maximum(cnt - 20 * v - np.arange(B) % 7, 0)
        dw = binding.DeviceWorkload(w)
        versions.append(dict(pool=dw.kv_pool, table=dw.block_table, lens=dw.seq_lens, sel=ints(sel), cnt=ints(cnt), q=dw.q))
    a = Arena(versions)
    a.check(lambda: binding.splash_mla_decode_sparse(a.view("q"), a.view("pool"), a.view("table"), a.view("lens"), a.view("sel"), a.view("cnt"),
                                                     softmax_scale=w.softmax_scale))


@pytest.mark.parametrize("parts,rows", [(5, 40), (200, 3), (3, 2000)])
def test_merge(parts, rows):
    import torch
    from paper_2609_37626_b200 import binding
    g = torch.Generator(device="cuda").manual_seed(parts)
    versions = [dict(o=torch.randn((parts, rows, 512), generator=g, device="cuda"), l=torch.randn((parts, rows), generator=g, device="cuda")) for _ in range(2)]
    a = Arena(versions)
    a.check(lambda: binding.splash_lse_merge(a.view("o"), a.view("l")))


@pytest.mark.parametrize("entries", [0, 5000])
def test_migration(entries):
    import torch
    from paper_2609_37626_b200 import binding
    P, n = 60, 40
    versions = []
    for v in range(2):
        g = torch.Generator(device="cuda").manual_seed(v)
        versions.append(dict(src=torch.randint(0, 255, (P, 64, 576), generator=g, device="cuda", dtype=torch.uint8),
                             scales=torch.randn((P, 64), generator=g, device="cuda"),
                             sid=torch.randperm(P, generator=g, device="cuda")[:n].to(torch.int32),
                             did=torch.randperm(n, generator=g, device="cuda").to(torch.int32),
                             table=torch.randint(-1, P, (entries,), generator=g, device="cuda", dtype=torch.int32)))
    a = Arena(versions)
    dst, ds = torch.zeros((n, 64, 576), dtype=torch.uint8, device="cuda"), torch.zeros((n, 64), device="cuda")

    def call():
        binding.splash_kv_page_migrate(a.view("src"), dst, a.view("sid"), a.view("did"), a.view("table"), src_scales=a.view("scales"), dst_scales=ds, dst_id_base=P)
        return dst, ds, a.view("table")
    a.check(call)


@pytest.mark.parametrize("odd", [0, 1])      # wide and 2-byte vectors
def test_layout_changes(odd):
    import torch
    from paper_2609_37626_b200 import binding
    n, h, d = 50, 4, 64 + odd
    versions = []
    for v in range(2):
        g = torch.Generator(device="cuda").manual_seed(v)
        versions.append(dict(a=torch.randint(-9000, 9000, (n, h, d), generator=g, device="cuda", dtype=torch.int16),
                             row=torch.randperm(n, generator=g, device="cuda").to(torch.int32)))
    a = Arena(versions)
    out = torch.zeros((n, h, d), dtype=torch.int16, device="cuda")
    a.check(lambda: (binding.splash_dop_pack_rows(a.view("a"), None, a.view("row")),))
    a.check(lambda: (binding.splash_dop_unpack_rows(a.view("a"), a.view("row"), out),))
    a.check(lambda: (binding.splash_dop_swap_outer(a.view("a")),))
