"""A NaN among the data that a row depends on (its query, a listed entry that is out of range, a token's scale) makes that row's output
and LSE NaN and no other's, whether the request is computed in one piece, in several pieces or as parts of a merge: none of them may be
taken for a piece without tokens and left out.  Every kernel family, batches on both sides of the inline plan and combines of
every kind (a piece per worker of few rows, of many rows, few pieces of many requests)."""
import numpy as np
import pytest

from paper_2609_37626_b200 import workloads as W

pytestmark = pytest.mark.gpu

LONG = 64 * 200                     # 200 pages: cut into pieces on every kernel (at most 148 workers)
FAMILIES = [(0, 16), (0, 32), (0, 64), (0, 100), (0, 128), (1, 16), (1, 32), (1, 48), (1, 64), (1, 128)]      # kv_dtype, heads


def run(dw, **kw):
    import torch
    out, lse = dw.decode(**kw)
    torch.cuda.synchronize()
    return out.cpu().numpy(), lse.cpu().numpy()


@pytest.mark.parametrize("kv_dtype,H", FAMILIES)
@pytest.mark.parametrize("lens", [[100, 40], [LONG], [LONG, 300, 70], [LONG] + [200] * 50])
def test_a_nan_query_row(kv_dtype, H, lens):
    from paper_2609_37626_b200 import binding
    w = W.make_workload("nanq", 9100 + H + len(lens), lens, H=H, kv_dtype=kv_dtype)
    dw = binding.DeviceWorkload(w)
    good = run(dw)
    dw.q[0, H // 2, 5] = float("nan")
    out, lse = run(dw)
    assert np.isnan(out[0, H // 2]).all() and np.isnan(lse[0, H // 2])
    keep = np.ones(lse.shape, bool)
    keep[0, H // 2] = False
    assert np.array_equal(out[keep], good[0][keep]) and np.array_equal(lse[keep], good[1][keep])


@pytest.mark.parametrize("kv_dtype,H", FAMILIES)
def test_a_nan_in_one_piece_of_several(kv_dtype, H):
    from paper_2609_37626_b200 import binding
    w = W.make_workload("nanp", 9200 + H, [300, LONG, 70], H=H, kv_dtype=kv_dtype)
    dw = binding.DeviceWorkload(w)
    good = run(dw)
    page = int(w.block_table[1, 101])
    if kv_dtype:
        dw.kv_scales[page, 7] = float("nan")
    else:
        dw.kv_pool[page, 7, 3] = float("nan")
    out, lse = run(dw)
    assert np.isnan(out[1]).all() and np.isnan(lse[1]).all()
    assert np.array_equal(out[[0, 2]], good[0][[0, 2]]) and np.array_equal(lse[[0, 2]], good[1][[0, 2]])


@pytest.mark.parametrize("kv_dtype,H,R", [(0, 16, 4), (0, 64, 2), (1, 8, 4), (1, 64, 2)])
def test_a_nan_among_several_rows_and_a_row_without_tokens(kv_dtype, H, R):
    """Rows of one request: one with a NaN query, one whose causal range is empty (O = 0, LSE = -inf, as ever)."""
    import torch
    from paper_2609_37626_b200 import binding
    lens = [R - 1, LONG]                       # request 0's first row sees nothing
    w = W.make_workload("nanr", 9300 + H, lens, H=H, kv_dtype=kv_dtype)
    dw = binding.DeviceWorkload(w)
    g = torch.Generator(device="cuda").manual_seed(H)
    dw.q = torch.randn((2, H, R, 576), generator=g, device="cuda").to(torch.bfloat16)
    good = run(dw)
    dw.q[1, 3, 1, 9] = float("nan")
    out, lse = run(dw)
    assert np.all(out[0, :, 0] == 0) and np.all(np.isneginf(lse[0, :, 0]))
    assert np.isnan(out[1, 3, 1]).all() and np.isnan(lse[1, 3, 1])
    keep = np.ones(lse.shape, bool)
    keep[1, 3, 1] = False
    assert np.array_equal(out[keep], good[0][keep]) and np.array_equal(lse[keep], good[1][keep])


@pytest.mark.parametrize("H", [16, 64, 100, 128])
@pytest.mark.parametrize("listed", [60, 64 * 160])          # in one piece, and cut
def test_a_bad_list_entry(H, listed):
    import torch
    from paper_2609_37626_b200 import binding
    n = listed + 30
    w = W.make_workload("nans", 9400 + H, [300, n, 300], H=H, kv_dtype=2)
    dw = binding.DeviceWorkload(w)
    sel, cnt = W.select_tokens(9400 + H, w.seq_lens, listed)

    def sparse(sel, cnt, **kw):
        out, lse = binding.splash_mla_decode_sparse(dw.q, dw.kv_pool, dw.block_table, dw.seq_lens, torch.from_numpy(sel).cuda(),
                                                    torch.from_numpy(cnt).cuda(), softmax_scale=w.softmax_scale, **kw)
        torch.cuda.synchronize()
        return out.cpu().numpy(), lse.cpu().numpy()

    good = sparse(sel, cnt)
    bad = sel.copy()
    bad[1, listed // 2] = n                                   # one position past the end
    out, lse = sparse(bad, cnt)
    assert np.isnan(out[1]).all() and np.isnan(lse[1]).all()
    assert np.array_equal(out[[0, 2]], good[0][[0, 2]]) and np.array_equal(lse[[0, 2]], good[1][[0, 2]])
    over = cnt.copy()
    over[0] = sel.shape[1] + 1                                # a count above max_selected (which cuts the lists along other lines)
    out, lse = sparse(sel, over)
    assert np.isnan(out[0]).all() and np.isnan(lse[0]).all() and np.isfinite(out[1:]).all() and np.isfinite(lse[1:]).all()


@pytest.mark.parametrize("parts", [1, 2, 31, 33, 129])
def test_merge_of_nan_parts(parts):
    import torch
    from paper_2609_37626_b200 import binding
    o = torch.ones((parts, 4, 8), device="cuda")
    L = torch.zeros((parts, 4), device="cuda")
    L[:, 1] = float("nan")                     # every part
    L[parts - 1, 2] = float("nan")             # one of them
    L[:, 3] = -np.inf                          # none has seen a token
    out, lse = binding.splash_lse_merge(o, L)
    torch.cuda.synchronize()
    assert torch.isnan(out[1:3]).all() and torch.isnan(lse[1:3]).all()
    assert torch.isfinite(out[0]).all() and (out[3] == 0).all() and torch.isneginf(lse[3])
