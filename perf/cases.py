"""Calls that a user of this library makes, over the range in which they make them.

A decode step of a serving process calls the attention of one rank's shard: a head slice (TP / DOP), a request slice
(DP-attention) or a KV range (CP) of a batch whose contexts reach from a handful of tokens to hundreds of thousands,
from a bf16 or an e4m3 cache, with one query row per request or a few; or attention over a token list.  Around it stand
the merge of partial results, the page migration of a layout switch and the layout changes of the DOP exchange.

Lengths of a batch are the quantiles of a distribution, dealt to the requests in an order that the seed decides: the work
of a case does not depend on the seed, its inputs do.
"""
import math
import statistics

import numpy as np
import torch

from paper_2609_37626_b200 import binding as B

D_QK, D_V, PAGE = 576, 512, 64
SCALE = 1.0 / math.sqrt(192.0)          # 1 / sqrt(d_nope + d_rope)
ROW_BYTES = {"bf16": 2 * D_QK, "e4m3": D_QK + 4, "rows656": 656}


def listed():
    return [
        # The smallest batch: four short contexts, one TP-8 rank's heads.  Launches and host work are all there is.
        dict(name="tiny", kind="decode", kv="bf16", batch=4, lengths="log", low=1, high=256, heads=16, first=0, slice=16, rows=1),
        # One decode step of a small interactive batch: a TP-8 rank goes through eight layers, each with its own cache; the
        # first layer's call cuts the work, the others take its cut over.
        dict(name="small_batch_layers", kind="layers", kv="e4m3", batch=8, lengths="rollout", low=16, high=131072, heads=16, layers=8),
        # DP-attention: all 128 heads over a rank's own requests, contexts of 1k to 8k tokens.
        dict(name="dp_attention", kind="decode", kv="bf16", batch=64, lengths="uniform", low=1024, high=8192, heads=128, first=0, slice=128, rows=1),
        # A TP / DOP rank's 16 of 128 heads over the complete histories, written into the shared [B][128] buffers.
        dict(name="tp8_slice_32k", kind="decode", kv="bf16", batch=16, lengths="uniform", low=32768, high=32768, heads=128, first=32, slice=16, rows=1),
        # Position-sharded CP on one very long context: the rank's eighth of it, then the merge of the eight partial results.
        dict(name="cp_shard_256k", kind="cp", kv="bf16", batch=1, lengths="uniform", low=262144, high=262144, heads=128, ranks=8),
        # RL rollout: 512 requests, many short and a few very long, all heads, the cache in e4m3 with a scale per token.
        dict(name="rollout", kind="decode", kv="e4m3", batch=512, lengths="rollout", low=16, high=131072, heads=128, first=0, slice=128, rows=1),
        # The same batch on a TP-8 rank.
        dict(name="rollout_tp8", kind="decode", kv="e4m3", batch=512, lengths="rollout", low=16, high=131072, heads=16, first=0, slice=16, rows=1),
        # A TP-2 rank's 64 heads, a batch in the middle of the range.
        dict(name="tp2_e4m3", kind="decode", kv="e4m3", batch=100, lengths="log", low=500, high=20000, heads=64, first=0, slice=64, rows=1),
        # Several query rows per request (a drafted continuation is verified in one step), a TP-4 rank.
        dict(name="draft_rows", kind="decode", kv="bf16", batch=48, lengths="uniform", low=1000, high=8000, heads=32, first=0, slice=32, rows=4),
        # Sparse decode: an indexer has picked 2,048 tokens per request, 656-byte rows, all heads.
        dict(name="sparse_top2048", kind="sparse", kv="rows656", batch=64, lengths="uniform", low=1024, high=8192, heads=128, topk=2048),
        # Layout switch: 30 % of the rollout batch's pages move into the new view, the block table follows.
        dict(name="migrate", kind="migrate", kv="e4m3", batch=512, lengths="rollout", low=16, high=131072, share=0.3),
        # DOP: both layout changes on either side of the two all-to-alls, a prefill-sized exchange among eight ranks.
        dict(name="dop_exchange", kind="dop", n=16384, heads=16, ranks=8),
    ]


def _log(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    most = work(next(c for c in listed() if c["name"] == "rollout"))
    while True:
        kind = rng.choice(["decode"] * 6 + ["layers", "cp", "sparse", "sparse", "migrate", "dop"])
        if kind == "dop":
            ranks = rng.choice([2, 4, 8])
            case = dict(kind=kind, n=ranks * _log(rng, 1, 16384 // ranks), heads=128 // ranks, ranks=ranks)
            if case["n"] * case["heads"] > 16384 * 16:
                continue
            return case
        lengths = rng.choice(["rollout", "uniform", "log"])
        if lengths == "rollout":
            low, high = 16, 131072
        else:
            low = _log(rng, 1, 65536)
            high = min(262144, low * rng.randint(1, 16) + rng.randint(0, 63))
        case = dict(kind=kind, kv=rng.choice(["bf16", "e4m3"]), batch=_log(rng, 1, 512), lengths=lengths, low=low, high=high)
        heads = rng.choice([8, 16, 16, 32, 64, 128, 128, rng.randint(1, 128)])
        if kind == "decode":
            shared = rng.random() < 0.25        # a slice of buffers that hold all heads, or the rank's own buffers
            rows = rng.choice([1, 1, 1, rng.randint(2, 8)])
            total = 128 if shared else heads
            case.update(heads=total, first=rng.randint(0, total - heads), slice=heads, rows=rows)
        elif kind == "layers":
            case.update(heads=heads, layers=rng.randint(2, 8))
        elif kind == "cp":
            case.update(heads=heads, ranks=rng.choice([2, 4, 8]))
        elif kind == "sparse":
            case.update(kv="rows656", heads=heads, topk=_log(rng, 64, 2048))
        else:
            case.update(share=round(rng.uniform(0.05, 1.0), 2))
        w = work(case)
        if w["bytes"] <= most["bytes"] and w["flops"] <= most["flops"] and _pages(case).sum() * case.get("layers", 1) <= 65536:
            return case


# ---- sizes ----------------------------------------------------------------------------------------------------------

def _lengths(case):
    """The batch's context lengths, ascending."""
    at = [(i + 0.5) / case["batch"] for i in range(case["batch"])]
    low, high = case["low"], case["high"]
    if case["lengths"] == "rollout":        # lognormal, median 2,048, sigma 1.2
        normal = statistics.NormalDist(math.log(2048.0), 1.2)
        x = [math.exp(normal.inv_cdf(u)) for u in at]
    elif case["lengths"] == "log":
        x = [math.exp(math.log(low) + u * (math.log(high) - math.log(low))) for u in at]
    else:
        x = [low + u * (high - low) for u in at]
    return np.array([min(high, max(low, round(v))) for v in x], dtype=np.int64)


def _pages(case):
    return (_lengths(case) + PAGE - 1) // PAGE


def _shard(lengths, rank, ranks):
    """Position-sharded CP: rank's tokens of every request."""
    return lengths * rank // ranks, lengths * (rank + 1) // ranks


def work(case):
    if case["kind"] == "dop":
        q, o = case["n"] * case["heads"] * D_QK * 2, case["n"] * case["heads"] * D_V * 4
        return {"bytes": 4 * q + 4 * o + 8 * case["n"], "flops": 0}     # four moves, each reads and writes its rows once
    lens, batch = _lengths(case), case["batch"]
    if case["kind"] == "migrate":
        n = max(1, round(case["share"] * int(_pages(case).sum())))
        page = PAGE * ROW_BYTES[case["kv"]]
        return {"bytes": n * (2 * page + 8) + 8 * batch * int(_pages(case).max()), "flops": 0}
    rows = case.get("rows", 1) * case.get("slice", case["heads"])
    ends = rows * batch * (D_QK * 2 + (D_V + 1) * 4)                    # the query rows in, O and LSE out
    if case["kind"] == "sparse":
        tokens = int(np.minimum(lens, case["topk"]).sum())
        more, extra = 4 * tokens, 0
    elif case["kind"] == "cp":
        a, b = _shard(lens, case["ranks"] // 2, case["ranks"])
        tokens = int((b - a).sum())
        more, extra = 4 * int(_pages(case).sum()), (case["ranks"] + 1) * rows * batch * (D_V + 1) * 4
    else:
        tokens, more, extra = int(lens.sum()), 4 * int(_pages(case).sum()), 0
    layers = case.get("layers", 1)
    return {"bytes": layers * (tokens * ROW_BYTES[case["kv"]] + ends + more + 8 * batch) + extra,
            "flops": layers * 2 * rows * (D_QK + D_V) * tokens}


def tolerance(case):
    if case["kind"] in ("migrate", "dop"):
        return "exact"
    # softmax weights and (e4m3) query rows enter the tensor cores with about 8 significant bits
    return {"rel": 1e-2}


# ---- inputs ---------------------------------------------------------------------------------------------------------

def _normal(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _quantise(x):
    """e4m3 codes and the fp32 scale that puts the largest value of the last dimension at 448."""
    scale = x.abs().amax(dim=-1, keepdim=True) / 448.0
    return (x / scale).clamp(-448.0, 448.0).to(torch.float8_e4m3fn).view(torch.uint8), scale


def _cache(g, kv, pages):
    """N(0, 1) rows in the cache's format: (pool, scales or None)."""
    width = {"bf16": D_QK, "e4m3": D_QK, "rows656": 656}[kv]
    pool = torch.empty((pages, PAGE, width), dtype=torch.bfloat16 if kv == "bf16" else torch.uint8, device="cuda")
    scales = torch.empty((pages, PAGE), device="cuda") if kv == "e4m3" else None
    for p in range(0, pages, 2048):
        n = min(2048, pages - p)
        x = _normal(g, n, PAGE, D_QK)
        if kv == "bf16":
            pool[p:p + n] = x
        elif kv == "e4m3":
            codes, s = _quantise(x)
            pool[p:p + n], scales[p:p + n] = codes, s[..., 0]
        else:
            codes, s = _quantise(x[..., :D_V].reshape(n, PAGE, 4, 128))
            pool[p:p + n, :, :D_V] = codes.reshape(n, PAGE, D_V)
            pool[p:p + n, :, D_V:D_V + 16] = s.reshape(n, PAGE, 4).contiguous().view(torch.uint8)
            pool[p:p + n, :, D_V + 16:] = x[..., D_V:].to(torch.bfloat16).contiguous().view(torch.uint8)
    return pool, scales


def _batch(case, g, seed):
    """(lengths, block table, pages of the pool, ids in use): the pages of a pool a quarter larger than needed, dealt at random."""
    order = np.random.default_rng(seed)
    lens = order.permutation(_lengths(case))
    pages = (lens + PAGE - 1) // PAGE
    used, most = int(pages.sum()), int(pages.max())
    pool = used + (used + 3) // 4
    ids = torch.randperm(pool, generator=g, device="cuda")[:used].to(torch.int32)
    mine = torch.from_numpy(np.arange(most)[None, :] < pages[:, None]).cuda()
    table = torch.full((len(lens), most), -1, dtype=torch.int32, device="cuda")
    table[mine] = ids
    return lens, table, pool, ids


def _ints(x):
    return torch.from_numpy(np.asarray(x, dtype=np.int32)).cuda()


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["kind"] == "dop":
        n, h, t = case["n"], case["heads"], case["ranks"]
        q = _normal(g, n, h, D_QK).to(torch.bfloat16)
        return dict(case=case, nope=q[..., :D_V].contiguous(), rope=q[..., D_V:].contiguous(),
                    send_row=torch.randperm(n, generator=g, device="cuda").to(torch.int32),
                    received=_normal(g, t, n // t, h, D_QK).to(torch.bfloat16), computed=_normal(g, n // t, t, h, D_V),
                    returned=_normal(g, n, h, D_V), out=torch.zeros((n, h, D_V), device="cuda"))
    lens, table, pages, used = _batch(case, g, seed)
    batch = case["batch"]
    if case["kind"] == "migrate":
        n = max(1, round(case["share"] * used.numel()))
        pool, scales = _cache(g, case["kv"], pages)
        return dict(case=case, pool=pool, scales=scales, table=table, new_pool=torch.zeros_like(pool[:n]),
                    new_scales=None if scales is None else torch.zeros_like(scales[:n]),
                    src=used[torch.randperm(used.numel(), generator=g, device="cuda")[:n]],
                    dst=torch.randperm(n, generator=g, device="cuda").to(torch.int32))
    state = dict(case=case, table=table, lens=_ints(lens))
    if case["kind"] == "layers":
        state["layers"] = []
        for _ in range(case["layers"]):
            pool, scales = _cache(g, case["kv"], pages)
            state["layers"].append((_normal(g, batch, case["heads"], D_QK).to(torch.bfloat16), pool, scales))
        q = state["layers"][0][0]
        out, lse = q.new_empty((batch, case["heads"], D_V), dtype=torch.float32), q.new_empty((batch, case["heads"]), dtype=torch.float32)
        shape = B.make_shape(q, pool, table, out, lse, SCALE)
        state["workspace"] = torch.empty(B.splash_mla_decode_workspace_bytes(shape, 0, case["heads"]), dtype=torch.uint8, device="cuda")
        return state
    state["pool"], state["scales"] = _cache(g, case["kv"], pages)
    if case["kind"] == "decode":
        rows = (case["rows"],) if case["rows"] > 1 else ()
        state["q"] = _normal(g, batch, case["heads"], *rows, D_QK).to(torch.bfloat16)
        if case["slice"] < case["heads"]:   # one rank's part of buffers that the ranks share
            state["out"] = torch.zeros((batch, case["heads"]) + rows + (D_V,), device="cuda")
            state["lse"] = torch.zeros((batch, case["heads"]) + rows, device="cuda")
        return state
    state["q"] = _normal(g, batch, case["heads"], D_QK).to(torch.bfloat16)
    if case["kind"] == "sparse":
        count = np.minimum(lens, case["topk"])
        # distinct positions, uniformly drawn, in no order: what is hardest to fetch
        sel = torch.full((batch, case["topk"]), -1, dtype=torch.int32, device="cuda")
        for i in range(batch):
            sel[i, :int(count[i])] = torch.randperm(int(lens[i]), generator=g, device="cuda")[:int(count[i])].to(torch.int32)
        state["sel"], state["count"] = sel, _ints(count)
        return state
    a, b = _shard(lens, case["ranks"] // 2, case["ranks"])
    state["begin"], state["end"] = _ints(a), _ints(b)
    # the other ranks' partial results, as the gather of the CP step delivers them; this rank's own come beside them
    state["part_out"] = 0.05 * _normal(g, case["ranks"], batch * case["heads"], D_V)
    state["part_lse"] = math.log(float(lens.mean()) / case["ranks"] + 1.0) + 1.5 + 0.1 * _normal(g, case["ranks"], batch * case["heads"])
    return state


# ---- the calls ------------------------------------------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "decode":
        first, end = case["first"], case["first"] + case["slice"]
        return B.splash_mla_decode(state["q"], state["pool"], state["table"], state["lens"], softmax_scale=SCALE,
                                   kv_scales=state["scales"], head_begin=first, head_end=end,
                                   out=state.get("out"), lse=state.get("lse"))
    if kind == "layers":
        done = []
        for i, (q, pool, scales) in enumerate(state["layers"]):
            done.append(B.splash_mla_decode(q, pool, state["table"], state["lens"], softmax_scale=SCALE, kv_scales=scales,
                                            workspace=state["workspace"], flags=B.SPLASH_FLAG_REUSE_PLAN if i else 0))
        return done
    if kind == "cp":
        rank, n = case["ranks"] // 2, case["batch"] * case["heads"]
        own_out, own_lse = state["part_out"][rank].view(case["batch"], case["heads"], D_V), state["part_lse"][rank].view(case["batch"], case["heads"])
        B.splash_mla_decode(state["q"], state["pool"], state["table"], state["lens"], softmax_scale=SCALE, kv_scales=state["scales"],
                            kv_begin=state["begin"], kv_end=state["end"], out=own_out, lse=own_lse)
        out, lse = B.splash_lse_merge(state["part_out"], state["part_lse"])
        return own_out, own_lse, out, lse
    if kind == "sparse":
        return B.splash_mla_decode_sparse(state["q"], state["pool"], state["table"], state["lens"], state["sel"], state["count"],
                                          softmax_scale=SCALE)
    if kind == "migrate":
        # one arena: the new pool's page ids follow the old one's in the table
        B.splash_kv_page_migrate(state["pool"], state["new_pool"], state["src"], state["dst"], state["table"], src_scales=state["scales"],
                                 dst_scales=state["new_scales"], src_id_base=0, dst_id_base=state["pool"].shape[0])
        return state["new_pool"], state["new_scales"], state["table"]
    send = B.splash_dop_pack_rows(state["nope"], state["rope"], state["send_row"])
    queries = B.splash_dop_swap_outer(state["received"])            # source-rank major -> all heads of the owned rows
    back = B.splash_dop_swap_outer(state["computed"])               # and the results' way back
    B.splash_dop_unpack_rows(state["returned"], state["send_row"], state["out"])
    return send, queries, back, state["out"]
