"""Slices of 33 to 64 heads over an e4m3 cache run as a CTA pair of 32 heads each, the two 8-bit terms of q and of P as rows of
one operand: head counts that leave the second CTA short or end inside a group of sixteen, slices inside wider buffers,
contexts at the edges of a page, of a two-page step and of the four-stage ring, ranges cut at both ends, split requests."""
import numpy as np
import pytest

from paper_2609_37626_b200 import workloads as W
from _util import compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,hb,he", [(33, 0, 33), (48, 0, 48), (64, 0, 64), (128, 5, 54), (128, 64, 127)])
@pytest.mark.parametrize("lens", [[1, 63, 64, 65, 127, 128, 129], [512, 513, 575, 576, 640, 0, 2], [9000]])
def test_slices_and_lengths(H, hb, he, lens):
    w = W.make_workload("half", 8100 + H + he + len(lens), lens, H=H, head_begin=hb, head_end=he, kv_dtype=1)
    out, lse = gpu_run(w, sentinel=7.0)
    # the bound of the 8-bit path, 5e-2, is for the largest value scales it is used at; what the format gives on N(0, 1) rows is
    # eight significant bits of P and q against outputs of order one: 2^-8 with a factor two for the accumulated tail
    worst = compare(out, lse, *oracle_run(w), kv_dtype=1, rows=[(i, g) for i in range(len(lens)) for g in range(hb, he)])
    assert worst["abs_o"] <= 2e-2, worst
    mask = np.ones(H, bool)
    mask[hb:he] = False
    assert np.all(out[:, mask] == 7.0) and np.all(lse[:, mask] == 7.0)


@pytest.mark.parametrize("batch", [5, 40])      # planned by the decode kernel and by the plan kernel
def test_ranges(batch):
    import torch
    rng = np.random.default_rng(batch)
    lens = rng.integers(1, 900, size=batch).astype(np.int32)
    w = W.make_workload("halfr", 8200 + batch, lens, H=64, kv_dtype=1)
    a, b = np.sort(rng.integers(0, 900, size=(2, batch)), axis=0).astype(np.int32)
    a[0], b[0] = 3, 9                           # inside one page
    ref = oracle_run(w, kv_begin=a, kv_end=b)
    out, lse = gpu_run(w, kv_begin=torch.from_numpy(a).cuda(), kv_end=torch.from_numpy(b).cuda())
    compare(out, lse, *ref, kv_dtype=1)
