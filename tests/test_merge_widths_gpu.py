"""The merge of partial results at part counts around its eight (four) loads in flight and the 128 parts whose weights it holds at
a time, for few rows and for more than are resident at once; parts without tokens hold NaN rows, which must not be looked at."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("parts", [1, 4, 5, 8, 9, 127, 128, 129, 260])
@pytest.mark.parametrize("rows", [3, 1185])
@pytest.mark.parametrize("d_v", [512, 20])
def test_parts_and_rows(parts, rows, d_v):
    import torch
    from paper_2609_37626_b200 import binding
    g = torch.Generator(device="cuda").manual_seed(parts * 7 + rows)
    o = torch.randn((parts, rows, d_v), generator=g, device="cuda")
    L = 3.0 * torch.randn((parts, rows), generator=g, device="cuda")
    gone = torch.rand((parts, rows), generator=g, device="cuda") < 0.3
    gone[:, 0] = True                       # a row that no part has seen
    L[gone] = -np.inf
    o[gone] = float("nan")
    out, lse = binding.splash_lse_merge(o, L)
    ref_l = torch.logsumexp(L.double(), 0)
    w = torch.where(gone, 0.0, torch.exp(L.double() - ref_l))
    ref_o = (torch.where(gone[..., None], 0.0, o.double()) * torch.where(w.isnan(), 0.0, w)[..., None]).sum(0)
    empty = ref_l.isinf()
    assert torch.equal(out[empty], torch.zeros_like(out[empty])) and torch.equal(lse.isinf(), empty)
    # sums of `parts` fp32 terms whose weights carry the error of exp, about 2^-22 each
    bound = (parts + 16) * 2.0 ** -22
    assert (out.double() - ref_o).abs().max() <= bound * 4
    assert (lse.double() - ref_l)[~empty].abs().max() <= bound * 4
