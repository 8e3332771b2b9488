"""Accuracy of the current token's probability where it is far below the largest: one rounding in the
exponent, none of the maximum's."""
import math

import pytest
import torch

from paper_2608_26574_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_probability_far_below_the_maximum(dtype):
    """Two logits in a row of -inf, 4 to 60 apart: p = 1 / (1 + e^gap). The exponent, up to 87 in
    powers of two, is rounded once (2^-18, times ln 2); ex2.approx, the products, the sums and the divide
    add less than 2^-20."""
    rows, vocab = 128, 8008
    g = torch.Generator("cuda").manual_seed(4)
    x = torch.full((rows, vocab), -float("inf"), device="cuda")
    gap = torch.linspace(4, 60, rows, device="cuda")
    top = 40 * torch.rand(rows, generator=g, device="cuda")
    at = torch.arange(rows, device="cuda")
    x[at, 5000 + at] = top
    x[at, at] = top - gap
    x = x.to(dtype)
    st = torch.full((rows,), 2, dtype=torch.uint8, device="cuda")

    def out(dt):
        return torch.zeros(rows, dtype=dt, device="cuda")
    p_cur, ent = out(torch.float32), out(torch.float32)
    ws = torch.zeros(B.dard_score_workspace_size(rows, vocab, 1), dtype=torch.uint8, device="cuda")
    B.ScoreCall([rows], st, 0.5, 0.8, 0.9, 0.1, out(torch.float32), out(torch.int32), out(torch.uint8), ws,
                cur_token=at.int(), p_cur=p_cur, entropy=ent)(x, x)
    torch.cuda.synchronize()
    lp = torch.log_softmax(x.double(), -1)
    want = lp[at, at].exp()
    assert float(((p_cur.double() - want) / want).abs().max()) <= math.log(2) * 2.0 ** -18 + 2.0 ** -20
    h = -torch.where(lp > -1e300, lp.exp() * lp, 0.0).sum(-1)
    assert torch.allclose(ent.double(), h, rtol=1e-5, atol=1e-5)
