"""Accuracy of one row's confidence where its largest term dominates: the rounding of the maximum's
product with log2 e does not reach it."""
import pytest
import torch

from paper_2608_26574_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extras", [False, True])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_a_single_term(dtype, extras):
    """One logit in a row of -inf: its probability is 1. One ex2.approx (2^-22), the products and
    sums around it (each 2^-24, below 4 in all) and the reciprocal's rounding: 2^-21 in all."""
    rows, vocab = 128, 20001 if dtype == torch.float32 else 20008
    pitch = (vocab + 7) // 8 * 8
    g = torch.Generator("cuda").manual_seed(9)
    x = torch.full((rows, pitch), -float("inf"), device="cuda")
    at = torch.randint(vocab, (rows,), generator=g, device="cuda")
    x[torch.arange(rows, device="cuda"), at] = torch.linspace(-99.0, 99.0, rows, device="cuda")
    x = x.to(dtype)[:, :vocab]
    st = torch.full((rows,), 2, dtype=torch.uint8, device="cuda")

    def out(dt):
        return torch.zeros(rows, dtype=dt, device="cuda")
    conf, token, p_cur = out(torch.float32), out(torch.int32), out(torch.float32)
    ws = torch.zeros(B.dard_score_workspace_size(rows, vocab, 1), dtype=torch.uint8, device="cuda")
    B.ScoreCall([rows], st, 0.5, 0.8, 0.9, 0.1, conf, token, out(torch.uint8), ws,
                **(dict(cur_token=at.int(), p_cur=p_cur) if extras else {}))(x, x)
    torch.cuda.synchronize()
    assert torch.equal(token.long(), at)
    assert float((conf.double() - 1).abs().max()) <= 2.0 ** -21
    if extras:
        assert float((p_cur.double() - 1).abs().max()) <= 2.0 ** -21
