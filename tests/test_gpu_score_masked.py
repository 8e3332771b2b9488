"""Scoring of logits masked by the lowest value of their type, a finite number whose product with
log2 e is not: a vector, a round and every share of a row but one, in each copy."""
import pytest
import torch

from paper_2608_26574_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extras", [False, True])
@pytest.mark.parametrize("masked", [(0, 8), (0, 40), (0, 8192), (8192, 33000), (7, 39990), (16, 17)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_lowest_value_masks(dtype, masked, extras):
    rows, vocab = 8, 40000
    g = torch.Generator("cuda").manual_seed(masked[1])
    x = (2 * torch.randn(2, rows, vocab, generator=g, device="cuda")).to(dtype)
    x[:, :, masked[0]:masked[1]] = torch.finfo(dtype).min
    x[:, :, 39995] = 9.0
    st = torch.tensor([0, 2] * 4, dtype=torch.uint8, device="cuda")  # M and U: w = 1 (no C rows)

    def out(dt):
        return torch.zeros(rows, dtype=dt, device="cuda")
    conf, token, state, status = out(torch.float32), out(torch.int32), out(torch.uint8), out(torch.int32)
    ent, mar = out(torch.float32), out(torch.float32)
    ws = torch.zeros(B.dard_score_workspace_size(rows, vocab, 1), dtype=torch.uint8, device="cuda")
    B.ScoreCall([rows], st, 0.5, 0.8, 0.9, 0.1, conf, token, state, ws, status=status,
                **(dict(entropy=ent, margin=mar) if extras else {}))(x[0], x[1])
    torch.cuda.synchronize()
    assert int(status[0]) == 0
    lp = torch.log_softmax(torch.where(st[:, None] == 0, x[0], x[1]).double(), -1)
    two = lp.exp().topk(2).values
    assert torch.allclose(conf.double(), two[:, 0], rtol=1e-5, atol=0)
    assert torch.equal(token.long(), lp.argmax(-1))
    if extras:
        assert torch.allclose(ent.double(), -(lp.exp() * lp).sum(-1), rtol=1e-5, atol=1e-4)
        assert torch.allclose(mar.double(), two[:, 0] - two[:, 1], rtol=1e-5, atol=1e-6)
