"""What a row does not see does not reach its output: shadow rows that hold NaN between others that
do not, in the fp32 attention kernels (few heads: attn_simt, more: attn_f32)."""
import pytest
import torch

from paper_2608_26574_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads", [2, 16])
@pytest.mark.parametrize("d", [64, 128])
def test_single_hidden_rows_may_hold_anything(d, heads):
    """A block of settled (U) positions: shadow row j is seen by itself only. Rows next to a
    poisoned one (of the same step of four keys, of the next step, of another tile) see their own
    key among hidden ones."""
    n, b0, blen = 509, 250, 40
    g = torch.Generator("cuda").manual_seed(d + heads)
    q, k, v = (torch.randn(n + blen, heads, d, generator=g, device="cuda") for _ in range(3))
    call = B.AttentionCall([n], [b0], [blen], [blen],
                           torch.full((blen,), 2, dtype=torch.uint8, device="cuda"),
                           torch.full((blen,), 0.9, device="cuda"),
                           torch.arange(b0, b0 + blen, dtype=torch.int32, device="cuda"))
    clean, out = torch.zeros_like(q), torch.zeros_like(q)
    call(q, k, v, clean)
    bad = torch.zeros(n + blen, dtype=torch.bool, device="cuda")
    for j in (1, 6, 7, 8, 13, 34, 39):
        bad[n + j] = True
    v[bad] = float("nan")
    k[bad] = float("inf")
    call(q, k, v, out)
    torch.cuda.synchronize()
    assert torch.isfinite(clean).all() and torch.equal(out[~bad], clean[~bad])
    assert torch.isnan(out[bad]).all()
