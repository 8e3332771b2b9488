"""Both fp32 attention kernels are equally close to 64 bits: which of them runs depends on a call's
size alone, and must not cost it accuracy."""
import math

import pytest
import torch

from paper_2608_26574_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _error(q, k, v, copies):
    """Relative error of the heads, `copies` times over in one call; the CTAs of the launch."""
    qs, ks, vs = (torch.cat([t] * copies, 1).contiguous() for t in (q, k, v))
    none = dict(dtype=torch.int32, device="cuda")
    call = B.AttentionCall([len(q)], [0], [0], [0], torch.zeros(1, dtype=torch.uint8, device="cuda"),
                           torch.zeros(1, device="cuda"), torch.zeros(1, **none))
    o = torch.zeros_like(qs)
    ctas = call.plan(qs, ks, vs, o)["ctas"]
    call(qs, ks, vs, o)
    z = torch.einsum("qhd,khd->hqk", q.double(), k.double()) / math.sqrt(q.shape[-1])
    ref = torch.einsum("hqk,khd->qhd", z.softmax(-1), v.double())
    o = o[:, :q.shape[1]].double()
    return float((o - ref).norm() / ref.norm()), ctas


@pytest.mark.parametrize("d", [64, 128])
def test_the_choice_of_kernel_costs_no_accuracy(d):
    """600 rows of 2 heads (attn_simt, four CTAs per 128 rows) and of 20 (attn_f32, two): both add up
    dot products and weighted values in short chains, and their errors, averages over 77000 or more
    outputs, stay within a quarter of one another."""
    g = torch.Generator("cuda").manual_seed(d)
    q, k, v = (torch.randn(600, 2, d, generator=g, device="cuda") for _ in range(3))
    (few, c1), (many, c2) = _error(q, k, v, 1), _error(q, k, v, 10)
    print(d, few, many, c1, c2)
    assert c1 == 4 * 5 * 2 and c2 == 2 * 5 * 20
    assert few <= 1.25 * many
