"""GPU parity of bf16 scoring with end-of-step outputs on either side of the lines where its kernels
change: pass 1's and pass 2's register shares by CTAs per launch, one round or two per CTA by the
clusters that fit. Line by line for 152 SMs; elsewhere the same calls, wherever the lines lie."""
import pytest
import torch

from paper_2608_26574_gb300 import binding as B
from paper_2608_26574_gb300 import workloads as W
from paper_2608_26574_gb300.device import DeviceStep

from . import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,vocab", [
    (532, 1000), (533, 1000),        # rows of one CTA: pass 2 with three or four CTAs per SM
    (607, 9000), (608, 9000),        # two CTAs per row: one round, or two in one CTA
    (62, 16 * 8192 - 5), (64, 16 * 8192 - 5),  # clusters of 16
    (128, 8 * 8192), (128, 9 * 8192),  # clusters of 8 and of 9
    (1216, 1001), (1217, 1001),      # pass 1 with 56 registers or 48
])
def test_extras_around_the_launch_rules(rows, vocab):
    lens = [128] * (rows // 128) + ([rows % 128] if rows % 128 else [])
    specs = [dict(n_orig=140, block_start=10, block_len=n, fractions=(0.4, 0.3, 0.3)) for n in lens]
    wl = W.custom(specs, 1, 1, 64, vocab=vocab, seed=rows + vocab, logit_std=2.0)
    ds = DeviceStep(wl, attention=False, logit_pitch=(vocab + 7) // 8 * 8)
    ent, mar, key = (torch.zeros(rows, device="cuda") for _ in range(3))
    B.dard_score_and_transition(ds.lx, ds.ls, ds.block_len, ds.state, wl.tau_c, wl.tau_u, wl.lam,
                                wl.p0, ds.conf, ds.token, ds.state_out, ds.workspace,
                                w_out=ds.w_out, counts=ds.counts, status=ds.status, entropy=ent,
                                margin=mar, order_key=key, order_mode=B.ORDER_ENTROPY)
    torch.cuda.synchronize()
    out = [t.cpu().numpy() for t in (ds.conf, ds.token, ds.state_out, ds.w_out, ds.counts)]
    P.compare_scores(wl, *out[:3], w_out=out[3], counts=out[4], entropy=ent.cpu().numpy(),
                     margin=mar.cpu().numpy(), order_key=key.cpu().numpy(),
                     order_mode=B.ORDER_ENTROPY)
    assert int(ds.status.item()) == 0
