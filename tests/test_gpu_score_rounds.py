"""GPU parity of scoring where a CTA's share of a row is more than one round of 4096 fp32 or
8192 bf16 entries, at the edges of rounds, vectors and shares: vocabularies one entry either
side of them, padded rows, ties between rounds, rounds of -inf, NaN and +inf."""
import numpy as np
import pytest
import torch

from paper_2608_26574_gb300 import binding as B
from paper_2608_26574_gb300 import workloads as W
from paper_2608_26574_gb300.device import DeviceStep

from . import parity as P

pytestmark = pytest.mark.gpu

ROUND = {"bf16": 8192, "f32": 4096}


def _score(wl, pitch=None):
    ds = DeviceStep(wl, attention=False, logit_pitch=pitch)
    ds.score()
    torch.cuda.synchronize()
    return ds, (ds.conf.cpu().numpy(), ds.token.cpu().numpy(), ds.state_out.cpu().numpy(),
                ds.w_out.cpu().numpy(), ds.counts.cpu().numpy())


def _check(wl, outs):
    conf, token, st, w, counts = outs
    return P.compare_scores(wl, conf, token, st, w_out=w, counts=counts)


@pytest.mark.parametrize("rounds,extra", [(16, 1), (17, -1), (32, 0), (32, 9), (33, 5), (48, 3)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_vocabularies_around_rounds(dtype, rounds, extra):
    """At most 16 CTAs share a row: past 16 rounds a CTA takes two or more."""
    vocab = rounds * ROUND[dtype] + extra
    specs = [dict(n_orig=20, block_start=4, block_len=12, fractions=(0.4, 0.3, 0.3))]
    wl = W.custom(specs, 1, 1, 64, dtype=dtype, vocab=vocab, seed=vocab, logit_std=2.0)
    per16 = 8 if dtype == "bf16" else 4
    pitch = (vocab + per16 - 1) // per16 * per16 + per16
    ds, outs = _score(wl, pitch)
    _check(wl, outs)
    assert int(ds.status.item()) == 0


def test_many_rows_ties_and_nonfinite():
    """600 rows: a few CTAs per row, several rounds each. Equal maxima in different rounds,
    vectors and the tail (the lowest index wins), a round of -inf, NaN and +inf rows."""
    vocab = 5 * ROUND["bf16"] + 11
    specs = [dict(n_orig=140, block_start=10, block_len=120, fractions=(0.4, 0.3, 0.3))
             for _ in range(5)]
    wl = W.custom(specs, 1, 1, 64, vocab=vocab, seed=77, logits="plain")
    rng = np.random.default_rng(7)
    for arr in (wl.logits_x, wl.logits_s):
        for r in range(arr.shape[0]):
            cols = rng.choice(vocab, size=3, replace=False)
            if r % 3 == 0:
                cols = np.append(cols, vocab - 1)
            arr[r, cols] = 18.0  # bf16-exact: ties
        arr[1, ROUND["bf16"]:2 * ROUND["bf16"]] = -np.inf
        arr[2, :-1] = -np.inf
    wl.logits_s[7, 3 * ROUND["bf16"] + 5] = np.nan
    wl.logits_s[8, vocab - 1] = np.inf
    wl.logits_x[7, 0] = np.nan
    wl.logits_x[8, 9] = np.inf
    ds, outs = _score(wl, (vocab + 7) // 8 * 8)
    _check(wl, outs)
    assert int(ds.status.item()) & 0x4


@pytest.mark.parametrize("block", [58, 59, 93, 94])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_rows_around_the_launch_rules(dtype, block):
    """13 CTAs of one round per row: either side of 5 CTAs per SM on 152 SMs (the bf16 variant
    with end-of-step outputs changes) and of 8 (two rounds per CTA from there on)."""
    specs = [dict(n_orig=140, block_start=10, block_len=block, fractions=(0.4, 0.3, 0.3))]
    wl = W.custom(specs, 1, 1, 64, dtype=dtype, vocab=13 * ROUND[dtype], seed=block, logit_std=2.0)
    ds, outs = _score(wl)
    _check(wl, outs)
    ent, mar, key = (torch.zeros(block, device="cuda") for _ in range(3))
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
