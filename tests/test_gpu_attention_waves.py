"""GPU parity of the attention kernels of larger launches: the persistent tensor-core kernel
(more than one work item per SM: odd head groups, lone tiles, sequences down to one row, query
starts, several sequences per CTA) and the fp32 kernel for more than one wave of query tiles,
with RoPE in the call and without; a wait that runs out in a persistent launch."""
import numpy as np
import pytest
import torch

from paper_2608_26574_gb300 import binding as B
from paper_2608_26574_gb300 import workloads as W
from paper_2608_26574_gb300.device import DeviceStep

from . import parity as P

pytestmark = pytest.mark.gpu

ROPE = {0: None, 1: (500000.0, B.DARD_ROPE_INTERLEAVED), 2: (10000.0, B.DARD_ROPE_HALF)}
LENGTHS = [1, 2, 31, 64, 65, 97, 127, 128, 129, 255, 257, 300, 383, 385, 500, 641]


def _specs(seed, starts):
    rng = np.random.default_rng(seed)
    specs = []
    for i, n in enumerate(LENGTHS):
        blen = min(n, int(rng.integers(0, 129))) if i % 4 else 0
        sp = dict(n_orig=n, block_start=int(rng.integers(0, n - blen + 1)), block_len=blen,
                  fractions=tuple(rng.dirichlet([1, 1, 1])),
                  shadow=["paper", "candidates"][i % 2])
        if starts and i % 3 == 0:
            sp["query_start"] = int(rng.integers(0, n + 1))
        specs.append(sp)
    return specs


def _run(wl, rope):
    ds = DeviceStep(wl, layers=[0], scoring=False)
    q = ds.layers[0][0]
    out = torch.full_like(q, 7.0)
    ds.attention(0, out=out, rope=rope)
    torch.cuda.synchronize()
    assert int(ds.status.item()) == 0
    o = out.float().cpu().numpy()
    offs = wl.row_offsets()
    for si, s in enumerate(wl.seqs):  # rows before the first query row are left alone
        assert np.all(o[offs[si]:offs[si] + s.query_start] == 7.0)
    return ds, o


@pytest.mark.parametrize("tc", ["1", "2"])
@pytest.mark.parametrize("rope", [0, 1, 2])
@pytest.mark.parametrize("d", [64, 128])
def test_persistent_items(d, rope, tc, monkeypatch):
    monkeypatch.setenv("DARD_ATTN_TC", tc)
    wl = W.custom(_specs(10 + d, rope == 0), 21, 3, d, seed=d + rope, qkv_std=0.7)
    ds, o = _run(wl, ROPE[rope])
    q, k, v, out = ds.layers[0]
    plan = ds.attention_call(0.0, ROPE[rope]).plan(q, k, v, out)
    assert plan["kernel"] == int(tc)
    assert plan["ctas"] <= torch.cuda.get_device_properties(0).multi_processor_count
    mx, mean, n = P.compare_attention(wl, 0, o, sample=24, rope=ROPE[rope], bf16_operands=True) \
        if rope else P.compare_attention(wl, 0, o, sample=24)
    print("persistent", d, rope, tc, plan, mx, mean, n)
    assert mx <= P.att_tol(wl) and mean <= P.ATT_MEAN_ABS


@pytest.mark.parametrize("probe", [False, True])
@pytest.mark.parametrize("rope", [0, 1, 2])
@pytest.mark.parametrize("d", [64, 128])
def test_fp32_larger_launch(d, rope, probe):
    """fp32 throughout, as for the small calls: 2e-4 of the largest value; with Q = 0 every
    attended key weighs 1/N, and a wrong one would move the output by far more than 0.25 / N."""
    if probe and rope:
        pytest.skip("Q = 0 has nothing to rotate")
    wl = W.custom(_specs(20 + d, not rope), 12, 4, d, dtype="f32", seed=50 + d + rope, probe=probe,
                  qkv_std=1.0)
    _, o = _run(wl, ROPE[rope])
    mx, mean, n = P.compare_attention(wl, 0, o, sample=None if probe else 24, rope=ROPE[rope])
    print("fp32", d, rope, probe, mx, mean, n)
    vmax = max(1.0, float(np.abs(wl.v[0]).max()))
    assert mx <= (0.25 / max(LENGTHS) if probe else 2e-4 * vmax)


@pytest.mark.parametrize("tc", ["1", "2"])
def test_wait_runs_out_in_a_persistent_launch(monkeypatch, tc):
    """The K copy of key tile 1 is never issued (nothing invalid is): every dependent wait
    gives up, and a normal call on the device afterwards matches the oracle."""
    specs = [dict(n_orig=300, block_start=200, block_len=32, fractions=(0.4, 0.3, 0.3))] * 2
    wl = W.custom(specs, 96, 96, 128, seed=5)
    ds = DeviceStep(wl, layers=[0], scoring=False)
    monkeypatch.setenv("DARD_ATTN_TC", tc)
    monkeypatch.setenv("DARD_TEST_WAIT_CYCLES", str(1 << 20))  # about half a millisecond
    monkeypatch.setenv("DARD_TEST_DROP_KV", "1")
    ds.attention(0)
    torch.cuda.synchronize()
    assert int(ds.status.item()) & 0x8
    monkeypatch.delenv("DARD_TEST_WAIT_CYCLES")
    monkeypatch.delenv("DARD_TEST_DROP_KV")
    ds.status.zero_()
    o = ds.attention(0)
    torch.cuda.synchronize()
    assert int(ds.status.item()) == 0
    mx, mean, _ = P.compare_attention(wl, 0, o.float().cpu().numpy(), sample=8)
    assert mx <= P.ATT_MAX_ABS and mean <= P.ATT_MEAN_ABS


@pytest.mark.parametrize("heads", [2, 16])
@pytest.mark.parametrize("d", [64, 128])
def test_fp32_hidden_rows_may_hold_anything(d, heads):
    """A block of settled (U) positions: shadow row j is seen by itself only. With NaN in the first
    16 shadow keys and values, every other row stays what it is."""
    n, b0, blen = 512, 256, 32
    g = torch.Generator("cuda").manual_seed(d + heads)
    q, k, v = (torch.randn(n + blen, heads, d, generator=g, device="cuda") for _ in range(3))
    call = B.AttentionCall([n], [b0], [blen], [blen],
                           torch.full((blen,), 2, dtype=torch.uint8, device="cuda"),
                           torch.full((blen,), 0.9, device="cuda"),
                           torch.arange(b0, b0 + blen, dtype=torch.int32, device="cuda"))
    clean, out = torch.zeros_like(q), torch.zeros_like(q)
    call(q, k, v, clean)
    k[n:n + 16] = float("nan")
    v[n:n + 16] = float("nan")
    call(q, k, v, out)
    torch.cuda.synchronize()
    others = torch.ones(n + blen, dtype=torch.bool, device="cuda")
    others[n:n + 16] = False
    assert torch.isfinite(clean).all() and torch.equal(out[others], clean[others])
    assert torch.isnan(out[~others]).all()
