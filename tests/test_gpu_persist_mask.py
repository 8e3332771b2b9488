"""The persistent tensor-core kernel (launches of more than one work item per SM) where a wrong
mask, a wrong rescale or another item's block would show: uniform attention over the attended keys,
scores whose maximum grows between key tiles, invalid block data in a sequence that is not a CTA's
first item, and RoPE together with query starts (the fp32 kernel of larger launches too)."""
import numpy as np
import pytest
import torch

from paper_2608_26574_gb300 import workloads as W
from paper_2608_26574_gb300.device import DeviceStep

from . import parity as P
from .test_gpu_attention_waves import ROPE, _run, _specs

pytestmark = pytest.mark.gpu


def _persistent(ds, tc):
    """The plan of a call: fewer CTAs than single tiles or pairs of a head's tiles."""
    q, k, v, o = ds.layers[0]
    plan = ds.attention_call().plan(q, k, v, o)
    wl = ds.wl
    tiles = [(s.rows - s.query_start + 127) // 128 for s in wl.seqs]
    assert plan["kernel"] == tc
    assert plan["ctas"] < wl.hq * sum(-(-t // tc) for t in tiles)


def _probe_close(wl, o, rows_of=None):
    """Q = 0: P is 1 for every attended key and the row sum their number, both exact; what is left
    is the output's rounding to bf16 (half an ulp, at most 2^-8 of it) and fp32 sums of at most 700
    products (under 1e-5 for |v| < 6). A wrong key moves a row by |v_a - v_b| / N, about 2e-3 in
    a typical element at N = 640 and more in the largest."""
    offs = wl.row_offsets()
    for si, s in enumerate(wl.seqs):
        rows = np.arange(s.query_start, s.rows)
        if len(rows) == 0:
            continue
        ref = P.oracle_attention(wl, 0, si, rows=rows)
        got = o[offs[si] + rows].astype(np.float64)
        assert np.all(np.abs(got - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-5), si


@pytest.mark.parametrize("tc", [1, 2])
@pytest.mark.parametrize("starts", [False, True])
@pytest.mark.parametrize("d", [64, 128])
def test_every_attended_key(d, starts, tc, monkeypatch):
    monkeypatch.setenv("DARD_ATTN_TC", str(tc))
    wl = W.custom(_specs(30 + d, starts), 21, 3, d, seed=60 + d, probe=True)
    ds, o = _run(wl, None)
    _persistent(ds, tc)
    _probe_close(wl, o)


@pytest.mark.parametrize("tc", [1, 2])
@pytest.mark.parametrize("growth", ["every", "first", "last", "none"])
@pytest.mark.parametrize("d", [64, 128])
def test_reference_maximum_grows(d, growth, tc, monkeypatch):
    """As in test_gpu_attention_tiles, in launches of several items per CTA; sequences of 128 k rows
    before their shadow rows give items whose two tiles take different numbers of key tiles."""
    monkeypatch.setenv("DARD_ATTN_TC", str(tc))
    specs = [dict(n_orig=n, block_start=b0, block_len=16, fractions=(0.3, 0.4, 0.3))
             for n, b0 in ((84, 34), (112, 48), (113, 48), (240, 112), (512, 100), (369, 176),
                           (256, 10), (624, 304))]
    wl = W.custom(specs, 42, 14, d, seed=71 + d, qkv_std=1.0)
    offs = wl.row_offsets()
    for a, b in zip(offs[:-1], offs[1:]):
        tile = np.arange(b - a) // 128
        f = {"every": 1 + 8 * tile, "first": 1 + 24 * (tile == 0), "last": 1 + 24 * (tile == tile[-1]),
             "none": np.ones_like(tile)}[growth]
        wl.k[0][a:b] = W.round_bf16(wl.k[0][a:b] * f[:, None, None].astype(np.float32))
    ds, o = _run(wl, None)
    _persistent(ds, tc)
    mx, mean, n = P.compare_attention(wl, 0, o, sample=40)
    print("growth", d, growth, tc, mx, mean, n)
    assert mx <= P.att_tol(wl) and mean <= P.ATT_MEAN_ABS


@pytest.mark.parametrize("tc", [1, 2])
@pytest.mark.parametrize("d", [64, 128])
def test_invalid_block_data_stays_in_its_sequence(d, tc, monkeypatch):
    """Sequence 7 of 12 has a repeated and an out-of-block shadow row, sequence 9 a state byte of 7
    (read as M): both are flagged; every other row, and theirs, sees the keys of the valid ones."""
    monkeypatch.setenv("DARD_ATTN_TC", str(tc))
    base = dict(n_orig=140, block_start=64, block_len=16, fractions=(0.4, 0.3, 0.3))
    specs = [dict(base) for _ in range(12)]
    specs[7]["shadow"] = np.array([64, 65, 65, 20, 70, 79, 78], np.int32)
    wl = W.custom(specs, 21, 3, d, seed=81 + d, probe=True)
    offs, boffs = wl.row_offsets(), wl.block_offsets()
    for si, s in enumerate(wl.seqs):  # the same states and confidences, without the two bad rows
        specs[si] = dict(n_orig=140, block_start=64, state=s.state, prev_conf=s.prev_conf,
                         shadow=np.array([64, 65, 70, 79, 78], np.int32) if si == 7 else s.shadow_src)
    good = W.custom(specs, 21, 3, d, seed=0, probe=True)
    keep = np.delete(np.arange(wl.total_rows), [offs[7] + 142, offs[7] + 143])
    good.q[0], good.k[0], good.v[0] = wl.q[0][keep], wl.k[0][keep], wl.v[0][keep]
    ds = DeviceStep(wl, layers=[0], scoring=False)
    m = int(np.flatnonzero(wl.seqs[9].state == 0)[0])
    ds.state[boffs[9] + m] = 7
    _persistent(ds, tc)
    o = ds.attention(0).float().cpu().numpy()
    assert int(ds.status.item()) == 0x1 | 0x2
    _probe_close(good, o[keep])


@pytest.mark.parametrize("rope", [1, 2])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("kernel", [1, 2, "f32"])
def test_rope_with_query_starts(kernel, d, rope, monkeypatch):
    f32 = kernel == "f32"
    if not f32:
        monkeypatch.setenv("DARD_ATTN_TC", str(kernel))
    wl = W.custom(_specs(90 + d, True), 12 if f32 else 21, 4 if f32 else 3, d,
                  dtype="f32" if f32 else "bf16", seed=95 + d + rope, qkv_std=1.0 if f32 else 0.7)
    ds, o = _run(wl, ROPE[rope])
    if not f32:
        _persistent(ds, kernel)
    mx, mean, n = P.compare_attention(wl, 0, o, sample=24, rope=ROPE[rope], bf16_operands=not f32)
    print("rope with starts", kernel, d, rope, mx, mean, n)
    assert mx <= (2e-4 * max(1.0, float(np.abs(wl.v[0]).max())) if f32 else P.att_tol(wl))
    assert f32 or mean <= P.ATT_MEAN_ABS
