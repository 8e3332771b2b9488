"""GPU parity of the tensor-core attention's key-tile loop at its edges: sequences of one to
five key tiles (odd tile counts, ragged ends), one or two query tiles per CTA, and scores
whose maximum grows from tile to tile, so that the reference maximum is raised (weights
computed again, O rescaled) on every tile, on the first or on the last only."""
import numpy as np
import pytest
import torch

from paper_2608_26574_gb300 import workloads as W
from paper_2608_26574_gb300.device import DeviceStep

from . import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tc", ["1", "2"])
@pytest.mark.parametrize("growth", ["every", "first", "last", "none"])
@pytest.mark.parametrize("d", [64, 128])
def test_reference_maximum_over_key_tiles(d, growth, tc, monkeypatch):
    monkeypatch.setenv("DARD_ATTN_TC", tc)
    rows = [100, 128, 129, 256, 257, 385, 640]
    specs = [dict(n_orig=r - 16, block_start=(r - 32) // 2, block_len=16, fractions=(0.3, 0.4, 0.3))
             for r in rows]
    wl = W.custom(specs, 6, 2, d, seed=41 + d, qkv_std=1.0)
    offs = wl.row_offsets()
    for a, b in zip(offs[:-1], offs[1:]):
        tile = np.arange(b - a) // 128
        # the tile's scores have a spread of about this factor: a step of 8 raises the row
        # maximum by far more than 2^8 in probability
        f = {"every": 1 + 8 * tile, "first": 1 + 24 * (tile == 0), "last": 1 + 24 * (tile == tile[-1]),
             "none": np.ones_like(tile)}[growth]
        wl.k[0][a:b] = W.round_bf16(wl.k[0][a:b] * f[:, None, None].astype(np.float32))
    ds = DeviceStep(wl, layers=[0], scoring=False)
    o = ds.attention(0)
    torch.cuda.synchronize()
    mx, mean, n = P.compare_attention(wl, 0, o.float().cpu().numpy())
    print("tiles", d, growth, tc, mx, mean, n)
    assert mx <= P.att_tol(wl) and mean <= P.ATT_MEAN_ABS
    assert int(ds.status.item()) == 0
