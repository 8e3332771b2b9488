"""The bf16 attention kernels where the keys after the first tile weigh a few times as much as those
of it: a tile's sum passes the line at which the row's reference is raised, its largest weight does
not, or the scores go on growing beyond the room the reference was given."""
import numpy as np
import pytest

from paper_2608_26574_gb300 import workloads as W

from . import parity as P
from .test_gpu_attention_waves import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads", [(2, 1), (42, 14)])  # one wave of work, and several items per CTA
@pytest.mark.parametrize("tc", ["1", "2"])
@pytest.mark.parametrize("growth", [1.5, 2.0, 4.0, 5.5, "ramp"])
@pytest.mark.parametrize("d", [64, 128])
def test_later_keys_weigh_more(d, growth, tc, heads, monkeypatch):
    """Element 0 of the queries is sqrt(d), so that element 0 of a key is added to its score (in
    bf16: multiples of 1/2 up to 128 are exact)."""
    monkeypatch.setenv("DARD_ATTN_TC", tc)
    specs = [dict(n_orig=n, block_start=b0, block_len=16, fractions=(0.3, 0.4, 0.3))
             for n, b0 in ((84, 34), (240, 112), (512, 100), (369, 176), (624, 304), (1100, 640))]
    wl = W.custom(specs, *heads, d, seed=31 + d, qkv_std=1.0)
    offs = wl.row_offsets()
    wl.q[0][:, :, 1:] = W.round_bf16(0.5 * wl.q[0][:, :, 1:])
    wl.q[0][:, :, 0] = W.round_bf16(np.full_like(wl.q[0][:, :, 0], np.sqrt(d)))
    for a, b in zip(offs[:-1], offs[1:]):
        tile = np.arange(b - a) // 128
        wl.k[0][a:b, :, 0] = (6 * tile if growth == "ramp" else (tile > 0) * growth)[:, None]
    _, o = _run(wl, None)
    mx, mean, n = P.compare_attention(wl, 0, o, sample=24)
    print("growth", d, growth, tc, heads, mx, mean, n)
    assert mx <= P.att_tol(wl) and mean <= P.ATT_MEAN_ABS
