"""Which fp32 attention kernel a call runs on the device, and its results on either side of the line:
attn_simt while its CTAs that hold query rows (32 each) are at most one per SM, whatever the number of
128-row tiles they belong to, else attn_f32."""
import numpy as np
import pytest
import torch

from paper_2608_26574_gb300 import workloads as W
from paper_2608_26574_gb300.device import DeviceStep

from . import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beyond", [False, True])
@pytest.mark.parametrize("rows,start", [(200, 0), (129, 0), (300, 235)])
@pytest.mark.parametrize("d", [64, 128])
def test_ctas_with_query_rows_decide(d, rows, start, beyond):
    """Seven, five and three CTAs with query rows per head, of 8, 8 and 4 in the launch."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    heads = sms // ((rows - start + 31) // 32) + beyond
    tiles = (rows - start + 127) // 128
    spec = dict(n_orig=rows - 16, block_start=rows - 60, block_len=32, fractions=(0.4, 0.3, 0.3),
                shadow=np.arange(rows - 60, rows - 44))
    if start:
        spec["query_start"] = start
    wl = W.custom([spec], heads, heads, d, dtype="f32", seed=rows + d, qkv_std=1.0)
    ds = DeviceStep(wl, layers=[0], scoring=False)
    q, k, v, _ = ds.layers[0]
    out = torch.full_like(q, 7.0)
    plan = ds.attention_call().plan(q, k, v, out)
    assert plan["kernel"] == 3 and plan["ctas"] == (2 if beyond else 4) * tiles * heads
    ds.attention(0, out=out)
    torch.cuda.synchronize()
    assert int(ds.status.item()) == 0
    o = out.cpu().numpy()
    assert np.all(o[:start] == 7.0)
    mx, _, _ = P.compare_attention(wl, 0, o, sample=24)
    assert mx <= 2e-4 * max(1.0, float(np.abs(wl.v[0]).max()))
