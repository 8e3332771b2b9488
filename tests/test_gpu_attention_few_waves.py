"""GPU parity of launches of one to three waves, which the cost model gives to the kernels of one CTA per
query tile or pair of tiles, or to the persistent one."""
import pytest
import torch

from paper_2608_26574_gb300 import workloads as W

from . import parity as P
from .test_gpu_attention_waves import ROPE, _run

pytestmark = pytest.mark.gpu

CASES = {  # sequences, rows before the first query, heads, the kernel picked on 152 SMs at d = 128 without RoPE
    "pairs": ([310] * 3, 0, (32, 32), 2),
    "single tiles": ([560] * 10, 500, (16, 16), 1),
    "two waves of odd tiles": ([620, 333, 257, 600], 0, (24, 8), None),
    "short": ([150] * 9, 0, (32, 8), None),
}


@pytest.mark.parametrize("rope", [0, 1, 2])
@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("d", [64, 128])
def test_few_waves(d, case, rope):
    lens, start, heads, picked = CASES[case]
    specs = [dict(n_orig=n, block_start=n - 40, block_len=32, fractions=(0.4, 0.3, 0.3),
                  query_start=min(start, n)) for n in lens]
    wl = W.custom(specs, *heads, d, seed=d + len(lens) + rope, qkv_std=0.7)
    ds, o = _run(wl, ROPE[rope])
    q, k, v, out = ds.layers[0]
    plan = ds.attention_call(0.0, ROPE[rope]).plan(q, k, v, out)
    tiles = [(s.rows - s.query_start + 127) // 128 for s in wl.seqs]
    units = heads[0] * sum(-(-t // plan["kernel"]) for t in tiles)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if picked and sms == 152 and d == 128 and not rope:
        assert (plan["kernel"], plan["ctas"]) == (picked, units) and units > sms
    assert plan["ctas"] in (units, sms)
    mx, mean, n = P.compare_attention(wl, 0, o, sample=24, rope=ROPE[rope], bf16_operands=True) \
        if rope else P.compare_attention(wl, 0, o, sample=24)
    print("few waves", d, case, rope, plan, mx, mean, n)
    assert mx <= P.att_tol(wl) and mean <= P.ATT_MEAN_ABS
