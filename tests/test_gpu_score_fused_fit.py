"""One-launch scoring, whose rows wait for one another: each of its kernels is launched by its own
occupancy, whichever of them ran first in the process with as many CTAs per row."""
import pytest
import torch

from paper_2608_26574_gb300 import binding as B
from paper_2608_26574_gb300 import workloads as W
from paper_2608_26574_gb300.device import DeviceStep

from . import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extras", [False, True])
def test_each_kernel_by_its_own_occupancy(extras, monkeypatch):
    """64 rows of eight rounds: 512 CTAs, which fit 152 SMs at four per SM and not at three."""
    specs = [dict(n_orig=140, block_start=10, block_len=32, fractions=(0.5, 0.3, 0.2))] * 2
    for dtype, vocab in (("f32", 8 * 4096), ("bf16", 8 * 8192)):
        wl = W.custom(specs, 1, 1, 64, dtype=dtype, vocab=vocab, seed=vocab, logit_std=2.0)
        ds = DeviceStep(wl, attention=False)
        monkeypatch.setenv("DARD_SCORE_PATH", "fused")
        kw = dict(entropy=torch.zeros(64, device="cuda")) if extras else {}
        B.dard_score_and_transition(ds.lx, ds.ls, ds.block_len, ds.state, wl.tau_c, wl.tau_u, wl.lam,
                                    wl.p0, ds.conf, ds.token, ds.state_out, ds.workspace,
                                    w_out=ds.w_out, counts=ds.counts, status=ds.status, **kw)
        torch.cuda.synchronize()
        assert int(ds.status.item()) == 0
        out = [t.cpu().numpy() for t in (ds.conf, ds.token, ds.state_out, ds.w_out, ds.counts)]
        P.compare_scores(wl, *out[:3], w_out=out[3], counts=out[4])
