"""dard_add_rmsnorm and dard_swiglu with every output in place of every input that the header allows,
at widths within and beyond what a thread keeps in registers: the same bits as with outputs of their
own; and a result that is rounded once, to the nearest."""
import pytest
import torch

from paper_2608_26574_gb300 import binding as B

pytestmark = pytest.mark.gpu

# (add, sum, out): "new", or the tensor that it replaces
PLACES = [("none", "none", "x"), ("add", "none", "x"), ("add", "none", "add"), ("add", "x", "new"),
          ("add", "add", "new"), ("add", "x", "add"), ("add", "add", "x"), ("none", "x", "new"),
          ("none", "new", "x")]


@pytest.mark.parametrize("place", PLACES)
@pytest.mark.parametrize("width", [1, 31, 1000, 8192, 8200, 20000, 20001])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_add_rmsnorm_in_place(dtype, width, place):
    add, total, out = place
    g = torch.Generator("cuda").manual_seed(width)
    x, d = (torch.randn(5, width, generator=g, device="cuda").to(dtype) for _ in range(2))
    other = None if add == "none" else d
    want_s, want = torch.empty_like(x), torch.empty_like(x)
    B.add_rmsnorm(x.clone(), want, None if other is None else d.clone(), want_s)
    bufs = {"x": x, "add": d, "none": None}
    t = bufs[total] if total != "new" else torch.empty_like(x)
    o = bufs[out] if out != "new" else torch.empty_like(x)
    B.add_rmsnorm(x, o, other, t)
    assert torch.equal(o, want) and (t is None or torch.equal(t, want_s))


@pytest.mark.parametrize("out", ["new", "a", "b"])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_swiglu_in_place(dtype, out):
    g = torch.Generator("cuda").manual_seed(3)
    a, b = (torch.randn(20001, generator=g, device="cuda").to(dtype) for _ in range(2))
    want = B.swiglu(a.clone(), b.clone(), torch.empty_like(a))
    got = B.swiglu(a, b, {"new": torch.empty_like(a), "a": a, "b": b}[out])
    assert torch.equal(got, want)


def test_bf16_results_are_rounded_once():
    """Against the 64-bit value: half an ulp of the result, and the fp32 arithmetic's 2^-17 of it
    (sums of at most 64 terms in a chain, rsqrtf, expf, the divide)."""
    g = torch.Generator("cuda").manual_seed(4)
    x, b = (3 * torch.randn(64, 1024, generator=g, device="cuda", dtype=torch.float64) for _ in range(2))
    x, b = x.bfloat16(), b.bfloat16()
    refs = (x.double() * (x.double().pow(2).mean(-1, keepdim=True) + 1e-6).rsqrt(),
            x.double() / (1 + (-x.double()).exp()) * b.double())
    outs = (B.add_rmsnorm(x, torch.empty_like(x)), B.swiglu(x, b, torch.empty_like(x)))
    for got, ref in zip(outs, refs):
        ulp = torch.ldexp(torch.ones_like(ref), torch.frexp(ref)[1] - 8)  # bf16: 8 significant bits
        assert torch.all((got.double() - ref).abs() <= 0.5 * ulp + 2.0 ** -17 * ref.abs() + 1e-36)
