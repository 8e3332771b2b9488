"""GPU parity of the elementwise kernels between a layer's projections (residual add with RMSNorm,
SwiGLU gate) against 64-bit references: widths around the 16-byte vectors, the registers a thread
keeps and the rows beyond them, unaligned rows, outputs in place of inputs."""
import pytest
import torch

from paper_2608_26574_gb300 import binding as B

pytestmark = pytest.mark.gpu

# relative error of one result: bf16 rounds by at most 2^-9; in fp32 sums of at most 64 terms in
# a chain, rsqrtf, expf and the divide stay under 2^-17
TOL = {torch.bfloat16: 2.0 ** -8, torch.float32: 2.0 ** -17}


def _close(got, ref, dtype):
    assert torch.all((got.double() - ref).abs() <= TOL[dtype] * ref.abs() + 1e-36)


@pytest.mark.parametrize("place", ["new", "in place", "no sum"])
@pytest.mark.parametrize("width", [1, 7, 8, 31, 264, 1000, 1024, 8191, 8192, 8200])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_add_rmsnorm(dtype, width, place):
    g = torch.Generator("cuda").manual_seed(width)
    x, d = (torch.randn(5, width, generator=g, device="cuda").to(dtype) for _ in range(2))
    s = x if place == "no sum" else x + d
    ref = s.double() * (s.double().pow(2).mean(-1, keepdim=True) + 1e-6).rsqrt()
    if place == "no sum":
        out = B.add_rmsnorm(x, torch.empty_like(x))
    else:
        total, out = (x, d) if place == "in place" else (torch.empty_like(x), torch.empty_like(x))
        B.add_rmsnorm(x, out, d, total)
        assert torch.equal(total, s)
    _close(out, ref, dtype)


@pytest.mark.parametrize("n", [1, 7, 8, 2047, 2048, 100003])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_swiglu(dtype, n):
    g = torch.Generator("cuda").manual_seed(n)
    a, b = ((8 * torch.randn(n, generator=g, device="cuda")).to(dtype) for _ in range(2))
    ref = a.double() / (1 + (-a.double()).exp()) * b.double()
    _close(B.swiglu(a, b, torch.empty_like(a)), ref, dtype)
    B.swiglu(a, b, b)
    _close(b, ref, dtype)


def test_rejections():
    x = torch.zeros(4, 8, device="cuda")
    for bad in (x.bfloat16(), x[:2], x.t(), x.cpu()):
        with pytest.raises(ValueError):
            B.add_rmsnorm(x, bad)
        with pytest.raises(ValueError):
            B.swiglu(x, x, bad)
    with pytest.raises(B.DardError):
        B.add_rmsnorm(x, x, eps=-1.0)
