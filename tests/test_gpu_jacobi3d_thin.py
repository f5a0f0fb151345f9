"""Boxes of few large planes run a step per launch, in the plain order: bit for bit
the operation as written, each step rounded in FP32 (BF16: and when it is stored);
boxes just across either line run fused passes, to the FP32 tolerance."""
import pytest
import torch

from paper_1902_10345_gb300 import binding, build

pytestmark = pytest.mark.gpu


def steps(x, T, dtype):
    """T steps of `dtype`'s arithmetic, FP32 rounded to `x`'s type at each store."""
    a = x.clone()
    seventh = torch.tensor(1.0 / 7.0, dtype=dtype, device="cuda")
    for _ in range(T):
        f = a.to(dtype)
        s = (f[1:-1, :-2, 1:-1] + f[1:-1, 2:, 1:-1]) + (f[1:-1, 1:-1, :-2] + f[1:-1, 1:-1, 2:])
        s = f[1:-1, 1:-1, 1:-1] + (s + (f[:-2, 1:-1, 1:-1] + f[2:, 1:-1, 1:-1]))
        a[1:-1, 1:-1, 1:-1] = (seventh * s).to(a.dtype)
    return a


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("shape,T,alone", [((3, 1024, 768), 2, True), ((8, 1024, 768), 5, True), ((5, 901, 1003), 3, True),
                                           ((9, 1024, 768), 5, False), ((8, 1024, 767), 5, False)])
@pytest.mark.parametrize("in_place", [False, True])
def test_thin_boxes(shape, T, alone, dtype, in_place):
    build.build()
    binding.sdfg_device_error(True)
    torch.manual_seed(1)
    x = torch.rand(shape, device="cuda").to(dtype)
    x0 = x.clone()
    y = x if in_place else torch.empty_like(x)
    binding.jacobi3d(x, y, T)
    torch.cuda.synchronize()
    assert binding.sdfg_device_error(True) == 0
    assert in_place or torch.equal(x, x0)
    same = steps(x0, T, torch.float32)
    if alone:
        assert torch.equal(y, same)
    else:
        # seven roundings a step and the pass's factors; BF16 one per pass of two steps or more
        tol = 12 * T * 2.0 ** -24 + (T * 2.0 ** -9 if dtype == torch.bfloat16 else 0.0)
        want = steps(x0.double(), T, torch.float64)
        assert float((y.double() - want).abs().max()) <= tol
        assert not torch.equal(y, same)
