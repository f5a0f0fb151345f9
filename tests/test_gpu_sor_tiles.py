"""Red-black SOR on the register tiles (the path of FP32 and BF16 grids that the
chip's registers hold): bit for bit the stated FP32 sequence -- q = (n + s) +
(w + e), then (1 - omega) c + (omega / 4) q, every operation rounded on its own,
BF16 storage rounded at every update -- so equal to the launches per pass, for
tile edges, overlapping last tiles, right ring columns at every lane element,
partial last passes, odd layouts and in place, and either side of the least
iteration count (32) that goes there."""
import numpy as np
import pytest
import torch

from paper_1902_10345_gb300 import binding, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    binding.sdfg_device_error(True)


def sequence(g, T, omega, bf16):
    """The sequence on the GPU in plain torch (elementwise, nothing fused)."""
    a, b = np.float32(1.0 - omega), np.float32(0.25 * omega)
    x = g.float().clone()
    R, C = x.shape
    i, j = torch.meshgrid(torch.arange(1, R - 1, device="cuda"), torch.arange(1, C - 1, device="cuda"), indexing="ij")
    for _ in range(T):
        for colour in (0, 1):
            q = (x[:-2, 1:-1] + x[2:, 1:-1]) + (x[1:-1, :-2] + x[1:-1, 2:])
            ac, bq = x[1:-1, 1:-1] * float(a), q * float(b)
            v = ac + bq
            if bf16:
                v = v.to(torch.bfloat16).float()
            x[1:-1, 1:-1] = torch.where((i + j) % 2 == colour, v, x[1:-1, 1:-1])
    return x


def check(R, C, T, omega, dtype=torch.float32, pad=0, offset=0, in_place=False):
    g = torch.rand((R, C), generator=torch.Generator(device="cuda").manual_seed(R * 13 + C), device="cuda").to(dtype)
    flat = torch.zeros(R * (C + pad) + offset, dtype=dtype, device="cuda")
    x = flat[offset:].view(R, C + pad)[:, :C]
    x.copy_(g)
    y = x if in_place else torch.full_like(flat, 7.0)[offset:].view(R, C + pad)[:, :C]
    binding.sor2d(x, y, T, omega)
    torch.cuda.synchronize()
    assert binding.sdfg_device_error(True) == 0
    want = sequence(g, T, omega, dtype == torch.bfloat16)
    diff = y.float() != want
    assert not bool(diff.any()), (int(diff.sum()), diff.nonzero()[:4].tolist())


@pytest.mark.parametrize("shape", [(16, 3), (17, 120), (32, 112), (40, 233), (57, 336), (130, 337), (272, 450), (700, 1021)])
@pytest.mark.parametrize("T,omega", [(3, 1.0), (32, 1.9), (35, 1.5)])
def test_shapes(shape, T, omega):
    check(*shape, T, omega)


@pytest.mark.parametrize("cols", [240, 241, 242, 243])
@pytest.mark.parametrize("pad,offset,in_place", [(0, 0, False), (1, 1, False), (4, 0, True)])
@pytest.mark.parametrize("T", [31, 34])
def test_layouts(cols, pad, offset, in_place, T):
    check(90, cols, T, 1.7, torch.float32, pad, offset, in_place)
    check(90, cols, T, 1.3, torch.bfloat16, pad, offset, in_place)
