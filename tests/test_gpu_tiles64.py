"""FP64 grids on the kernels chosen for them by default -- shared-memory tiles
(tiles64.cu) or, past their range, one step per launch -- and FP64 boxes (the
flat 3-D kernel): bit for bit the FP64 oracle.

Shapes cover fewer points than SMs, thin grids, tiles that differ by a row or a
column, the largest tiles and the next larger grid; T covers single passes,
partial last passes and both parities of the exchange words.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1902_10345_gb300 import binding, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    binding.sdfg_device_error(True)


def view(g, pad, offset):
    flat = torch.zeros(int(np.prod(g.shape[:-1])) * (g.shape[-1] + pad) + offset, dtype=torch.float64, device="cuda")
    x = flat[offset:].view(*g.shape[:-1], g.shape[-1] + pad)[..., :g.shape[-1]]
    x.copy_(torch.from_numpy(g))
    return x


def check2(R, C, T, pad=0, offset=0, in_place=False):
    g = np.random.default_rng(R * 17 + C).standard_normal((R, C))
    x = view(g, pad, offset)
    y = x if in_place else view(np.full_like(g, 7.0), pad, offset)
    binding.jacobi2d(x, y, T)
    torch.cuda.synchronize()
    assert binding.sdfg_device_error(True) == 0
    assert np.array_equal(y.cpu().numpy(), oracle.jacobi2d(g, T, threads=0)), (R, C, T, pad, offset, in_place)


@pytest.mark.parametrize("shape", [(3, 3), (3, 900), (900, 3), (12, 13), (48, 50), (151, 155), (256, 256), (333, 97), (700, 301)])
@pytest.mark.parametrize("T", [1, 4, 7, 26])
def test_2d_shapes(shape, T):
    check2(*shape, T)


@pytest.mark.parametrize("pad,offset,in_place", [(1, 0, False), (0, 1, False), (3, 1, True), (0, 0, True)])
@pytest.mark.parametrize("T", [1, 6, 13])
def test_2d_layouts(pad, offset, in_place, T):
    check2(130, 211, T, pad, offset, in_place)


def test_2d_largest_tiles_and_the_next():
    for n in (1400, 1460, 1600):
        check2(n, n - 1, 5)


@pytest.mark.parametrize("shape", [(3, 3, 3), (3, 50, 4), (40, 3, 33), (31, 32, 33), (129, 40, 51)])
@pytest.mark.parametrize("T,pad,offset,in_place", [(1, 0, 0, False), (4, 1, 1, False), (5, 0, 1, True)])
def test_3d(shape, T, pad, offset, in_place):
    g = np.random.default_rng(sum(shape)).standard_normal(shape)
    x = view(g, pad, offset)
    y = x if in_place else view(np.full_like(g, 7.0), pad, offset)
    binding.jacobi3d(x, y, T)
    torch.cuda.synchronize()
    assert binding.sdfg_device_error(True) == 0
    assert np.array_equal(y.cpu().numpy(), oracle.jacobi3d(g, T, threads=0))
