"""The fused 3-D kernel (passes of 2 and 3 steps, FP32 and BF16) against the FP64
oracle: boxes at the edges of its tiles (30 or 42 rows x 120 columns, 112 for
BF16), column C-1 at every lane element and just past a tile, boxes of one
interior plane, row or column, many and few planes per CTA, and every mix of
passes (T = 2..7).

Tolerance: a step is at most seven FP32 roundings of sums of weights that add
up to one, each at most 2^-24 of the largest value (1), and does not amplify
what it is given; scaling and the shell's rounded factors add at most four per
pass of two steps.  Hence 9 T 2^-24.  BF16 adds the rounding of the stored box
after each pass, 2^-9 each.
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


def check(shape, T, dtype=torch.float32, pad=0, in_place=False):
    D, R, C = shape
    g = np.random.default_rng(sum(shape) * 7 + T).random(shape)
    x = torch.zeros((D, R, C + pad), dtype=dtype, device="cuda")[:, :, :C]
    x.copy_(torch.from_numpy(g))
    x0 = x.double().cpu().numpy()
    full = torch.full((D, R, C + pad), 7.0, dtype=dtype, device="cuda")
    y = x if in_place else full[:, :, :C]
    binding.jacobi3d(x, y, T)
    torch.cuda.synchronize()
    assert binding.sdfg_device_error(True) == 0
    got = y.double().cpu().numpy()
    tol = 9 * T * 2.0 ** -24 + (2.0 ** -9 * ((T + 1) // 2) if dtype == torch.bfloat16 else 0.0)
    assert np.abs(got - oracle.jacobi3d(x0, T, threads=0)).max() <= tol, (shape, T, dtype, pad, in_place)
    shell = np.ones(shape, bool)
    shell[1:-1, 1:-1, 1:-1] = False
    assert np.array_equal(got[shell], x0[shell])
    if pad and not in_place:
        assert bool((full[:, :, C:] == 7.0).all()), "wrote between the rows"


@pytest.mark.parametrize("shape", [(3, 3, 3), (3, 31, 121), (4, 30, 120), (5, 43, 122), (9, 60, 123), (40, 3, 124), (33, 61, 241),
                                   (150, 33, 3), (70, 29, 357), (8, 85, 240)])
@pytest.mark.parametrize("T", [2, 3, 4, 5, 7])
def test_shapes(shape, T):
    check(shape, T)


@pytest.mark.parametrize("cols", [112, 113, 114, 115, 225])
@pytest.mark.parametrize("T", [2, 6])
def test_bf16(cols, T):
    check((21, 47, cols), T, torch.bfloat16, pad=(8 - cols % 8) % 8)


@pytest.mark.parametrize("T", [2, 3, 4, 6])
@pytest.mark.parametrize("pad,in_place", [(3, False), (0, True), (1, True), (4, False)])
def test_layouts(T, pad, in_place):
    check((20, 50, 125), T, pad=pad, in_place=in_place)
