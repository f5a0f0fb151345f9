"""The register-tile kernel (what an untuned call runs where the chip's
registers hold the grid) against the FP64 oracle.

Shapes lie at the edges of its geometry: the least tile height (16 rows), one
tile and one row or column more, last tiles that overlap their neighbours,
grids narrower than a tile, right ring columns at every lane element, and grids
just off its range (which run elsewhere); layouts are pitched, odd, unaligned
and in place; T covers one pass, partial last passes and both parities of the
exchange buffers.

Tolerance: a step is at most five FP32 roundings of sums of weights that add up
to one, each at most 2^-24 of the largest value (1), and does not amplify what
it is given; the scaling of a pass and the ring's rounded factors add at most
8 + 2 per pass of 8 steps.  Hence 7 T 2^-24, and one more for a partial pass.
BF16 adds the rounding of the result: 2^-9.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1902_10345_gb300 import binding, build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    binding.sdfg_device_error(True)


def check(R, C, T, dtype=torch.float32, pad=0, offset=0, in_place=False):
    g = inputs.uniform_grid(R, C, seed=R * 31 + C)
    flat = torch.zeros(R * (C + pad) + offset, dtype=dtype, device="cuda")
    x = flat[offset:].view(R, C + pad)[:, :C]
    x.copy_(torch.from_numpy(g))
    x0 = x.double().cpu().numpy()
    out = torch.full((R * (C + pad) + offset,), 7.0, dtype=dtype, device="cuda")
    y = x if in_place else out[offset:].view(R, C + pad)[:, :C]
    binding.jacobi2d(x, y, T)
    torch.cuda.synchronize()
    assert binding.sdfg_device_error(True) == 0
    got = y.double().cpu().numpy()
    tol = 7 * (T + 8) * 2.0 ** -24 + (2.0 ** -9 if dtype == torch.bfloat16 else 0.0)
    assert np.abs(got - oracle.jacobi2d(x0, T, threads=0)).max() <= tol, (R, C, T, dtype, pad, offset, in_place)
    for a, b in ((got[0], x0[0]), (got[-1], x0[-1]), (got[:, 0], x0[:, 0]), (got[:, -1], x0[:, -1])):
        assert np.array_equal(a, b)
    if not in_place and pad:
        assert bool((out[offset:].view(R, C + pad)[:, C:] == 7.0).all()), "wrote between the rows"


@pytest.mark.parametrize("shape", [(16, 3), (16, 112), (17, 120), (24, 113), (25, 121), (32, 225), (33, 226), (40, 227),
                                   (48, 228), (57, 336), (130, 337), (257, 64), (272, 450), (500, 1000), (1000, 131)])
@pytest.mark.parametrize("T", [1, 8, 13, 24, 35])
def test_shapes(shape, T):
    check(*shape, T)


@pytest.mark.parametrize("cols", [200, 201, 202, 203])
@pytest.mark.parametrize("pad,offset", [(0, 0), (1, 0), (5, 1), (8, 2)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_layouts(cols, pad, offset, dtype):
    check(77, cols, 19, dtype, pad, offset)


@pytest.mark.parametrize("T", [1, 8, 9, 32])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_in_place(T, dtype):
    check(300, 517, T, dtype, in_place=True)


def test_largest_grids_and_the_next():
    for R, C in [(2176, 2128), (2176, 2129), (4352, 1064)]:
        check(R, C, 11)


def test_two_streams_at_once():
    a = [torch.rand((900, 800), device="cuda") for _ in range(2)]
    b = [torch.empty_like(v) for v in a]
    want = []
    for v in a:
        y = torch.empty_like(v)
        binding.jacobi2d(v, y, 64)
        want.append(y)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    for _ in range(10):
        for v, y, s in zip(a, b, streams):
            binding.jacobi2d(v, y, 64, stream=s)
    torch.cuda.synchronize()
    assert binding.sdfg_device_error(True) == 0
    assert all(torch.equal(y, w) for y, w in zip(b, want))


def test_replayed_graph_takes_new_inputs():
    x, y, z = (torch.rand((700, 650), device="cuda") for _ in range(3))
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        binding.jacobi2d(x, y, 40)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            binding.jacobi2d(x, y, 40, stream=torch.cuda.current_stream())
        for _ in range(3):
            x.copy_(torch.rand_like(x))
            graph.replay()
            binding.jacobi2d(x, z, 40, stream=s)
            s.synchronize()
            assert torch.equal(y, z)
    assert binding.sdfg_device_error(True) == 0
