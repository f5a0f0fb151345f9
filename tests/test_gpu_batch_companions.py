"""A grid's result in an untuned fixed-step batch that takes the reassociated pipe is
a function of the grid, its steps and its type: bit for bit the same beside one
companion, among few, and among so many that the launch takes taller segments;
through a plan and through the blocking call.  (FP32 and BF16 at depth 8; FP32 at
depth 4, the batches of 12 M points and more in short runs.)"""
import ctypes

import pytest
import torch

from paper_1902_10345_gb300 import binding, build

pytestmark = pytest.mark.gpu

GRIDS = [(64, 64, 16), (40, 50, 16), (16, 113, 9), (300, 517, 8), (300, 517, 7), (700, 401, 21), (129, 1000, 40), (65, 72, 13),
         (900, 5, 30), (5, 900, 30), (1000, 1000, 11)]


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    binding.sdfg_device_error(True)


def pitched(R, C, dtype, pad):
    return torch.zeros((R, C + pad), dtype=dtype, device="cuda")[:, :C]


def run(xs, Ts, tols, plan, pads):
    ys = [pitched(*x.shape, x.dtype, pad) for x, pad in zip(xs, pads)]
    descs = [binding.desc_for(x, y, T, tol) for x, y, T, tol in zip(xs, ys, Ts, tols)]
    torch.cuda.synchronize()
    if plan:
        arr, h, L = (binding.sdfg_desc * len(descs))(*descs), ctypes.c_void_p(), binding.lib()
        binding.check(L.sdfg_batch_plan_create(ctypes.byref(h), arr, len(descs), 64, None, 0))
        try:
            for _ in range(2):
                binding.check(L.sdfg_batch_plan_run(h, torch.cuda.current_stream().cuda_stream))
                binding.check(L.sdfg_batch_plan_results(h, arr, len(descs)))
        finally:
            binding.check(L.sdfg_batch_plan_destroy(h))
        assert [d.steps_done for d in arr] == Ts
    else:
        binding.check(binding.sdfg_jacobi2d_batch(descs, 64))
    assert binding.sdfg_device_error(True) == 0
    return ys


@pytest.mark.parametrize("dtype,counts,T", [(torch.float32, (0, 1, 2, 24, 48), 40), (torch.bfloat16, (1, 2, 24, 48), 40),
                                            (torch.float32, (3, 24, 48), 20)])
def test_bits_do_not_depend_on_companions(dtype, counts, T):
    """Large companions of 2400 x 2400, T steps, beside the grids: 2 M points and more (FP32 in short runs: 19 M)."""
    torch.manual_seed(7)
    grids = [(R, C, min(t, T)) for R, C, t in GRIDS]
    pads = [(-C) % 8 if i != 5 else 3 for i, (R, C, t) in enumerate(grids)]  # the sixth is staged
    xs = []
    for (R, C, _), pad in zip(grids, pads):
        x = pitched(R, C, dtype, pad)
        x.copy_(torch.rand((R, C), device="cuda"))
        xs.append(x)
    Ts, n = [t for _, _, t in grids], len(grids)
    large = [torch.rand((2400, 2400), device="cuda").to(dtype) for _ in range(48)]  # 276 M points
    few = 2 if T == 40 else 4
    one = [run([x] + large[:few], [t] + [T] * few, [0.0] * (1 + few), False, [pad] + [0] * few)[0]
           for x, t, pad in zip(xs, Ts, pads)]
    for count in counts:
        for plan in (True, False):
            ys = run(xs + large[:count], Ts + [T] * count, [0.0] * (n + count), plan, pads + [0] * count)
            for g, y, want in zip(grids, ys, one):
                assert torch.equal(y, want), (count, plan, g)
