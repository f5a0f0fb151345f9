"""An untuned batch of more grids than a launch is high (65535): every grid
against the stencil in 64 bits.  Tolerance as in test_gpu_batch_untuned.py: 12 T 2^-24."""
import ctypes

import pytest
import torch

from paper_1902_10345_gb300 import binding, build

pytestmark = pytest.mark.gpu


def run(xs, ys, T):
    n = len(xs)
    arr = (binding.sdfg_desc * n)(*[binding.desc_for(x, y, T) for x, y in zip(xs, ys)])
    plan, L = ctypes.c_void_p(), binding.lib()
    torch.cuda.synchronize()
    binding.check(L.sdfg_batch_plan_create(ctypes.byref(plan), arr, n, 64, None, 0))
    try:
        binding.check(L.sdfg_batch_plan_run(plan, torch.cuda.current_stream().cuda_stream))
        binding.check(L.sdfg_batch_plan_results(plan, arr, n))
    finally:
        binding.check(L.sdfg_batch_plan_destroy(plan))


def test_more_grids_than_a_launch_is_high():
    build.build()
    n, R, C, T = 65600, 72, 72, 9
    x = torch.rand((n, R, C), device="cuda")
    y = torch.zeros_like(x)
    run(list(x), list(y), T)
    assert binding.sdfg_device_error(True) == 0
    a = x.double()
    for _ in range(T):
        c = 0.2 * (a[:, 1:-1, 1:-1] + ((a[:, :-2, 1:-1] + a[:, 2:, 1:-1]) + (a[:, 1:-1, :-2] + a[:, 1:-1, 2:])))
        a[:, 1:-1, 1:-1] = c
    assert float((y - a).abs().max()) <= 12 * T * 2.0 ** -24
    for got, was in ((y[:, 0], x[:, 0]), (y[:, -1], x[:, -1]), (y[:, :, 0], x[:, :, 0]), (y[:, :, -1], x[:, :, -1])):
        assert torch.equal(got, was)
