"""The tiles' bounded halo waits: one for a pass that never comes runs out after its
limit (1 ms here), the launch ends and the error word says so; the next call is right."""
import time

import pytest
import torch

from paper_1902_10345_gb300 import binding, build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["jacobi2d f32", "jacobi2d bf16", "jacobi2d f64", "sor2d f32"])
def test_a_halo_wait_runs_out(name):
    build.build()
    binding.sdfg_device_error(True)
    dtype = {"f32": torch.float32, "bf16": torch.bfloat16, "f64": torch.float64}[name.split()[1]]
    x = torch.rand((300, 500), device="cuda").to(dtype)
    y, z = torch.empty_like(x), torch.empty_like(x)

    def call(out):
        if name.startswith("sor"):
            binding.sor2d(x, out, 40, 1.5)
        else:
            binding.jacobi2d(x, out, 40)
        torch.cuda.synchronize()

    call(y)
    assert binding.sdfg_device_error(True) == 0
    try:
        binding.sdfg_test_hook(1, 1)
        binding.sdfg_test_hook(2, 1000000)
        t = time.perf_counter()
        call(z)
        assert time.perf_counter() - t < 1.0
        assert binding.sdfg_device_error(True) == binding.SDFG_ERR_TIMEOUT
    finally:
        binding.sdfg_test_hook(1, 0)
        binding.sdfg_test_hook(2, 0)
    assert binding.sdfg_device_error(True) == 0
    call(z)
    assert binding.sdfg_device_error(True) == 0
    assert torch.equal(y, z)
