"""The chain length that an untuned BF16 call takes (by the grid's size, the steps and
the passes of their remainder) changes no bit: on both sides of the line the result
is that of every explicit length."""
import pytest
import torch

from paper_1902_10345_gb300 import binding, build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 8, 9, 131, 231])
def test_untuned_bf16_equals_explicit_lengths(T):
    build.build()
    binding.sdfg_device_error(True)
    x = torch.rand((2500, 2504), device="cuda").to(torch.bfloat16)
    y, z = torch.empty_like(x), torch.empty_like(x)
    binding.jacobi2d(x, y, T)
    for rows in (128, 512, 640):
        binding.jacobi2d(x, z, T, binding.config(kernel=binding.SDFG_KERNEL_SKEWED, k=8, seg_rows=rows))
        torch.cuda.synchronize()
        assert torch.equal(y, z), rows
    assert binding.sdfg_device_error(True) == 0
