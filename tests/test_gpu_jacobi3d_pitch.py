"""A 3-D box whose row pitch is so large that two rows lie more than 2^31 elements apart."""
import pytest
import torch

from paper_1902_10345_gb300 import binding, build

pytestmark = pytest.mark.gpu


def test_rows_two_to_the_thirty_apart():
    build.build()
    D, R, C, ld, T = 3, 4, 16, 2 ** 30 + 8, 3
    size = ((D - 1) * R + R - 1) * ld + C
    if torch.cuda.mem_get_info()[0] < 4 * 2 * size:
        pytest.skip("needs about 77 GB")
    small = torch.rand((D, R, C), device="cuda").to(torch.bfloat16)
    want = torch.empty_like(small)
    binding.jacobi3d(small, want, T)
    x, y = (torch.empty(size, dtype=torch.bfloat16, device="cuda").as_strided((D, R, C), (R * ld, ld, 1)) for _ in range(2))
    x.copy_(small)
    binding.jacobi3d(x, y, T)
    torch.cuda.synchronize()
    assert binding.sdfg_device_error(True) == 0
    assert torch.equal(y, want)
