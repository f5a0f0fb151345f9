"""Which untuned calls the tile kernels take: one launch of all steps there, none
where the planner has no tiling (a grid too low for a tile, a last tile row or column
whose halo would lie in two others -- 17 to 23 rows, 113 to 119 columns, 225 to
236 --, a grid past the registers)."""
import pytest
import torch

from paper_1902_10345_gb300 import binding, build

pytestmark = pytest.mark.gpu


def launches(family, call):
    build.build()
    torch.cuda.synchronize()
    binding.sdfg_stats_enable(True)
    binding.sdfg_stats_reset()
    try:
        call()
        torch.cuda.synchronize()
        return binding.sdfg_stats_get(family)[0]
    finally:
        binding.sdfg_stats_enable(False)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("shape,tiles", [((16, 3), 1), ((16, 112), 1), ((17, 120), 0), ((23, 120), 0),
                                         ((24, 120), 1), ((25, 121), 1), ((40, 224), 1), ((40, 237), 1),
                                         ((40, 238), 1), ((40, 239), 1), ((57, 336), 1), ((257, 64), 1), ((272, 450), 1),
                                         ((1000, 131), 1), ((2176, 2128), 1), ((15, 112), 0), ((24, 113), 0), ((40, 119), 0),
                                         ((32, 225), 0), ((40, 236), 0), ((2500, 2500), 0)])
def test_jacobi2d(shape, tiles, dtype):
    x = torch.rand(shape, device="cuda").to(dtype)
    assert launches("resident", lambda: binding.jacobi2d(x, torch.empty_like(x), 19)) == tiles


@pytest.mark.parametrize("shape,tiles", [((3, 3), 1), ((256, 256), 1), ((700, 300), 1), ((1400, 1400), 1), ((2048, 2048), 0)])
def test_jacobi2d_f64(shape, tiles):
    x = torch.rand(shape, device="cuda", dtype=torch.float64)
    assert launches("resident", lambda: binding.jacobi2d(x, torch.empty_like(x), 19)) == tiles


@pytest.mark.parametrize("shape,T,one", [((40, 224), 32, True), ((777, 1023), 100, True), ((40, 237), 40, True), ((1500, 1500), 40, True),
                                         ((40, 233), 40, False), ((777, 1023), 31, False), ((1600, 1600), 40, False)])
def test_sor2d(shape, T, one):
    x = torch.rand(shape, device="cuda")
    assert (launches("sor", lambda: binding.sor2d(x, torch.empty_like(x), T, 1.5)) == 1) == one
