"""Large values, infinities and NaN: what the exact order of operations gives for
them, the faster orders give too.  Infinities and NaN appear at the same points as in
64 bits; finite results, up to 5e37 (five of which still add up to an FP32 number),
agree to the relative tolerance of the other tests times the largest value, and points
that no large value can have reached to that tolerance itself.

Tolerance: 12 T 2^-24 as in test_gpu_batch_untuned.py; BF16 adds a rounding per pass,
at most 2^-8 of the value (half a unit of an 8-bit significand), which is 2^-9 for
values up to 1."""
import ctypes

import pytest
import torch

from paper_1902_10345_gb300 import binding, build

pytestmark = pytest.mark.gpu

INF, NAN, BIG = float("inf"), float("nan"), 5e37


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    binding.sdfg_device_error(True)


def jacobi2d64(x, T):
    a = x.double()
    for _ in range(T):
        c = 0.2 * (a[1:-1, 1:-1] + ((a[:-2, 1:-1] + a[2:, 1:-1]) + (a[1:-1, :-2] + a[1:-1, 2:])))
        a[1:-1, 1:-1] = c
    return a


def plant(x, what):
    """`x` in [0, 1] with something large in it, and where that was put."""
    R, C = x.shape
    spots = {
        "ring inf": [(0, slice(None), INF)],
        "column -inf": [(slice(None), C - 1, -INF)],
        "point inf": [(R // 2, C // 2, INF)],
        "inf and -inf": [(0, slice(None), INF), (R - 1, slice(None), -INF), (R // 3, C // 3, -INF)],
        "nan": [(R // 2, C // 3, NAN)],
        "ring large": [(0, slice(None), BIG), (slice(None), 0, -BIG)],
        "point large": [(R // 2, C // 2, BIG), (R - 2, 1, -BIG)],
        "all large": [(slice(None), slice(None), BIG)],
    }[what]
    put = torch.zeros(x.shape, dtype=torch.bool, device="cuda")
    for r, c, v in spots:
        x[r, c] = v
        put[r, c] = True
    return put


WHAT = ["ring inf", "column -inf", "point inf", "inf and -inf", "nan", "ring large", "point large", "all large"]


def reached(put, T):
    """Points within T steps of a planted one."""
    for _ in range(T):
        n = put.clone()
        n[1:] |= put[:-1]
        n[:-1] |= put[1:]
        n[:, 1:] |= put[:, :-1]
        n[:, :-1] |= put[:, 1:]
        put = n
    return put


def compare(got, want, put, T, rounds):
    got = got.double()
    assert torch.equal(got.isnan(), want.isnan())
    assert torch.equal(got.isinf(), want.isinf()) and torch.equal(got[got.isinf()], want[want.isinf()])
    tol = 12 * T * 2.0 ** -24 + rounds * 2.0 ** -9
    rel = 12 * T * 2.0 ** -24 + rounds * 2.0 ** -8
    fin = want.isfinite()
    err = torch.where(fin, (got - want).abs(), 0.0)
    assert float(err.max()) <= rel * max(1.0, float(torch.where(fin, want.abs(), 0.0).max()))
    far = ~reached(put, T)
    assert float(torch.where(far, err, 0.0).max()) <= tol


@pytest.mark.parametrize("what", WHAT)
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_batch(what, dtype):
    """Untuned batches on the reassociated pipe: one strip and several, one segment and
    several, every remainder depth; a second replay of the plan with other inputs."""
    shapes = [(100, 100, 1), (300, 517, 8), (300, 517, 11), (64, 300, 7), (700, 90, 29), (500, 700, 45), (500, 701, 3)]
    torch.manual_seed(3)
    xs, ys, descs, puts = [], [], [], []
    for R, C, T in shapes:
        pad = (-C) % 8
        x, y = (torch.zeros((R, C + pad), dtype=dtype, device="cuda")[:, :C] for _ in range(2))
        x.copy_(torch.rand((R, C), device="cuda"))
        puts.append(plant(x, what))
        xs.append(x)
        ys.append(y)
        descs.append(binding.desc_for(x, y, T))
    arr, plan, L = (binding.sdfg_desc * len(descs))(*descs), ctypes.c_void_p(), binding.lib()
    torch.cuda.synchronize()
    binding.check(L.sdfg_batch_plan_create(ctypes.byref(plan), arr, len(descs), 64, None, 0))
    try:
        for again in range(3):
            if again == 2:  # the large values are gone
                for x, put in zip(xs, puts):
                    x[put] = 0.5
                    put[:] = False
            torch.cuda.synchronize()
            binding.check(L.sdfg_batch_plan_run(plan, torch.cuda.current_stream().cuda_stream))
            binding.check(L.sdfg_batch_plan_results(plan, arr, len(descs)))
            for (R, C, T), x, y, put in zip(shapes, xs, ys, puts):
                compare(y, jacobi2d64(x, T), put, T, T // 8 + 4 if dtype == torch.bfloat16 else 0)
            if again == 0:
                first = [y.clone() for y in ys]
            elif again == 1:
                assert all(torch.equal(a.nan_to_num(7.0), b.nan_to_num(7.0)) for a, b in zip(first, ys))
    finally:
        binding.check(L.sdfg_batch_plan_destroy(plan))
    assert binding.sdfg_device_error(True) == 0


@pytest.mark.parametrize("what", WHAT)
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("shape,T", [((100, 100), 1), ((100, 100), 11), ((300, 517), 3), ((300, 517), 8), ((300, 517), 45),
                                     ((1301, 1777), 31)])
def test_tiles(shape, T, dtype, what):
    """The register tiles: one tile and many, one pass and several, every kind of last pass."""
    x = torch.zeros((shape[0], shape[1] + 3), dtype=dtype, device="cuda")[:, :shape[1]]
    torch.manual_seed(5)
    x.copy_(torch.rand(shape, device="cuda"))
    put = plant(x, what)
    if what in ("point inf", "point large"):
        x[-1, :] = 1e-38  # the ring is copied exactly
    y = torch.empty_strided(x.shape, x.stride(), dtype=dtype, device="cuda")
    binding.jacobi2d(x, y, T)
    want = jacobi2d64(x, T)
    compare(y, want, put, T, 1 if dtype == torch.bfloat16 else 0)
    for got, was in ((y[0], x[0]), (y[-1], x[-1]), (y[:, 0], x[:, 0]), (y[:, -1], x[:, -1])):
        assert torch.equal(got.nan_to_num(7.0), was.nan_to_num(7.0))
    if what == "nan":
        x.nan_to_num_(0.25)
        x[3, 3] = BIG
        binding.jacobi2d(x, y, T)
    binding.jacobi2d(x, x, T)  # in place: the same
    assert torch.equal(x.nan_to_num(7.0), y.nan_to_num(7.0))
    assert binding.sdfg_device_error(True) == 0


def jacobi3d64(x, T):
    a = x.double()
    c = a[1:-1, 1:-1, 1:-1]
    for _ in range(T):
        s = (a[1:-1, :-2, 1:-1] + a[1:-1, 2:, 1:-1]) + (a[1:-1, 1:-1, :-2] + a[1:-1, 1:-1, 2:])
        c.copy_((c + (s + (a[:-2, 1:-1, 1:-1] + a[2:, 1:-1, 1:-1]))) / 7.0)
    return a


@pytest.mark.parametrize("what", ["shell inf", "point -inf", "inf and -inf", "nan", "shell large", "point large", "all large"])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("T", [1, 2, 3, 4, 7])
def test_box(T, dtype, what):
    """The 7-point stencil: one step, passes of 2 and of 3; 3.5e37, seven of which add up to an FP32 number."""
    torch.manual_seed(6)
    D, R, C = 21, 70, 263
    x = torch.rand((D, R, C + 1), device="cuda").to(dtype)[:, :, :C]
    put = torch.zeros(x.shape, dtype=torch.bool, device="cuda")
    every = (slice(None),) * 3
    for at, v in {
        "shell inf": [((0, slice(None), slice(None)), INF)],
        "point -inf": [((9, 33, 130), -INF)],
        "inf and -inf": [((slice(None), 0, slice(None)), INF), ((slice(None), slice(None), C - 1), -INF), ((5, 5, 5), INF)],
        "nan": [((11, 20, 121), NAN)],
        "shell large": [((D - 1, slice(None), slice(None)), 3.5e37), ((slice(None), slice(None), 0), -3.5e37)],
        "point large": [((9, 33, 119), 3.5e37)],
        "all large": [(every, 3.5e37)],
    }[what]:
        x[at] = v
        put[at] = True
    y = torch.empty_strided(x.shape, x.stride(), dtype=dtype, device="cuda")
    binding.jacobi3d(x, y, T)
    got, want = y.double(), jacobi3d64(x, T)
    assert torch.equal(got.isnan(), want.isnan())
    assert torch.equal(got.isinf(), want.isinf()) and torch.equal(got[got.isinf()], want[want.isinf()])
    # seven roundings a step and the pass's factors; BF16 one per pass or step
    rel = 12 * T * 2.0 ** -24 + (T * 2.0 ** -8 if dtype == torch.bfloat16 else 0.0)
    fin = want.isfinite()
    err = torch.where(fin, (got - want).abs(), 0.0)
    assert float(err.max()) <= rel * max(1.0, float(torch.where(fin, want.abs(), 0.0).max()))
    assert binding.sdfg_device_error(True) == 0
