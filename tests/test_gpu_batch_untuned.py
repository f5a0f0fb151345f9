"""Untuned fixed-step batch plans whose size takes them to the reassociated
persistent kernel (2^18 points and more), on both sides of each line of the rule:
uneven grids, thin ones, one pitched, one unaligned (staged), one in place, one
with nothing to do; every grid whole against the FP64 oracle, the ring exact, and
a second replay equal to the first.

Tolerance: a step is at most five FP32 roundings of sums of weights that add up
to one, each at most 2^-24 of the largest value (1), and does not amplify what
it is given; scaling and the ring's rounded factors add at most ten per pass of
four steps or more, remainder passes of one and two steps as many again.  Hence
12 T 2^-24, and for BF16 a rounding of 2^-9 per pass."""
import ctypes

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


SMALL = [(300, 517), (700, 401), (3, 900), (900, 3), (2, 40), (64, 64), (129, 1000), (16, 113)]
LARGE = SMALL + [(1800, 1701), (1702, 1900), (1601, 1750), (1500, 2048)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("shapes", [SMALL, LARGE])
def test_untuned_plan(shapes, dtype):
    assert sum(r * c for r, c in shapes) >= (1 << 18 if shapes is SMALL else 12_000_000 - 100_000)
    rng = np.random.default_rng(len(shapes))
    xs, ys, descs, Ts, inputs = [], [], [], [], []
    for i, (R, C) in enumerate(shapes):
        pad = (-C) % 8 + (8 if i == 1 else 0) if i != 6 else 3
        x = torch.zeros((R, C + pad), dtype=dtype, device="cuda")[:, :C]
        x.copy_(torch.from_numpy(rng.random((R, C))))
        y = x if i == 5 else torch.zeros((R, C + pad), dtype=dtype, device="cuda")[:, :C]
        T = 0 if i == 7 else 5 + 7 * (i % 6)
        inputs.append(x)  # the plan reads it at every replay
        xs.append(x.double().cpu().numpy())
        ys.append(y)
        Ts.append(T)
        descs.append(binding.desc_for(x, y, T))
    L = binding.lib()
    arr = (binding.sdfg_desc * len(descs))(*descs)
    plan = ctypes.c_void_p()
    torch.cuda.synchronize()
    binding.check(L.sdfg_batch_plan_create(ctypes.byref(plan), arr, len(descs), 64, None, 0))
    try:
        start = ys[5].clone()
        first = None
        for _ in range(2):
            ys[5].copy_(start)
            torch.cuda.synchronize()
            binding.check(L.sdfg_batch_plan_run(plan, torch.cuda.current_stream().cuda_stream))
            binding.check(L.sdfg_batch_plan_results(plan, arr, len(descs)))
            if first is None:
                first = [y.clone() for y in ys]
            assert all(torch.equal(a, b) for a, b in zip(first, ys))
    finally:
        binding.check(L.sdfg_batch_plan_destroy(plan))
    assert binding.sdfg_device_error(True) == 0
    for (R, C), x, y, T in zip(shapes, xs, ys, Ts):
        got = y.double().cpu().numpy()
        want = oracle.jacobi2d(x, T, threads=0)
        tol = 12 * T * 2.0 ** -24 + (2.0 ** -9 * (T // 8 + 4) if dtype == torch.bfloat16 else 0.0)
        assert np.abs(got - want).max() <= tol, (R, C, T, np.abs(got - want).max())
        for a, b in ((got[0], x[0]), (got[-1], x[-1]), (got[:, 0], x[:, 0]), (got[:, -1], x[:, -1])):
            assert np.array_equal(a, b)
