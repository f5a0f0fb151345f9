"""Performance cases: the library's work as a program calls it, over the sizes its users run.

Every case goes through the public entry points of ``paper_1902_10345_gb300.binding`` with their defaults: a program
that has not run the autotuner.  The kinds:

* ``jacobi2d`` -- one grid, T steps (FP32, BF16 or FP64 storage; rows pitched or odd);
* ``batch``    -- many uneven grids through a batch plan that is built once and replayed;
* ``serve``    -- Laplace requests solved to a relative residual by the continuous-batching server;
* ``jacobi3d`` -- the 7-point stencil on a box;
* ``sor2d``    -- red-black SOR on one grid.

Sizes are the repository's own workloads (256^2, the paper's 2048^2, 8192^2, 16384^2, the 512-grid batch, 512^3) and
ragged ones between.
"""
import ctypes
import math
import random

import torch

from paper_1902_10345_gb300 import binding

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f64": torch.float64}
SIZE = {"f32": 4, "bf16": 2, "f64": 8}


# ---- the cases --------------------------------------------------------------------------------------------------------

def _grid(name, dtype, rows, cols, T, field="uniform", pad=0):
    return {"name": name, "kind": "jacobi2d", "dtype": dtype, "rows": rows, "cols": cols, "T": T, "field": field, "pad": pad}


def _box(name, dtype, depth, rows, cols, T):
    return {"name": name, "kind": "jacobi3d", "dtype": dtype, "depth": depth, "rows": rows, "cols": cols, "T": T}


def _sor(name, dtype, rows, cols, T, omega):
    return {"name": name, "kind": "sor2d", "dtype": dtype, "rows": rows, "cols": cols, "T": T, "omega": omega}


def listed():
    return [
        # a small solve inside a larger program: launches and latency
        _grid("jacobi2d f32 256", "f32", 256, 256, 100),
        # the double-precision parity workload: one small grid, exact order
        _grid("jacobi2d f64 256", "f64", 256, 256, 100),
        # a ragged grid whose odd row pitch a caller did not choose for this library
        _grid("jacobi2d f32 odd", "f32", 1301, 1777, 150, pad=2),
        # the paper's Jacobi workload: fits in L2
        _grid("jacobi2d f32 2048", "f32", 2048, 2048, 1024, field="zero ring"),
        # the headline workload
        _grid("jacobi2d f32 8192", "f32", 8192, 8192, 1000),
        # the precision workload's storage type and size: the largest grid
        _grid("jacobi2d bf16 16384", "bf16", 16384, 16384, 500, field="waves"),
        # the uneven batch: parameter studies, ensembles
        {"name": "batch 512", "kind": "batch", "dtype": "f32", "n": 512, "lo": 64, "hi": 2048, "t_lo": 50, "t_hi": 500, "shapes": 0},
        # a burst of served requests of mixed size
        {"name": "serve 24", "kind": "serve", "n": 24, "lo": 32, "hi": 768, "tol": 1e-6, "cap": 20000, "shapes": 1},
        # the 3-D workload
        _box("jacobi3d f32 512", "f32", 512, 512, 512, 100),
        # a ragged double-precision box of ordinary size
        _box("jacobi3d f64 odd", "f64", 129, 150, 131, 30),
        # the SOR workload's grid
        _sor("sor2d f32 8192", "f32", 8192, 8192, 200, 1.9),
        # an ordinary ragged SOR solve
        _sor("sor2d f32 odd", "f32", 777, 1023, 100, 1.7),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["jacobi2d", "jacobi2d", "jacobi2d", "jacobi2d", "batch", "serve", "jacobi3d", "jacobi3d", "sor2d", "sor2d"])
    if kind == "jacobi2d":
        dtype = rng.choice(["f32", "f32", "f32", "bf16", "f64"])
        hi = 4096 if dtype == "f64" else 12288
        rows, cols = _log_int(rng, 48, hi), _log_int(rng, 48, hi)
        most = 2e9 if dtype == "f64" else 60e9          # point updates
        T = max(8, min(_log_int(rng, 16, 1100), int(most / (rows * cols))))
        field = rng.choice(["uniform", "zero ring"]) if dtype != "bf16" else "waves"
        return {"kind": kind, "dtype": dtype, "rows": rows, "cols": cols, "T": T, "field": field, "pad": rng.choice([0, 0, -1, 3])}
    if kind == "batch":
        n = _log_int(rng, 8, 384)
        hi = 2048 if n > 16 else _log_int(rng, 256, 2048)
        return {"kind": kind, "dtype": rng.choice(["f32", "f32", "bf16"]), "n": n, "lo": 64, "hi": hi, "t_lo": 50, "t_hi": 500,
                "shapes": rng.randrange(1 << 20)}
    if kind == "serve":
        return {"kind": kind, "n": rng.randint(4, 24), "lo": 32, "hi": _log_int(rng, 128, 768), "tol": rng.choice([1e-5, 1e-6]),
                "cap": 20000, "shapes": rng.randrange(1 << 20)}
    if kind == "jacobi3d":
        dtype = rng.choice(["f32", "f32", "bf16", "f64"])
        d, r, c = (_log_int(rng, 24, 400 if dtype != "f64" else 200) for _ in range(3))
        T = max(4, min(_log_int(rng, 8, 128), int((8e9 if dtype != "f64" else 5e8) / (d * r * c))))
        return {"kind": kind, "dtype": dtype, "depth": d, "rows": r, "cols": c, "T": T}
    dtype = rng.choice(["f32", "f32", "bf16", "f64"])
    rows, cols = (_log_int(rng, 48, 6000 if dtype != "f64" else 1500) for _ in range(2))
    T = max(4, min(_log_int(rng, 8, 400), int((2e10 if dtype != "f64" else 5e8) / (rows * cols))))
    return {"kind": kind, "dtype": dtype, "rows": rows, "cols": cols, "T": T, "omega": rng.choice([1.0, 1.5, 1.9])}


# ---- inputs -----------------------------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _field(case, seed):
    """The initial grid in FP64 or the storage type."""
    R, C, g = case["rows"], case["cols"], _gen(seed)
    if case.get("field", "uniform") == "waves":  # 0.5 + 8 sinusoids + noise, as the precision workload
        r = random.Random(seed)
        n = max(R, C)
        k_max = max(1, n // 256)                  # wavelengths of 256 cells and more
        y = torch.arange(R, dtype=torch.float32, device="cuda")[:, None] / n
        x = torch.arange(C, dtype=torch.float32, device="cuda")[None, :] / n
        w = [r.random() + 0.1 for _ in range(8)]
        f = torch.rand((R, C), generator=g, device="cuda").mul_(0.1).add_(0.45)
        for m in range(8):
            a, b, p = 2 * math.pi * r.randint(1, k_max), 2 * math.pi * r.randint(1, k_max), r.uniform(0, 2 * math.pi)
            f.addcmul_(torch.cos(b * y + p), torch.sin(a * x), value=0.5 * w[m] / sum(w))
            f.addcmul_(torch.sin(b * y + p), torch.cos(a * x), value=0.5 * w[m] / sum(w))
        return f
    f = torch.rand((R, C), generator=g, device="cuda", dtype=torch.float64 if case.get("dtype") == "f64" else torch.float32)
    if case.get("field") == "zero ring":
        f[0], f[-1], f[:, 0], f[:, -1] = 0, 0, 0, 0
    return f


def _pitched(f, dtype, pad):
    """`f` in storage type, rows `pad` elements apart beyond the columns (-1: up to a multiple of 16 bytes)."""
    R, C = f.shape
    a = 16 // SIZE[dtype]
    ld = (C + a - 1) // a * a if pad < 0 else C + pad
    buf = torch.zeros((R, ld), dtype=DTYPES[dtype], device="cuda")
    buf[:, :C].copy_(f)
    return buf[:, :C]


def _specs(case):
    """[(rows, cols, T, ld, offset)] of a batch or a burst, and the elements of all grids together (each starts on 256 bytes)."""
    r, at, out = random.Random(case["shapes"]), 0, []
    a = 16 // SIZE[case.get("dtype", "f32")]
    for _ in range(case["n"]):
        rows, cols = _log_int(r, case["lo"], case["hi"]), _log_int(r, case["lo"], case["hi"])
        T = r.randint(case["t_lo"], case["t_hi"]) if "t_lo" in case else case["cap"]
        ld = (cols + a - 1) // a * a
        out.append((rows, cols, T, ld, at))
        at += (rows * ld + 127) // 128 * 128
    return out, at


def _views(flat, specs):
    return [flat[at:at + rows * ld].view(rows, ld)[:, :cols] for rows, cols, T, ld, at in specs]


def _batch_input(case, seed):
    specs, n = _specs(case)
    flat = torch.zeros(n, dtype=DTYPES[case["dtype"]], device="cuda")
    noise = torch.rand(n, generator=_gen(seed), device="cuda").to(flat.dtype)
    for v, w in zip(_views(flat, specs), _views(noise, specs)):
        v.copy_(w)
    return specs, flat


def _serve_input(case, seed):
    """Boundary x^2 - y^2 on the unit square plus noise of amplitude 1e-3, zero interior."""
    specs, n = _specs(case)
    flat = torch.zeros(n, device="cuda")
    noise = torch.rand(n, generator=_gen(seed), device="cuda").mul_(2e-3).sub_(1e-3)
    for v, w in zip(_views(flat, specs), _views(noise, specs)):
        R, C = v.shape
        y = torch.arange(R, dtype=torch.float32, device="cuda")[:, None] / (R - 1)
        x = torch.arange(C, dtype=torch.float32, device="cuda")[None, :] / (C - 1)
        v.copy_(x * x - y * y + w)
        v[1:-1, 1:-1] = 0
    return specs, flat


class _Plan:
    """A batch plan and what it works on; destroyed with the state."""

    def __init__(self, case, seed):
        self.specs, self.inp = _batch_input(case, seed)
        self.out = torch.zeros_like(self.inp)
        descs = [binding.desc_for(x, y, s[2]) for x, y, s in zip(_views(self.inp, self.specs), _views(self.out, self.specs), self.specs)]
        self.arr = (binding.sdfg_desc * len(descs))(*descs)
        self.plan = ctypes.c_void_p()
        torch.cuda.current_stream().synchronize()
        binding.check(binding.lib().sdfg_batch_plan_create(ctypes.byref(self.plan), self.arr, len(descs), 64, None,
                                                           torch.cuda.current_stream().cuda_stream))

    def __del__(self):
        if self.plan:
            binding.lib().sdfg_batch_plan_destroy(self.plan)


class _Server:
    """A server and a burst of requests; destroyed with the state."""

    def __init__(self, case, seed):
        self.specs, self.inp = _serve_input(case, seed)
        self.out = torch.zeros_like(self.inp)
        self.descs = [binding.desc_for(x, y, s[2], case["tol"])
                      for x, y, s in zip(_views(self.inp, self.specs), _views(self.out, self.specs), self.specs)]
        self.handle = ctypes.c_void_p()
        torch.cuda.current_stream().synchronize()
        binding.check(binding.lib().sdfg_server_create(ctypes.byref(self.handle), 4 << 30, 64, 256, 64, 0))

    def __del__(self):
        if self.handle:
            binding.lib().sdfg_server_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return case, _Plan(case, seed)
    if kind == "serve":
        return case, _Server(case, seed)
    x = _storage(case, seed)
    return case, (x, torch.empty_strided(x.size(), x.stride(), dtype=x.dtype, device="cuda"))


def _storage(case, seed):
    if case["kind"] == "jacobi3d":
        shape = (case["depth"], case["rows"], case["cols"])
        return torch.rand(shape, generator=_gen(seed), device="cuda", dtype=torch.float64 if case["dtype"] == "f64" else torch.float32).to(DTYPES[case["dtype"]])
    return _pitched(_field(case, seed), case["dtype"], case.get("pad", 0))


# ---- one pass ---------------------------------------------------------------------------------------------------------

def run(state):
    case, s = state
    kind = case["kind"]
    if kind == "jacobi2d":
        binding.jacobi2d(s[0], s[1], case["T"])
        return s[1]
    if kind == "jacobi3d":
        binding.jacobi3d(s[0], s[1], case["T"])
        return s[1]
    if kind == "sor2d":
        binding.sor2d(s[0], s[1], case["T"], case["omega"])
        return s[1]
    L = binding.lib()
    if kind == "batch":
        binding.check(L.sdfg_batch_plan_run(s.plan, torch.cuda.current_stream().cuda_stream))
        return s.out
    ids = []
    for d in s.descs:
        rid = ctypes.c_uint64()
        binding.check(L.sdfg_server_submit(s.handle, ctypes.byref(d), ctypes.byref(rid)))
        ids.append(rid.value)
    binding.check(L.sdfg_server_drain(s.handle, 60000))
    got = []
    for rid in ids:
        d = binding.sdfg_desc()
        binding.check(L.sdfg_server_poll(s.handle, rid, ctypes.byref(d)))
        got.append(d)
    return {"grids": s.out, "steps": torch.tensor([d.steps_done for d in got]),
            "residuals": torch.tensor([d.rel_residual for d in got], dtype=torch.float64)}


# ---- what a pass cannot do without ------------------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        specs, _ = _specs(case)
        S = SIZE[case.get("dtype", "f32")]
        flops = sum(5.0 * (r - 2) * (c - 2) * T for r, c, T, _, _ in specs) if kind == "batch" else 0.0
        return {"bytes": 2.0 * S * sum(r * c for r, c, *_ in specs), "flops": flops}
    pts, S = case["rows"] * case["cols"], SIZE[case["dtype"]]
    inner = (case["rows"] - 2) * (case["cols"] - 2)
    if kind == "jacobi3d":
        pts, inner = pts * case["depth"], inner * (case["depth"] - 2)
    per = {"jacobi2d": 5.0, "jacobi3d": 7.0, "sor2d": 6.0}[kind]
    return {"bytes": 2.0 * S * pts, "flops": per * inner * case["T"]}


# ---- the same in 64 bits, in plain torch ------------------------------------------------------------------------------

def _jacobi2d64(a, T):
    t, w = torch.empty_like(a[1:-1, 1:-1]), torch.empty_like(a[1:-1, 1:-1])
    for _ in range(T):
        torch.add(a[:-2, 1:-1], a[2:, 1:-1], out=t)
        torch.add(a[1:-1, :-2], a[1:-1, 2:], out=w)
        t.add_(w).add_(a[1:-1, 1:-1])
        torch.mul(t, 0.2, out=a[1:-1, 1:-1])
    return a


def _jacobi3d64(a, T):
    c = a[1:-1, 1:-1, 1:-1]
    t, w = torch.empty_like(c), torch.empty_like(c)
    for _ in range(T):
        torch.add(a[1:-1, :-2, 1:-1], a[1:-1, 2:, 1:-1], out=t)
        torch.add(a[1:-1, 1:-1, :-2], a[1:-1, 1:-1, 2:], out=w)
        t.add_(w)
        torch.add(a[:-2, 1:-1, 1:-1], a[2:, 1:-1, 1:-1], out=w)
        t.add_(w).add_(c)
        torch.mul(t, 1.0 / 7.0, out=c)
    return a


def _sor64(a, T, omega):
    R, C = a.shape
    i, j = torch.arange(1, R - 1, device=a.device)[:, None], torch.arange(1, C - 1, device=a.device)[None, :]
    colour = [(i + j) % 2 == p for p in (0, 1)]
    c = a[1:-1, 1:-1]
    t, w = torch.empty_like(c), torch.empty_like(c)
    for _ in range(T):
        for p in (0, 1):
            torch.add(a[:-2, 1:-1], a[2:, 1:-1], out=t)
            torch.add(a[1:-1, :-2], a[1:-1, 2:], out=w)
            t.add_(w).mul_(0.25 * omega)
            torch.mul(c, 1.0 - omega, out=w)
            w.add_(t)
            c.copy_(torch.where(colour[p], w, c))
    return a


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return None  # the grid returned depends on the step at which the residual test of the storage type stops
    if kind == "batch":
        specs, flat = _batch_input(case, seed)
        flat = flat.double()
        for v, s in zip(_views(flat, specs), specs):
            _jacobi2d64(v, s[2])
        return flat
    x = _storage(case, seed).double()
    if kind == "jacobi2d":
        return _jacobi2d64(x, case["T"])
    if kind == "jacobi3d":
        return _jacobi3d64(x, case["T"])
    return _sor64(x, case["T"], case["omega"])
