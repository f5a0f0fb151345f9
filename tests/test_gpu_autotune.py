"""The autotuners where the class of their shape is tuned already: a preset cache
file (read once per process, hence a child process per test) must not take the
place of what an untuned call runs among the candidates."""
import os
import subprocess
import sys

import pytest

from paper_1902_10345_gb300 import build

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def child(tmp_path, entry, code):
    build.build()
    cache = tmp_path / "cache.txt"
    cache.write_text(entry + "\n")
    env = dict(os.environ, SDFG_AUTOTUNE_CACHE=str(cache), PYTHONPATH=ROOT)
    head = "import torch\nfrom paper_1902_10345_gb300 import binding\ntorch.zeros(1, device='cuda')\n"
    r = subprocess.run([sys.executable, "-c", head + code], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.split(), cache.read_text().split()


def test_retuning_a_class_times_the_tiles(tmp_path):
    """FP64 256 x 256: no candidate but the untuned call launches the tiles, so
    their family's count tells whether that candidate ran as itself."""
    out, _ = child(tmp_path, "2 8 8 2 4 96 4", """
binding.sdfg_stats_enable(True)
binding.sdfg_autotune(256, 256, 8, binding.SDFG_F64, torch.cuda.current_stream().cuda_stream)
print(binding.sdfg_stats_get("resident")[0])
""")
    assert out == ["2"]  # warm-up and timed run


BATCH = """
xs = [torch.rand((400, 400), device='cuda') for _ in range(8)]
ys = [torch.empty_like(x) for x in xs]
descs = [binding.desc_for(x, y, 16) for x, y in zip(xs, ys)]
torch.cuda.synchronize()
binding.sdfg_stats_enable(True)
"""


def test_retuning_a_batch_times_the_untuned_plan(tmp_path):
    """Aligned grids below the chain kernel's size: only the untuned plan copies
    rings, so the copies' count tells that it is a candidate."""
    out, cache = child(tmp_path, "0 -4 -18 3 8 96 4", BATCH + """
best = binding.sdfg_autotune_batch(descs, 64)
print(binding.sdfg_stats_get("copy")[0], best.kernel, best.k, best.seg_rows, best.warps)
""")
    assert out[0] == "2"  # warm-up and timed run
    assert cache == ["0", "-4", "-18"] + out[1:]


def test_a_cached_untuned_choice_is_the_untuned_plan(tmp_path):
    out, _ = child(tmp_path, "0 -4 -18 0 0 0 0", BATCH + """
binding.check(binding.sdfg_jacobi2d_batch(descs, 64))
print(binding.sdfg_stats_get("copy")[0])
""")
    assert out == ["1"]
