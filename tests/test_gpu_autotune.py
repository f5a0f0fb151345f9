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
