"""The file of tuning choices (GBD_AUTOTUNE_CACHE): lines without the generation of the kernels they were
timed on, which older versions wrote, are passed over; the lines this version writes are applied. The
file is read once per process, so each step runs in a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TUNE = """
import sys
from tests.gpu_util import lib
g = lib()
mesh = g.Mesh((64, 64, 16), (3e-9, 3e-9, 3e-9), 8e5)
print(*mesh.autotune(), *g.gbd_mesh_plan_dims(mesh.handle)[:2])
"""


def tune(path):
    env = dict(os.environ, GBD_AUTOTUNE_CACHE=str(path))
    out = subprocess.run([sys.executable, "-c", TUNE], cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, out.stderr[-2000:]
    return [int(v) for v in out.stdout.split()]


def test_lines_of_other_generations_are_passed_over(tmp_path):
    path = tmp_path / "tune.txt"
    key = "64 64 16 0 128 128 0"
    old = [key + " 3 0 1 1 0 1\n", "gbd1 " + key + " 3 0 1 1 0 1\n", "no choice\n", "\n"]
    path.write_text("".join(old))
    first = tune(path)                                   # tuned anew, and appended
    lines = path.read_text().splitlines(keepends=True)
    assert lines[:len(old)] == old and len(lines) == len(old) + 1
    gen, new = lines[-1].split(" ", 1)
    assert gen.startswith("gbd") and gen != "gbd1" and new.startswith(key)
    assert tune(path) == first and len(path.read_text().splitlines()) == len(lines)   # read back
    path.write_text(gen + " " + key + " 2 0 1 1 0 1\n")
    assert tune(path) == [2, 0, 1, 1, 128, 128]
