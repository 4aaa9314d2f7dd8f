"""A mesh that the autotuner moved onto its power-of-two plan keeps a status word of its own: a wait that
runs out on it (GBD_TEST_WAIT_TIMEOUT) is reported by this mesh, once, and by no other mesh that was
given the memory of its old plan. The move is made certain by the tuning cache's file, which a process
reads once, so the check runs in a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHECK = """
import os, re, sys
from paper_2308_08447_gb300 import workloads as W
from tests.gpu_util import lib, to_dev, to_host
g = lib()
path = os.environ["GBD_AUTOTUNE_CACHE"]
n, cell = (320, 48, 1), (3e-9, 3e-9, 3e-9)     # x length 320, on powers of two 512

def mesh():
    return g.Mesh(n, cell, 8e5, A_ex=1.3e-11, alpha=0.05)

if sys.argv[1] == "write":                     # a line of this version's format
    m = g.Mesh((64, 64, 16), cell, 8e5)
    m.autotune()
    text = open(path).read().splitlines()[0]
    gen = text.split()[0]
    open(path, "w").write(gen + " 320 48 1 0 640 96 0 1 0 1 0 1 1\\n")
    sys.exit(0)
os.environ["GBD_TEST_WAIT_TIMEOUT"] = "1"
a = mesh()
del os.environ["GBD_TEST_WAIT_TIMEOUT"]
assert g.gbd_mesh_plan_dims(a.handle)[:2] == (640, 96)
a.autotune()
assert g.gbd_mesh_plan_dims(a.handle)[:2] == (1024, 128)
others = [mesh() for _ in range(4)]            # may be given what the move freed
m = to_dev(W.vortex_noise(n, cell, 3))
a.llg_step(m, 1, 5e-14)
to_host(m)
assert [o.device_status() for o in others] == [g.GBD_OK] * 4
assert (a.device_status(), a.device_status()) == (g.GBD_ETIMEOUT, g.GBD_OK)
"""


def test_status_word_of_a_moved_mesh(tmp_path):
    env = dict(os.environ, GBD_AUTOTUNE_CACHE=str(tmp_path / "tune.txt"))
    for step in ("write", "check"):
        out = subprocess.run([sys.executable, "-c", CHECK, step], cwd=ROOT, env=env, capture_output=True, text=True,
                             timeout=600)
        assert out.returncode == 0, out.stderr[-2000:]
