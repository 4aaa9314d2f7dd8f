"""The bits of a result do not depend on a field's alignment, which chooses between a kernel's epilogues."""
import numpy as np
import pytest

from paper_2308_08447_gb300 import workloads as W
from tests.gpu_util import lib, to_dev, to_host

pytestmark = pytest.mark.gpu

CELL, MS, DT = (3e-9, 3e-9, 3e-9), 8e5, 5e-14


@pytest.fixture(scope="module")
def g():
    return lib()


def run(mesh, m, shift=0):
    """demag, H_eff, dm/dt, four RK4 steps in calls of 3 and 1, one RKF5(6) step, six extrapolated steps;
    the fields `shift` floats behind a 16-byte boundary."""
    def dev(v):
        t = to_dev(np.zeros(v.size + shift))[shift:].view(v.shape)
        return t.copy_(to_dev(v))

    out = []
    for f in (mesh.demag, mesh.effective_field, mesh.llg_rhs):
        H = dev(np.full_like(m, np.nan))
        f(dev(m), H)
        out.append(to_host(H))
    for f in (lambda v: (mesh.llg_step(v, 3, DT), mesh.llg_step(v, 1, DT)), lambda v: mesh.rkf56_step(v, DT),
              lambda v: mesh.llg_step(v, 6, DT, extrap=True)):
        md = dev(m)
        f(md)
        out.append(to_host(md))
    return out


@pytest.mark.parametrize("n", [(64, 48, 2), (256, 256, 1), (64, 64, 16), (250, 62, 4), (1024, 64, 1), (640, 128, 4), (1000, 60, 1)])
def test_alignment(g, n):
    m = W.random_unit(n, 53)
    mesh = g.Mesh(n, CELL, MS, A_ex=1.3e-11, alpha=0.05, Hext=(1e4, 0.0, 2e4))
    base = run(mesh, m)
    for shift in (1, 2):
        for a, b in zip(base, run(mesh, m, shift)):
            assert np.array_equal(a, b)
    mesh.close()
