"""Tile variants on meshes whose launches depend on them: every row, y and z variant runs the kernel it
stands for (named by the profiler's trace) and all give the same bits, in one call and split over calls;
and a field's alignment, which chooses between a kernel's epilogues, does not change its bits either."""
import numpy as np
import pytest

from paper_2308_08447_gb300 import workloads as W
from tests.gpu_util import lib, to_dev, to_host

pytestmark = pytest.mark.gpu

CELL, MS, DT = (3e-9, 3e-9, 3e-9), 8e5, 5e-14
DEFAULT = (1, 0, 0, 0)


@pytest.fixture(scope="module")
def g():
    return lib()


def traced(call):
    """Names of the kernels that call() launches."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as trace:
        call()
        torch.cuda.synchronize()
    return {e.name.replace("void ", "") for e in trace.events()}


def kernels(call):
    """Names of the library's kernels that call() launches. (A process's first trace may come back empty;
    without any trace of a torch kernel either, this machine has none to give.)"""
    import torch
    for _ in range(3):
        names = {n for n in traced(call) if "gbd::" in n}
        if names:
            return names
    x = torch.zeros(1 << 10, device="cuda")
    if not traced(lambda: x.add_(1.0)):
        pytest.skip("no kernel trace on this machine")
    return names


def has(names, part):
    return any(part in n for n in names)


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


@pytest.mark.parametrize("n", [(256, 256, 1), (512, 512, 1), (256, 1024, 1), (1024, 512, 1), (128, 128, 16)])
def test_row_variants(g, n):
    m = W.random_unit(n, 51)
    mesh = g.Mesh(n, CELL, MS, A_ex=1.3e-11, alpha=0.05)
    base = run(mesh, m)
    md = to_dev(m)
    for v in (0, 2, 3):
        g.gbd_mesh_set_tuning(mesh.handle, (v,) + DEFAULT[1:])
        for a, b in zip(base, run(mesh, m)):
            assert np.array_equal(a, b)
        names = kernels(lambda: mesh.llg_step(md, 1, DT))
        assert has(names, "row_kernel" if v == 0 else "row_pipe_kernel") and not has(names, "row_pair") and not has(names, "small_row")
    mesh.close()


@pytest.mark.parametrize("n", [(64, 48, 2), (256, 256, 1), (64, 64, 16), (250, 62, 4), (1024, 64, 1), (640, 128, 4), (1000, 60, 1)])
def test_alignment(g, n):
    m = W.random_unit(n, 53)
    mesh = g.Mesh(n, CELL, MS, A_ex=1.3e-11, alpha=0.05, Hext=(1e4, 0.0, 2e4))
    base = run(mesh, m)
    for shift in (1, 2):
        for a, b in zip(base, run(mesh, m, shift)):
            assert np.array_equal(a, b)
    mesh.close()


def test_y_and_z_variants(g):
    n = (128, 128, 16)
    m = W.random_unit(n, 52)
    mesh = g.Mesh(n, CELL, MS, A_ex=1.3e-11, alpha=0.05)
    base, ran = run(mesh, m), []
    H = to_dev(m)
    for v in ((1, 0, 0, 0), (1, 0, 1, 1)):
        g.gbd_mesh_set_tuning(mesh.handle, v)
        for a, b in zip(base, run(mesh, m)):
            assert np.array_equal(a, b)
        names = kernels(lambda: mesh.demag(to_dev(m), H))
        ran.append({n for n in names if "y_pass" in n or "z_conv" in n})
    assert len(ran[0]) == len(ran[1]) == 3 and not ran[0] & ran[1]
    mesh.close()
