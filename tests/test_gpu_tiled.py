"""The tiled and paired kernels on meshes that reach them (the small meshes of the other tests run the
small-mesh kernels): each case names the kernel its RK stages run and checks that the profiler's trace has
it, then guard words, the bounded wait, stream order, periodic axes and both extrapolations."""
import os

import numpy as np
import pytest

from oracle import conv as C
from oracle import extrap as X
from oracle import llg as L
from oracle import pbc as P
from oracle import rkf as R
from oracle import tensor as T
from oracle.tensor import demag_tensor
from paper_2308_08447_gb300 import workloads as W
from tests.gpu_util import TOL_FP32, e_inf, lib, to_dev, to_host
from tests.test_gpu_canary import Guarded
from tests.test_gpu_variants import has, kernels

pytestmark = pytest.mark.gpu

A, MS, CELL = 1.3e-11, 8e5, (3e-9, 3e-9, 3e-9)
STAGED, ROW, PAIR = ", 0, 2>", "row_kernel<", "row_pair_kernel<"   # staged: row_kernel's KIND 2 instances


@pytest.fixture(scope="module")
def g():
    return lib()


def periodic_kernel(n, per):
    """oracle.pbc.periodic_kernel with one image per side, summed one axis at a time (its single sum over
    all axes is quadratic in the mesh)."""
    terms = [P._axis_terms(n[d], per[d], 1) for d in range(3)]
    offs = [sorted({o for t in terms[d] for o, _ in t}) for d in range(3)]
    Z, Y, X = np.meshgrid(*(np.array(offs[d], float) for d in (2, 1, 0)), indexing="ij")
    K = demag_tensor(X, Y, Z, *CELL)
    for d in range(3):
        w = np.zeros((len(terms[d]), len(offs[d])))
        for b, t in enumerate(terms[d]):
            for o, weight in t:
                w[b, offs[d].index(o)] += weight
        K = np.moveaxis(np.tensordot(w, K, (1, 3 - d)), 0, 3 - d)
    return K


def stage_kernels(mesh, m):
    md = to_dev(m)
    return kernels(lambda: mesh.llg_step(md, 1, 1e-14))


# fields 16-, 4- and 8-byte aligned
@pytest.mark.parametrize("n,kernel,shift", [((64, 33, 21), PAIR, 0), ((64, 33, 21), PAIR, 1), ((250, 61, 3), PAIR, 2),
                                            ((63, 44, 17), PAIR, 0), ((256, 256, 1), ROW, 0), ((256, 256, 1), ROW, 1),
                                            ((250, 200, 1), ROW, 2), ((1024, 64, 1), STAGED, 0), ((640, 120, 4), "row_kernel<640", 0), ((640, 120, 4), "row_kernel<640", 1)])
def test_guard_words_untouched(g, n, kernel, shift):
    shape = (3, n[2], n[1], n[0])
    m0 = W.random_unit(n, 31)
    mesh = g.Mesh(n, CELL, MS, A_ex=A, alpha=0.1)
    assert has(stage_kernels(mesh, m0), kernel) and not has(stage_kernels(mesh, m0), "small_row")
    M, H, m = (Guarded(shape, v, shift) for v in (MS * m0, np.zeros(shape), m0))
    for call in (lambda: mesh.demag(M.t, H.t), lambda: mesh.effective_field(m.t, H.t), lambda: mesh.llg_rhs(m.t, H.t),
                 lambda: mesh.llg_step(m.t, 3, 1e-13), lambda: mesh.llg_step(m.t, 6, 1e-13, extrap=True),
                 lambda: mesh.rkf56_step(m.t, 1e-13), lambda: mesh.rkf56_step(m.t, 1e-13, extrap=True)):
        call()
        assert M.guards_intact() and H.guards_intact() and m.guards_intact()
    assert np.isfinite(m.t.cpu().numpy()).all()
    mesh.close()


def test_wait_that_runs_out_is_reported(g):
    n = (1024, 64, 1)                                # four rows per block, staged in shared memory
    m0 = W.vortex_noise(n, CELL, 3)
    out = {}
    for hook in ("1", "0"):
        os.environ["GBD_TEST_WAIT_TIMEOUT"] = hook
        try:
            mesh = g.Mesh(n, CELL, MS, A_ex=A, alpha=0.02)
        finally:
            os.environ.pop("GBD_TEST_WAIT_TIMEOUT", None)
        m = to_dev(m0)
        mesh.llg_step(m, 1, 1e-13)
        out[hook] = (mesh.device_status(), mesh.device_status(), to_host(m))
        mesh.close()
    assert out["1"][:2] == (g.GBD_ETIMEOUT, g.GBD_OK) and out["0"][:2] == (g.GBD_OK, g.GBD_OK)
    assert np.array_equal(out["1"][2], out["0"][2])


@pytest.mark.parametrize("extrap", [False, True])
@pytest.mark.parametrize("n,kernel,variants", [((1024, 64, 1), STAGED, (0, 1, 2)), ((64, 64, 16), PAIR, (0, 1)),
                                               ((640, 512, 1), "row_kernel<640", (1,)), ((32, 32, 8), "small_row", (0, 1))])
def test_writes_between_calls_are_seen(g, n, kernel, variants, extrap):
    # a torch kernel on the same stream reverses m between calls: seen as when the host waits each time
    import torch
    m0 = W.vortex_noise(n, CELL, 5)
    out = []
    for var in variants:
        for sync in (False, True):
            mesh = g.Mesh(n, CELL, MS, A_ex=A, alpha=0.02)
            if var == 1:
                assert has(stage_kernels(mesh, m0), kernel)
            g.gbd_mesh_set_tuning(mesh.handle, (var, 0, 0, 0))
            m = to_dev(m0)
            for _ in range(3):
                mesh.llg_step(m, 6, 1e-13, extrap=extrap)
                if sync:
                    torch.cuda.synchronize()
                m.mul_(-1.0)
                if sync:
                    torch.cuda.synchronize()
            out.append(to_host(m))
            mesh.close()
    assert np.isfinite(out[0]).all()
    for v in out[1:]:
        assert np.array_equal(v, out[0])


@pytest.mark.parametrize("n,per,kernel", [((256, 64, 8), (True, False, False), ROW), ((256, 256, 1), (True, True, False), ROW),
                                          ((64, 64, 16), (False, True, False), PAIR), ((64, 64, 16), (False, False, True), PAIR),
                                          ((1024, 64, 1), (False, True, False), STAGED)])
def test_periodic(g, n, per, kernel):
    alpha, dt = 0.1, 5e-14
    m = W.random_unit(n, 61)
    K = periodic_kernel(n, per)
    mesh = g.Mesh(n, CELL, MS, A_ex=A, alpha=alpha, pbc=per, pbc_images=1)
    assert has(stage_kernels(mesh, m), kernel)
    H = to_dev(np.full_like(m, np.nan))
    m64 = m.astype(np.float64)
    mesh.demag(to_dev(MS * m), H)
    assert e_inf(to_host(H), P.conv_periodic((MS * m).astype(np.float32).astype(np.float64), K, per)) <= TOL_FP32
    mesh.effective_field(to_dev(m), H)
    assert e_inf(to_host(H), P.effective_field(m64, K, CELL, MS, A, per)) <= TOL_FP32
    md = to_dev(m)
    mesh.llg_step(md, 3, dt)
    mesh.close()
    # FP32 rounding of the slopes (TOL_FP32 relative, dt |dm/dt| < 0.1) and of m, over three steps
    assert np.abs(to_host(md) - P.llg_run(m64, 3, dt, K, CELL, MS, A, alpha, per)).max() <= 6e-6


@pytest.mark.parametrize("n,kernel", [((1024, 64, 1), STAGED), ((256, 256, 1), ROW), ((250, 61, 3), PAIR), ((63, 44, 17), PAIR)])
def test_extrapolated_runs(g, n, kernel):
    alpha, dt, steps = 0.1, 5e-14, 9
    m = W.random_unit(n, 41)
    m64 = m.astype(np.float64)
    N = T.tensor_all_offsets(n, CELL)
    mesh = g.Mesh(n, CELL, MS, A_ex=A, alpha=alpha)
    assert has(stage_kernels(mesh, m), kernel)
    one, split = to_dev(m), to_dev(m)
    mesh.llg_step(one, steps, dt, extrap=True)
    mesh.llg_step(split, 6, dt, extrap=True)
    mesh.llg_step(split, steps - 6, dt, extrap=True, cont=True)
    assert np.array_equal(to_host(one), to_host(split))
    want, nev = X.llg_run_extrap(m64, steps, dt, N, CELL, MS, A, alpha)
    assert nev == 16 + (steps - 4)
    assert np.abs(to_host(one) - want).max() < 2e-5      # as for the small meshes
    md = to_dev(m)
    for i in range(8):
        mesh.rkf56_step(md, dt, extrap=True, cont=i > 0)
    demag = lambda v: MS * C.fft_conv(v, N)
    rest = lambda v, hd: L.llg_rhs(v, hd + L.exchange_field(v, CELL, MS, A), alpha)
    want, hist = m64, []
    for i in range(8):
        want, _, hd = R.rkf56_step_extrap(want, dt, demag, rest, [(-(q + 1) * dt, h) for q, h in enumerate(hist)])
        hist = [hd] + hist[:4]
    assert np.abs(to_host(md) - want).max() < 5e-5
    mesh.close()
