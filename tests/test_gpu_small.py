"""Meshes at the edges of the small-mesh kernels (one or two rows per block, one kx column per
block), against the FP64 oracle: lengths at the ends of the radix plans, 2 to 8 layers (every z
length in registers), odd sides, row counts that do not fill the last block, periodic x and y,
staged and unstaged field rows, and the same convolution run pass by pass (bit-identical)."""
import numpy as np
import pytest

from oracle import conv as C
from oracle import llg as L
from oracle import pbc as P
from oracle import tensor as T
from paper_2308_08447_gb300 import workloads as W
from tests.gpu_util import TOL_FP32, e_inf, lib, to_dev, to_host

pytestmark = pytest.mark.gpu

A, ALPHA, MS, DT = 1.3e-11, 0.05, 8e5, 5e-14


@pytest.fixture(scope="module")
def g():
    return lib()


@pytest.mark.parametrize("n", [(16, 16, 1), (9, 16, 8), (17, 9, 2), (95, 33, 3), (160, 20, 5), (61, 80, 4), (200, 150, 1),
                               (313, 21, 7), (20, 200, 6), (256, 17, 1), (640, 9, 1), (1250, 3, 2), (12, 500, 2)])
def test_demag_and_step(g, n):
    cell = (3e-9, 3e-9, 3e-9)
    m = W.random_unit(n, 7)
    N = T.tensor_all_offsets(n, cell)
    mesh = g.Mesh(n, cell, MS, A_ex=A, alpha=ALPHA)
    M = (MS * m).astype(np.float32)
    H = to_dev(np.full_like(m, np.nan))
    mesh.demag(to_dev(M), H)
    want = C.fft_conv(M.astype(np.float64), N)
    assert e_inf(to_host(H), want) <= TOL_FP32
    # pass by pass: events around each pass split the one-launch convolution
    H2 = to_dev(np.full_like(m, np.nan))
    g.gbd_mesh_set_timing(mesh.handle, True)
    mesh.demag(to_dev(M), H2)
    g.gbd_mesh_read_timing(mesh.handle)
    g.gbd_mesh_set_timing(mesh.handle, False)
    assert np.array_equal(to_host(H), to_host(H2))
    # RK4 with the fields 16-byte aligned (staged rows) and 4 bytes off (not staged)
    m64 = m.astype(np.float64)
    ref = L.rk4_step(m64, DT, lambda v: L.rhs(v, N, cell, MS, A, ALPHA))
    md = to_dev(m)
    buf = to_dev(np.zeros(m.size + 1))
    off = buf[1:].view(m.shape)
    off.copy_(md)
    mesh.llg_step(md, 1, DT)
    mesh.llg_step(off, 1, DT)
    a, b = to_host(md), to_host(off)
    # bound: FP32 rounding of the field (TOL_FP32 relative) over one step of |dm| <= 1, and of m
    assert np.abs(a - ref).max() <= 2e-6
    assert np.abs(b - ref).max() <= 2e-6
    mesh.close()


@pytest.mark.parametrize("n,per", [((32, 20, 4), (True, False, False)), ((24, 32, 8), (False, True, False)),
                                   ((16, 64, 1), (True, True, False)), ((32, 16, 8), (False, False, True))])
def test_periodic(g, n, per):
    cell = (3e-9, 3e-9, 3e-9)
    m = W.random_unit(n, 8)
    K = P.periodic_kernel(n, cell, per, 2)
    mesh = g.Mesh(n, cell, MS, A_ex=A, alpha=ALPHA, pbc=per, pbc_images=2)
    H = to_dev(np.full_like(m, np.nan))
    mesh.effective_field(to_dev(m), H)
    want = P.effective_field(m.astype(np.float64), K, cell, MS, A, per)
    assert e_inf(to_host(H), want) <= TOL_FP32
    mesh.close()
