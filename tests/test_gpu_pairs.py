"""Meshes that take the paired x rows and the fused z convolution, against the FP64 oracle: odd ny
(pairs across z planes, half vectors of the spectrum), a last pair with one row, row counts that do
not fill the last block, one pair per block, 3 * 2^k and 5 * 2^k lengths, odd nx (cell by cell), every
z radix plan, columns that do not fill the last tile; the RK4, general RK, H_eff and dm/dt epilogues."""
import numpy as np
import pytest

from oracle import conv as C
from oracle import llg as L
from oracle import rkf as R
from oracle import tensor as T
from paper_2308_08447_gb300 import workloads as W
from tests.gpu_util import TOL_FP32, e_inf, lib, to_dev, to_host

pytestmark = pytest.mark.gpu

A, ALPHA, MS, DT, CELL = 1.3e-11, 0.05, 8e5, 5e-14, (3e-9, 3e-9, 3e-9)


@pytest.fixture(scope="module")
def g():
    return lib()


@pytest.mark.parametrize("n", [(64, 33, 21), (250, 61, 3), (63, 44, 17), (500, 31, 3), (1000, 42, 1), (640, 103, 4)])
def test_rows_and_epilogues(g, n):
    m = W.random_unit(n, 9)
    N = T.tensor_all_offsets(n, CELL)
    mesh = g.Mesh(n, CELL, MS, A_ex=A, alpha=ALPHA)
    M = (MS * m).astype(np.float32)
    H = to_dev(np.full_like(m, np.nan))
    mesh.demag(to_dev(M), H)
    assert e_inf(to_host(H), C.fft_conv(M.astype(np.float64), N)) <= TOL_FP32
    m64 = m.astype(np.float64)
    heff = MS * C.fft_conv(m64, N) + L.exchange_field(m64, CELL, MS, A)
    f = lambda v: L.rhs(v, N, CELL, MS, A, ALPHA)
    k1 = f(m64)
    mesh.effective_field(to_dev(m), H)
    assert e_inf(to_host(H), heff) <= TOL_FP32
    mesh.llg_rhs(to_dev(m), H)
    assert e_inf(to_host(H), k1) <= TOL_FP32
    # one step of each kind, with fields 8 bytes and only 4 bytes aligned; bound: FP32 rounding of the
    # slopes (TOL_FP32 relative, dt |dm/dt| < 0.1) and of m
    buf = to_dev(np.zeros(m.size + 1))
    for step, want in ((lambda v: mesh.llg_step(v, 1, DT), L.rk4_step(m64, DT, f)),
                       (lambda v: mesh.rkf56_step(v, DT), R.rkf56_step(m64, DT, f)[0])):
        md = to_dev(m)
        off = buf[1:].view(m.shape)
        off.copy_(md)
        step(md)
        step(off)
        assert np.abs(to_host(md) - want).max() <= 2e-6
        assert np.abs(to_host(off) - want).max() <= 2e-6
    mesh.close()


@pytest.mark.parametrize("n", [(20, 9, 9), (24, 10, 17), (11, 13, 33), (9, 5, 65), (7, 3, 130), (130, 70, 12)])
def test_z_lengths(g, n):
    M = (MS * W.random_unit(n, 10)).astype(np.float32)
    mesh = g.Mesh(n, CELL, MS)
    H = to_dev(np.full_like(M, np.nan))
    mesh.demag(to_dev(M), H)
    assert e_inf(to_host(H), C.fft_conv(M.astype(np.float64), T.tensor_all_offsets(n, CELL))) <= TOL_FP32
    mesh.close()


@pytest.mark.parametrize("n", [(512, 400, 1), (400, 400, 1), (256, 800, 1), (800, 300, 1), (1024, 96, 1), (512, 1030, 1),
                               (300, 420, 1), (128, 64, 8), (250, 61, 3)])
def test_split_calls_equal_one_call(g, n):
    # a call's first forward transform, its stages and its last stage may run in different kernels:
    # their results are bit-identical
    import torch
    m = to_dev(W.vortex_noise(n, CELL, 11))
    mesh = g.Mesh(n, CELL, MS, A_ex=A, alpha=ALPHA)
    one, split = m.clone(), m.clone()
    mesh.llg_step(one, 6, DT)
    for k in (1, 2, 3):
        mesh.llg_step(split, k, DT)
    torch.cuda.synchronize()
    assert torch.equal(one, split)
    mesh.close()
