"""Which kernel a launch takes at the lines that the dispatch draws (named by the profiler's trace); the
reasons stand beside the rules. Correctness on both sides of a line is tested elsewhere."""
import numpy as np
import pytest

from paper_2308_08447_gb300 import workloads as W
from tests.gpu_util import lib, to_dev
from tests.test_gpu_variants import has, kernels

pytestmark = pytest.mark.gpu

CELL, MS = (3e-9, 3e-9, 3e-9), 8e5


@pytest.fixture(scope="module")
def g():
    return lib()


def launched(g, n, what):
    mesh = g.Mesh(n, CELL, MS, A_ex=1.3e-11, alpha=0.05)
    m = to_dev(W.random_unit(n, 3))
    H = to_dev(np.zeros(m.shape))
    names = kernels({"demag": lambda: mesh.demag(m, H), "heff": lambda: mesh.effective_field(m, H),
                     "rk4": lambda: mesh.llg_step(m, 1, 1e-14)}[what])
    mesh.close()
    return names


# the convolution: lines below 1024 values in one launch, longer ones by the tiled kernels
@pytest.mark.parametrize("n,one", [((100, 256, 1), True), ((100, 257, 1), True), ((100, 512, 1), False), ((20, 1024, 1), False),
                                   ((300, 320, 2), True), ((512, 400, 2), False)])
def test_convolution(g, n, one):
    names = launched(g, n, "demag")
    assert has(names, "small_conv") == one
    assert has(names, "film_conv" if n[2] == 1 else "z_conv") == (not one)


# x rows of power-of-two lengths: row_kernel's tiles of 4096 values up to one block per SM, the paired rows
# where they are few (3D) or make a second wave that is less than half full; no paired epilogue at L = 4096
@pytest.mark.parametrize("n,what,kernel", [((512, 1024, 1), "demag", "row_kernel<512, 8,"), ((128, 1024, 1), "demag", "row_kernel<128, 8,"), ((128, 512, 1), "heff", "row_kernel<128, 8,"),
                                           ((256, 608, 4), "demag", "row_kernel<256, 16,"), ((256, 152, 4), "demag", "row_pair_kernel<256,"),
                                           ((512, 1220, 1), "demag", "row_pair_kernel<512,"), ((512, 1830, 1), "demag", "row_kernel<512, 8,"),
                                           ((512, 399, 1), "rk4", "row_kernel<512,"), ((512, 400, 1), "rk4", "row_pair_kernel<512,"),
                                           ((2000, 61, 1), "heff", "row_pair_kernel<2048,"), ((4000, 61, 1), "heff", "row_kernel<4096,"),
                                           ((4000, 61, 1), "rk4", "row_kernel<4096,")])
def test_power_of_two_rows(g, n, what, kernel):
    names = launched(g, n, what)
    assert has(names, kernel), names
    if what == "demag":
        assert not has(names, "row_pair" if kernel.startswith("row_kernel") else "row_kernel"), names


# x rows of lengths 3 * 2^k and 5 * 2^k: row_kernel where its blocks make one wave that fills half of the SMs
@pytest.mark.parametrize("n,what,kernel", [((700, 300, 1), "demag", "row_kernel<768,"), ((700, 608, 1), "demag", "row_kernel<768,"),
                                           ((700, 609, 1), "demag", "row_pair_kernel<768,"), ((700, 400, 1), "rk4", "row_pair_kernel<768,"),
                                           ((600, 512, 1), "rk4", "row_kernel<640,"), ((300, 304, 4), "demag", "row_kernel<320,"),
                                           ((1500, 138, 1), "demag", "row_pair_kernel<1536,"), ((1500, 140, 1), "demag", "row_kernel<1536,"),
                                           ((2500, 16, 1), "heff", "row_kernel<2560,"), ((2500, 153, 1), "heff", "row_pair_kernel<2560,"),
                                           ((3000, 16, 1), "rk4", "row_kernel<3072,"), ((180, 1400, 1), "demag", "row_pair_kernel<192,"),
                                           ((600, 333, 1), "demag", "small_row_kernel"), ((700, 260, 1), "demag", "small_row_kernel")])
def test_mixed_rows(g, n, what, kernel):
    assert has(launched(g, n, what), kernel)


@pytest.mark.parametrize("n", [(700, 400, 1), (1500, 256, 1), (640, 103, 6), (128, 1024, 1), (250, 160, 8)])
def test_kernels_of_a_run_round_alike(g, n):
    # the first forward transform and the stages run in different kernels: a split run equals the unsplit one
    import torch
    m = to_dev(W.vortex_noise(n, CELL, 12))
    mesh = g.Mesh(n, CELL, MS, A_ex=1.3e-11, alpha=0.05)
    one, split = m.clone(), m.clone()
    mesh.llg_step(one, 4, 5e-14)
    for k in (1, 2, 1):
        mesh.llg_step(split, k, 5e-14)
    torch.cuda.synchronize()
    assert torch.equal(one, split)
    mesh.close()


# the autotuner times what the mesh runs: nothing for passes with one kernel
@pytest.mark.parametrize("n,not_timed,timed", [((96, 60, 1), ("film_conv", "row_kernel", "row_pipe"), None),
                                               ((72, 52, 6), ("y_pass", "z_conv", "row_kernel", "row_pipe"), None),
                                               ((260, 244, 2), ("y_pass", "z_conv", "film_conv"), "row_pipe"),
                                               ((256, 268, 1), (), "film_conv")])
def test_autotuner_times_what_runs(g, n, not_timed, timed):
    launched(g, n, "demag")               # a process's first trace may be empty, and tuning runs once
    mesh = g.Mesh(n, CELL, MS, pow2_pad=True)
    names = kernels(mesh.autotune)
    assert not any(has(names, part) for part in not_timed)
    assert timed is None or has(names, timed)
    if timed is None:
        assert g.gbd_mesh_get_tuning(mesh.handle) == (1, 0, 0, 0)
    mesh.close()
