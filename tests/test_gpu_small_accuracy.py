"""Rounding error of the small-mesh kernels. Their pass-by-pass counterparts reach these rms errors of the
field of random unit vectors against 64 bits (measured on the meshes below, mean of four inputs); the
small-mesh kernels may not be further off than that, with a tenth for the spread between inputs."""
import numpy as np
import pytest

from oracle import conv as C
from oracle import tensor as T
from paper_2308_08447_gb300 import workloads as W
from tests.gpu_util import lib, to_dev, to_host

pytestmark = pytest.mark.gpu

CELL = (3e-9, 3e-9, 3e-9)


@pytest.mark.parametrize("n,tiled", [((150, 150, 6), 1.391e-7), ((300, 150, 4), 1.433e-7), ((80, 48, 2), 1.502e-7),
                                     ((61, 80, 4), 1.365e-7), ((20, 600, 1), 1.330e-7), ((32, 32, 8), 1.961e-7)])
def test_rms_error(n, tiled):
    g = lib()
    M = (8e5 * W.random_unit(n, 21)).astype(np.float32)
    mesh = g.Mesh(n, CELL, 8e5)
    H = to_dev(np.full_like(M, np.nan))
    mesh.demag(to_dev(M), H)
    mesh.close()
    want = C.fft_conv(M.astype(np.float64), T.tensor_all_offsets(n, CELL))
    assert np.sqrt(((to_host(H) - want) ** 2).sum() / (want ** 2).sum()) <= 1.1 * tiled
