"""The 3D plane convolution (csrc/conv3d.cu, P = 64 and 128) at the sizes where
its tiling can go wrong: the smallest grid, the largest of each FFT side, grids
whose n^2 rows and n plane rows leave a partial CTA or warp.  A x and A^H x
against the FP64 oracle at the matvec bar of test_gpu_3d.py."""
import numpy as np
import pytest

from oracle import model
from paper_1708_01663_gb300 import build, cisor, synth
from tests.gpu_util import c64, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,pad,T", [(8, 0, 1), (9, 64, 3), (31, 0, 2), (32, 0, 1), (8, 128, 2), (45, 0, 2), (64, 0, 1)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_apply_A_plane(n, pad, T, adjoint):
    build.build()
    delta, dirs = 1.0 / 6, synth.hemisphere_directions()[:T]
    rx = synth.planar_receivers(4, 0.5, 0.6 * n * delta + 1.0)
    ctx = cisor.Cisor(n, delta, dirs, rx, complex_f=True, pad=pad, dim=3)
    prob = model.Problem(n, delta, dirs, rx, P=ctx.P, dim=3)
    f = synth.sphere_phantom(n, 4, (0.0, 0.6), 7, imag=0.05)
    x = synth.random_field(8, (T, n, n, n))
    y = np.empty((T, n, n, n), np.complex64)
    ctx.apply_A(c64(f), c64(x), y, adjoint=adjoint)
    op = prob.AH if adjoint else prob.A
    for t in range(T):
        assert rel(y[t], op(f, x[t])) < 2e-5
