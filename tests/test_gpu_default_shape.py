"""The column shape that a context starts with, also for few transforms at P = 512, and 3D passes with P = 256 for every shape that the autotuner can pick."""
import numpy as np
import pytest

from oracle import model
from paper_1708_01663_gb300 import build, cisor, synth
from tests.gpu_util import c64, rel

pytestmark = pytest.mark.gpu
DELTA = 1.0 / 6


@pytest.mark.parametrize("dim,n,pad,shape", [(2, 20, 0, 256), (2, 64, 0, 256), (2, 65, 0, 16), (2, 129, 0, 16), (3, 20, 0, 256),
                                             (3, 20, 256, 512)])
def test_default(dim, n, pad, shape):
    build.build()
    if dim == 2:
        ctx = cisor.Cisor(n, DELTA, synth.plane_wave_angles(2), synth.circle_receivers(4, DELTA * n), pad=pad)
    else:
        ctx = cisor.Cisor(n, DELTA, synth.hemisphere_directions()[:2], synth.planar_receivers(2, 0.5, DELTA * n), dim=3, pad=pad)
    assert ctx.tuning() == (shape, 0)


@pytest.mark.parametrize("shape", [512, 256, 16])
@pytest.mark.parametrize("n", [20, 33])
def test_columns_3d_p256(n, shape):
    """y forward, z with the spectrum, y back: A x and A^H x against the oracle (2e-5, the matvec's tolerance)."""
    build.build()
    dirs, rx = synth.hemisphere_directions()[:2], synth.planar_receivers(2, 0.5, DELTA * n)
    ctx = cisor.Cisor(n, DELTA, dirs, rx, complex_f=True, dim=3, pad=256)
    prob = model.Problem(n, DELTA, dirs, rx, P=256, dim=3)
    ctx.set_cols_cta(shape)
    f = synth.sphere_phantom(n, 4, (0.0, 0.6), 7, imag=0.05)
    x = synth.random_field(8, (2, n, n, n))
    y = np.empty((2, n, n, n), np.complex64)
    for adjoint, op in ((False, prob.A), (True, prob.AH)):
        ctx.apply_A(c64(f), c64(x), y, adjoint=adjoint)
        for t in range(2):
            assert rel(y[t], op(c64(f).astype(np.complex128), x[t])) < 2e-5


@pytest.mark.parametrize("T", [1, 2, 5, 6])
def test_few_transforms_p512(T):
    """By default a pass has the bits of the two-stage columns; solves of one and of three to five transmitters iterate with
    another kernel and agree with both shapes that can be set (1e-5, as solves to 1e-6 by different shapes do)."""
    build.build()
    n = 129
    new = lambda: cisor.Cisor(n, 0.125, synth.plane_wave_angles(T), synth.circle_receivers(8, 0.125 * n), complex_f=True)
    f = c64(synth.ellipse_phantom(n, 3, (0.05, 0.2), 31, 0.02))
    x = c64(synth.random_field(9, (T, n, n)))
    A, u, g = {}, {}, {}
    y = c64(synth.random_field(10, (T, 8)))
    for shape in (None, 512, 16):
        ctx = new()
        if shape:
            ctx.set_cols_cta(shape)
        A[shape], u[shape], g[shape] = np.empty_like(x), np.empty_like(x), np.empty_like(f)
        ctx.apply_A(f, x, A[shape])
        ctx.forward(f, u_out=u[shape], tol=1e-6, max_iter=2000)
        ctx.grad(f, y, g[shape], tol=1e-6, max_iter=2000)
        ctx.close()
    assert np.array_equal(A[None], A[16])
    assert np.array_equal(u[None], u[16]) == (T not in (1, 5))
    for shape in (512, 16):
        assert rel(u[None], u[shape]) < 1e-5 and rel(g[None], g[shape]) < 1e-5


@pytest.mark.parametrize("T,chunk", [(5, 2), (7, 3), (7, 1)])
def test_chunks_keep_the_shape_p512(T, chunk):
    """Transmitter chunks take the kernel of the whole pass: identical results, as for shapes that were set."""
    build.build()
    n = 129
    ctx = cisor.Cisor(n, 0.125, synth.plane_wave_angles(T), synth.circle_receivers(8, 0.125 * n), complex_f=True)
    f = c64(synth.ellipse_phantom(n, 3, (0.05, 0.2), 31, 0.02))
    x = c64(synth.random_field(9, (T, n, n)))
    y, u = [], []
    for k in (0, chunk):
        ctx.set_tx_chunk(k)
        y.append(np.empty_like(x))
        u.append(np.empty_like(x))
        ctx.apply_A(f, x, y[-1])
        ctx.forward(f, u_out=u[-1], tol=1e-6, max_iter=2000)
    assert np.array_equal(y[0], y[1]) and np.array_equal(u[0], u[1])
