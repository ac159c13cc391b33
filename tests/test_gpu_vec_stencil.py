"""The grad-div stencil of the vectorial model at the edges of its CTAs (256 columns, 4 planes): A x and A^H x against
the oracle, and <A x, y> = <x, A^H y>.

Tolerance 2e-5 (relative L2) as for every FP32 matvec here, 1e-5 of |A x| |y| for the identity: both sides carry the
FFTs' FP32 roundings, a few 1e-7 each."""
import numpy as np
import pytest

from oracle import vector
from paper_1708_01663_gb300 import build, cisor, synth
from tests.gpu_util import c64, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 9, 13, 16, 17, 23])
def test_stencil_edges(n):
    build.build()
    tx, rx, T = synth.polarised_hemisphere()[:2], synth.planar_receivers(2, 0.5, 3.0), 2
    ctx = cisor.Cisor(n, 0.1, tx, rx, complex_f=True, dim=3, vectorial=True)
    prob = vector.VectorProblem(n, 0.1, tx[:, :3], tx[:, 3:], rx, P=ctx.P)
    f = synth.sphere_phantom(n, 3, (0.1, 0.3), 5, 0.02)
    x, y = (synth.random_field(s, (T, 3, n, n, n)) for s in (1, 2))
    Ax, Ay = (np.empty(x.shape, np.complex64) for _ in range(2))
    ctx.apply_A(c64(f), c64(x), Ax)
    ctx.apply_A(c64(f), c64(y), Ay, adjoint=True)
    for t in range(T):
        assert rel(Ax[t], prob.A(f, x[t]).reshape(Ax[t].shape)) < 2e-5
        assert rel(Ay[t], prob.AH(f, y[t]).reshape(Ay[t].shape)) < 2e-5
    lhs, rhs = (np.vdot(a.astype(np.complex128), b.astype(np.complex128)) for a, b in ((Ax, y), (x, Ay)))
    assert abs(lhs - rhs) < 1e-5 * np.linalg.norm(Ax) * np.linalg.norm(y)
