"""The 2D FGP prox by tiles against the oracle: one launch that is first and last, one and several, unequal shares of the
iterations (7 = 3 + 4, 13 = 4 + 4 + 5), the most iterations a launch takes (6), images smaller than a tile, ragged last
tiles.  z is random over the whole image and the weight large, so that a halo one pixel too narrow shows (the blocks
restated in numpy with halos one short: 3e-5 after 12 iterations, 6e-4 and more after 7 and 13).

Tolerance 2e-5, as for the prox elsewhere: an iteration adds to r the dual step 1 / (8 lam) = 0.25 times the roundings of
two x (some 2^-22 each) and its own, about 5e-7; 13 iterations with momentum stay near 5e-6 as signs go, and x takes
4 lam = 2 of that."""
import numpy as np
import pytest

from oracle import prox
from paper_1708_01663_gb300 import build, cisor, synth
from tests.gpu_util import c64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("complex_f", [False, True])
@pytest.mark.parametrize("n", [8, 17, 45, 97])
def test_tiles(n, complex_f):
    build.build()
    ctx = cisor.Cisor(n, 0.125, synth.plane_wave_angles(1), synth.circle_receivers(4, 0.125 * n), complex_f=complex_f)
    z = c64(0.4 + 0.5 * synth.random_field(n, (n, n)))
    x = np.empty_like(z)
    for iters in (1, 2, 6, 7, 12, 13):
        ctx.tv_prox(z, x, 0.5, iters, -9.0, 9.0, 0.0, 0.9)
        ref = prox.prox_R(z.astype(np.complex128), 0.5, iters, (-9.0, 9.0), (0.0, 0.9) if complex_f else None)
        assert np.abs(x - ref).max() < 2e-5, iters
