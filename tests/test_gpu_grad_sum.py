"""The gradient's sum over transmitters at f = 0, where u = u_in and v = 0: g = -sum_t conj(u_in,t) H^H y_t, against
FP64 with the context's own tables, for fewer, as many and more transmitters than the kernel's warps and odd images.

Tolerance 3e-6 (relative L2): the sensing product is within 2e-6 of FP64, the FP32 sum adds 2^-24 sqrt(T)."""
import numpy as np
import pytest

from paper_1708_01663_gb300 import build, cisor, synth
from tests.gpu_util import c64, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,T", [(8, 1), (9, 7), (45, 8), (46, 9), (33, 17), (64, 33)])
def test_gradient_sum(n, T):
    build.build()
    M = 12
    ctx = cisor.Cisor(n, 0.1, synth.plane_wave_angles(T), synth.circle_receivers(M, 0.1 * n), complex_f=True)
    H, u = np.empty((M, ctx.Nf), np.complex64), np.empty((T, ctx.Nf), np.complex64)
    ctx.sensing_matrix(H)
    ctx.incident(u)
    y = synth.random_field(3, (T, M))
    g = np.empty(ctx.N, np.complex64)
    D, _, _ = ctx.grad(np.zeros(ctx.N, np.complex64), c64(y), g)
    yd = c64(y).astype(np.complex128)
    assert abs(D / (0.5 * np.sum(np.abs(yd) ** 2)) - 1) < 1e-6
    assert rel(g, -np.sum(u.conj().astype(np.complex128) * (yd @ H.conj().astype(np.complex128)), axis=0)) < 3e-6
