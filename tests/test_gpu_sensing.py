"""The warp-specialised sensing GEMMs at the edges of their tiles, on both sides of the 96 transmitters from which
the other kernel takes over, against FP64 products with the context's own H.

Tolerance 2e-6 (relative L2): the hi / lo products leave out lo.lo and the low bits of lo, at most 3 x 2^-22 of a
product; 12 chained MMAs, 64 chunks and the splits add FP32 roundings of 2^-24 each, some 20 in quadrature or 3e-7 to
1.2e-6 as random signs go."""
import numpy as np
import pytest

from paper_1708_01663_gb300 import build, cisor, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _rand(*shape):
    g = torch.Generator().manual_seed(sum(shape))
    return torch.complex(torch.randn(*shape, generator=g), torch.randn(*shape, generator=g)).cuda()


# one chunk and one row a tile; ragged rows and chunks; several tiles a CTA (one chunk each, and many); several row
# tiles and splits; each accumulator width; f repeated for three components
@pytest.mark.parametrize("n,T,M,vector", [(8, 1, 2, False), (46, 16, 36, False), (46, 17, 126, False), (204, 33, 2, False),
                                          (142, 48, 130, False), (142, 16, 128, False), (256, 16, 360, False), (30, 64, 128, False),
                                          (46, 65, 18, False), (142, 96, 34, False), (46, 97, 36, False),
                                          (8, 81, 36, True), (12, 17, 36, True)])
def test_sensing_gemms(n, T, M, vector):
    build.build()
    if vector:
        ctx = cisor.Cisor(n, 0.1, synth.polarised_hemisphere()[:T], synth.planar_receivers(6, 0.5, 3.0), complex_f=True,
                          dim=3, vectorial=True)
    else:
        ctx = cisor.Cisor(n, 0.1, synth.plane_wave_angles(T), synth.circle_receivers(M, 0.1 * n), complex_f=True)
    assert (ctx.T, ctx.M) == (T, M)
    H = torch.empty(M, ctx.Nf, dtype=torch.complex64, device="cuda")
    host = np.empty((M, ctx.Nf), np.complex64)
    ctx.sensing_matrix(H)
    ctx.sensing_matrix(host)
    assert np.array_equal(H.cpu().numpy(), host) and np.abs(host).min() > 0
    Hd = H.to(torch.complex128)
    # 8-byte aligned operands, 16-byte aligned ones, and outputs that were never written
    for off in (0, 1):
        f = _rand(ctx.N + off)[off:]
        u, w = _rand(T * ctx.Nf + off)[off:], _rand(T * M + off)[off:]
        fd = f.to(torch.complex128).repeat(ctx.Nf // ctx.N)
        Zr = (fd * u.reshape(T, -1)) @ Hd.T
        zr = w.reshape(T, M).to(torch.complex128) @ Hd.conj()
        for _ in range(10):  # the roles of a CTA run at different distances from each other each time
            Z, z, b = (torch.full((v.numel() + off,), float("nan"), dtype=torch.complex64, device="cuda")[off:]
                       for v in (w, u, u))
            ctx.sense(f, u, Z)
            ctx.sense_adjoint(f, w, z, b)
            for got, want in ((Z, Zr), (z, zr), (b, fd.conj() * zr)):
                got = got.reshape(T, -1)
                assert float((got - want).norm() / want.norm()) < 2e-6
