"""Calls on device operands in place, and the two ways a gradient gets z + G^H v.

Kernels read and write device arguments directly; arguments that overlap, or
lie on the host, go through the context's buffers.  Either way the values are
the ones of separate device arrays, bit for bit.  A gradient whose adjoint solve
iterates takes z + G^H v from the solve's last residual pass, one whose adjoint
solve starts converged from a pass of its own: the same arithmetic, so the
gradients agree to FP32 rounding of the sum over transmitters (1e-6)."""
import numpy as np
import pytest

from paper_1708_01663_gb300 import build, cisor, synth
from tests.gpu_util import c64, rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _ctx(kind, T=3):
    build.build()
    if kind == "2d":
        return cisor.Cisor(45, 0.1, synth.plane_wave_angles(T), synth.circle_receivers(12, 6.0), complex_f=True), \
            synth.ellipse_phantom(45, 3, (0.1, 0.3), 5, 0.02)
    rx = synth.planar_receivers(4, 0.5, 3.0)
    if kind == "3d":
        return cisor.Cisor(12, 0.1, synth.hemisphere_directions()[:T], rx, complex_f=True, dim=3), \
            synth.sphere_phantom(12, 3, (0.1, 0.3), 5, 0.02)
    return cisor.Cisor(12, 0.1, synth.polarised_hemisphere()[:T], rx, complex_f=True, dim=3, vectorial=True), \
        synth.sphere_phantom(12, 3, (0.1, 0.3), 5, 0.02)


def _dev(a):
    return torch.from_numpy(c64(a)).cuda()


@pytest.mark.parametrize("kind", ["2d", "3d", "vector"])
@pytest.mark.parametrize("adjoint", [False, True])
def test_apply_A_overlapping(kind, adjoint):
    ctx, f = _ctx(kind)
    fd, n = _dev(f), ctx.T * ctx.Nf
    x = _dev(synth.random_field(3, (n,)))
    want = torch.empty_like(x)
    ctx.apply_A(fd, x, want, adjoint=adjoint)
    same = x.clone()
    ctx.apply_A(fd, same, same, adjoint=adjoint)  # in place
    buf = torch.zeros(n + 5, dtype=torch.complex64, device="cuda")
    buf[:n] = x
    ctx.apply_A(fd, buf[:n], buf[5:], adjoint=adjoint)  # y starts inside x
    y = torch.zeros(n, dtype=torch.complex64, device="cuda")
    y[7:7 + ctx.N] = fd.reshape(-1)
    ctx.apply_A(y[7:7 + ctx.N], x, y, adjoint=adjoint)  # f inside y
    host = np.empty(n, np.complex64)
    ctx.apply_A(c64(f), x, host, adjoint=adjoint)  # host f and y, device x
    for got in (same, buf[5:], y, torch.from_numpy(host).cuda()):
        assert torch.equal(got, want)


@pytest.mark.parametrize("kind", ["2d", "3d", "vector"])
def test_sensing_operands(kind):
    ctx, f = _ctx(kind)
    fd = _dev(f)
    u, w = _dev(synth.random_field(4, (ctx.T * ctx.Nf,))), _dev(synth.random_field(5, (ctx.T * ctx.M,)))
    Z, z, b = torch.empty_like(w), torch.empty_like(u), torch.empty_like(u)
    ctx.sense(fd, u, Z)
    ctx.sense_adjoint(fd, w, z, b)
    hZ, hz, hb = (np.empty(v.numel(), np.complex64) for v in (Z, z, b))
    ctx.sense(c64(f), u.cpu().numpy(), hZ)
    ctx.sense_adjoint(fd, w.cpu().numpy(), hz, hb)
    b2 = torch.empty_like(u)
    ctx.sense_adjoint(fd, w, None, b2)
    over = torch.zeros_like(u)
    over[:w.numel()] = w
    ctx.sense_adjoint(fd, over[:w.numel()], over, None)  # w inside z
    for got, want in ((torch.from_numpy(hZ).cuda(), Z), (torch.from_numpy(hz).cuda(), z), (torch.from_numpy(hb).cuda(), b),
                      (b2, b), (over, z)):
        assert torch.equal(got, want)


@pytest.mark.parametrize("kind", ["2d", "3d"])
def test_prox_in_place(kind):
    ctx, f = _ctx(kind)
    z = _dev(f) + 0.1 * _dev(synth.random_field(6, f.shape))
    for aniso in (False, True):
        want, same = torch.empty_like(z), z.clone()
        ctx.tv_prox(z, want, 0.05, 7, 0.0, 2.0, 0.0, 0.5, aniso=aniso)
        ctx.tv_prox(same, same, 0.05, 7, 0.0, 2.0, 0.0, 0.5, aniso=aniso)
        assert torch.equal(same, want)


@pytest.mark.parametrize("kind", ["2d", "3d", "vector"])
def test_gradient_from_converged_start(kind):
    ctx, f = _ctx(kind)
    fd = _dev(f)
    y = torch.empty(ctx.T, ctx.M, dtype=torch.complex64, device="cuda")
    ctx.forward(1.1 * fd, y_out=y, tol=1e-6)
    g0, g1 = torch.empty_like(fd), torch.empty_like(fd)
    D0, _, i0 = ctx.grad(fd, y, g0, tol=1e-5)
    D1, _, i1 = ctx.grad(fd, y, g1, tol=1e-5, x0_mode=2)
    assert i0.iters_max > 0 and i0.adj_iters_max > 0 and (i1.iters_max, i1.adj_iters_max) == (0, 0)
    assert abs(D1 / D0 - 1) < 1e-6
    assert rel(g1.cpu().numpy(), g0.cpu().numpy()) < 1e-6
