"""The split-K sum of the sensing product where FP32's range ends: three splits that one warp sums hold 2.5e38, 2.5e38 and
-2.5e38, whose sum is taken in FP64.

Tolerance 2e-6 as in tests/test_gpu_sensing.py, relative to the sum over the splits' magnitudes."""
import pytest

from paper_1708_01663_gb300 import build, cisor, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_sum_beyond_fp32():
    build.build()
    n, T, M = 64, 2, 32  # splits of one image row each; warp 0 sums rows 0, 8, 16, ...
    ctx = cisor.Cisor(n, 0.5, synth.plane_wave_angles(T), synth.circle_receivers(M, 30.0), complex_f=True)
    H = torch.empty(M, n, n, dtype=torch.complex64, device="cuda")
    ctx.sensing_matrix(H)
    Hd = H.to(torch.complex128)
    u = torch.zeros(T, n, n, dtype=torch.complex128, device="cuda")
    for row, amp in ((0, 2.5e38), (8, 2.5e38), (16, -2.5e38)):
        h = Hd[5, row]  # in phase at receiver 5: its partials add up to amp
        u[0, row] = amp * h.conj() / h.abs() / h.abs().sum()
    g = torch.Generator().manual_seed(4)
    u[1] = torch.complex(torch.randn(n, n, generator=g), torch.randn(n, n, generator=g)).cuda()
    u = u.to(torch.complex64)
    Z = torch.empty(T, M, dtype=torch.complex64, device="cuda")
    ctx.sense(torch.ones(n * n, dtype=torch.complex64, device="cuda"), u, Z)
    parts = torch.einsum("mrc,trc->tmr", Hd, u.to(torch.complex128))
    assert 4.9e38 < float((parts[0, 5, 0] + parts[0, 5, 8]).real) < 5.1e38
    assert torch.isfinite(Z.real).all() and torch.isfinite(Z.imag).all()
    assert abs(float(Z[0, 5].real) / 2.5e38 - 1) < 1e-5
    err = (Z.to(torch.complex128) - parts.sum(2)).abs().amax(1)
    assert (err < 2e-6 * parts.abs().sum(2).amax(1)).all()
