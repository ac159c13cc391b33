"""cisor_sensing_matrix into host and device memory: the same bits either way, in slabs of rows and not row by row."""
import numpy as np
import pytest

from oracle import model
from paper_1708_01663_gb300 import build, cisor, synth
from tests.gpu_util import rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# rows of 512 KB: 64 a slab, so one, two (ragged) and three slabs; small tiled matrices with fewer transmitters than
# receivers; row-major ones (odd sizes, more than 96 transmitters)
@pytest.mark.parametrize("n,T,M", [(256, 1, 64), (256, 2, 100), (256, 1, 130), (16, 1, 200), (46, 3, 130), (45, 1, 101),
                                   (46, 97, 36)])
def test_read_back(n, T, M):
    build.build()
    rx = synth.circle_receivers(M, 0.2 * n)
    ctx = cisor.Cisor(n, 0.125, synth.plane_wave_angles(T), rx, complex_f=True)
    buf = torch.full((M * ctx.Nf + 1,), float("nan"), dtype=torch.complex64, device="cuda")
    ctx.sensing_matrix(buf[:-1])
    want = buf[:-1].cpu().numpy().reshape(M, -1)
    k, kb = model.wavenumbers(1.0)
    rows = [0, M // 2, M - 1]
    assert rel(want[rows], model.sensing_matrix(rx[rows], n, 0.125, k, kb)) < 1e-6
    assert torch.isnan(buf[-1].real)
    ctx.sensing_matrix(buf[1:])  # 8-byte aligned
    assert np.array_equal(buf[1:].cpu().numpy().reshape(M, -1), want)
    for host in (np.full((M, ctx.Nf), np.nan, np.complex64), torch.empty(M, ctx.Nf, dtype=torch.complex64).pin_memory()):
        for _ in range(2):  # (the second call uses the buffers of the first)
            before = ctx.launch_count()
            ctx.sensing_matrix(host)
            assert ctx.launch_count() - before <= 3
            assert np.array_equal(np.asarray(host), want)
    f = torch.zeros(ctx.N, dtype=torch.complex64, device="cuda")
    u = torch.zeros(T * ctx.Nf, dtype=torch.complex64, device="cuda")
    ctx.forward(f, u_out=u)  # the workspace is the solver's again
    inc = torch.empty_like(u)
    ctx.incident(inc)
    assert float((u - inc).norm() / inc.norm()) < 1e-6
