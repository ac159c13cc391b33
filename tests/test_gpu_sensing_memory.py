"""A context's memory for few receivers: both copies of the sensing matrix take what their M x N values take."""
import pytest

from paper_1708_01663_gb300 import build, cisor, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_few_receivers_are_not_padded():
    build.build()
    used = []
    for M in (4, 16):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        ctx = cisor.Cisor(64, 1.0 / 6, synth.hemisphere_directions()[:1], synth.planar_receivers(4, 0.5, 8.0)[:M], dim=3)
        used.append(free - torch.cuda.mem_get_info()[0])
        N = ctx.N
        ctx.close()
    # 12 receivers more in two matrices, within 1/6 for the granularity of allocations (padding gave about half)
    want = 2 * 12 * N * 8
    assert abs(used[1] - used[0] - want) < want / 6, (used, want)
