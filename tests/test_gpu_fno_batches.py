"""The network's forward pass and every gradient against the FP64 oracle for batches of one, a few, more than one item per
CTA and more than one chunk of the mode mixing (32 samples), with an f per sample and one for all.

Tolerance 2e-5 (relative L2 of each tensor).  An operand is held as BF16 hi + lo.  Without lo, its rounding (2^-9) moves
a tensor by 2e-5 to 2e-3 depending on the operand (the oracle with each operand rounded so, one and five samples); the
14 kinds of operands sum to 4e-3, and what hi + lo leaves out is 2^-9 of that, 8e-6.  FP32 sums and the GELU's
polynomial (2.5e-6 in erf) add less than as much again."""
import numpy as np
import pytest

from oracle import fno as ofno
from oracle import model
from paper_1708_01663_gb300 import build, cisor, synth

pytestmark = pytest.mark.gpu
N, TOL = 128, 2e-5


def _one(p, f, u, t):
    """Prediction, loss and gradients of one sample."""
    out, _ = ofno.forward(p, f, u)
    return out, *ofno.loss_and_grad(p, [f], [u], [t])


def _rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b)))


@pytest.mark.parametrize("B,per_sample", [(1, True), (5, False), (32, False), (33, True)])
def test_batch(B, per_sample):
    build.build()
    net = cisor.FNO(max_batch=B, seed=5)
    flat = np.empty(net.num_params, np.float32)
    net.get_params(flat, as_used=False)
    rng = np.random.default_rng(B)
    flat += np.where(flat == 0, 0.1 * rng.standard_normal(flat.size), 0).astype(np.float32)  # biases
    net.set_params(flat)
    net.get_params(flat, as_used=True)
    p = cisor.fno_param_dict(flat)
    c = lambda a: np.ascontiguousarray(a, dtype=np.complex64)
    f = c([synth.ellipse_phantom(N, 4, (0.0, 0.8), 3 + b, 0.02) for b in range(B if per_sample else 1)])
    u = c(model.plane_waves(synth.plane_wave_angles(B) + 0.3, N, 1.0 / 8, 2 * np.pi))
    t = c([0.3 * synth.random_field(60 + b, (N, N)) + 0.5 * f[b % len(f)] for b in range(B)])
    wide = lambda a: a.astype(np.complex128)
    args = [(p, wide(f[b % len(f)]), wide(u[b]), wide(t[b])) for b in range(B)]
    ref = [_one(*a) for a in args]
    out, g = np.empty_like(u), np.empty(net.num_params, np.float32)
    net.forward(f, u, out, f_per_sample=per_sample)
    assert max(_rel(out[b], ref[b][0]) for b in range(B)) < TOL
    loss = net.loss_grad(f, u, t, g, f_per_sample=per_sample)
    assert abs(loss / np.mean([r[1] for r in ref]) - 1) < TOL
    got = cisor.fno_param_dict(g)
    err = {k: _rel(got[k], np.mean([r[2][k] for r in ref], axis=0)) for k in p}
    assert max(err.values()) < TOL, err
    net.close()
