"""What a user of this library has it do, at the sizes its users run.

The library reconstructs a permittivity contrast f from scattered fields: per
outer iteration it solves A u = u_in and A^H v = b for every transmitter,
applies the sensing operator H and its adjoint, assembles the gradient, and
takes a TV proximal step with momentum.  A Fourier neural operator (FNO) gives
an optional warm start.  The cases are those calls through the Python binding:
single operators first (matvec, sensing, prox), then the gradients and steps
built from them at contrasts whose solves take a few iterations, then the
network's two directions and a batch of problems of uneven size.

Sizes follow the library's own workloads (64^2, 128^2, 256^2 at lambda/8; 64^3
at lambda/6; 32^3 vectorial at lambda/16; 128 x 128 FNO) and the ragged sizes
between them.  ``exact`` restates every path in 64 bits with torch alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1708_01663_gb300 import cisor, synth

C64, C128, F64 = torch.complex64, torch.complex128, torch.float64
DEV = torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")
# the FNO's fixed architecture: grid, width, modes, layers, hidden units
FN, FC, FM, FL, FH = 128, 32, 16, 4, 128


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # one operator application on the smallest workload: a user's own Krylov method or check on 64^2 images
        {"name": "matvec 2D 64", "kind": "matvec", "dim": 2, "n": 64, "T": 8, "adjoint": False, "complex_f": False},
        # the adjoint operator on the largest 2D grid with absorbing contrast and 64 transmitters
        {"name": "adjoint matvec 2D 256", "kind": "matvec", "dim": 2, "n": 256, "T": 64, "adjoint": True,
         "complex_f": True},
        # the operator on the 3D workload: 48 transmitters on 64^3 voxels
        {"name": "matvec 3D 64", "kind": "matvec", "dim": 3, "n": 64, "T": 48, "adjoint": False, "complex_f": False},
        # measurements of given fields and the adjoint's right-hand side, 1024 receivers on 64^3 voxels
        {"name": "sensing 3D 64", "kind": "sensing", "dim": 3, "n": 64, "T": 48, "M": 1024, "complex_f": False},
        # the prox of the largest 2D image, complex contrast, 20 FGP iterations as in every step
        {"name": "prox 2D 256", "kind": "prox", "dim": 2, "n": 256, "iters": 20, "complex_f": True, "aniso": False},
        # data term and gradient on the largest 2D grid: weak absorbing scatterers, cold solves to 1e-4
        {"name": "gradient 2D 256", "kind": "grad", "dim": 2, "n": 256, "T": 64, "M": 256, "delta": 0.125,
         "complex_f": True, "tx": "plane", "shapes": 10, "contrast": 0.05, "imag": 0.005, "its": 4},
        # a Fresnel-style reconstruction step: 8 line sources, 360 masked receivers, latency-bound sizes
        {"name": "step 2D 128", "kind": "step", "dim": 2, "n": 128, "T": 8, "M": 360, "delta": 1.5 / 128,
         "complex_f": False, "tx": "point", "shapes": 3, "contrast": 1.0, "imag": 0.0, "its": 4},
        # a reconstruction step of the 3D scalar workload
        {"name": "step 3D 64", "kind": "step", "dim": 3, "n": 64, "T": 48, "M": 1024, "delta": 1.0 / 6,
         "complex_f": False, "tx": "plane", "shapes": 5, "contrast": 0.3, "imag": 0.0, "its": 5},
        # the 3D vectorial gradient: 81 polarised plane waves on 32^3 voxels, 36 masked receivers
        {"name": "gradient vectorial 32", "kind": "grad", "dim": 3, "n": 32, "T": 81, "M": 36, "delta": 1.0 / 16,
         "complex_f": False, "tx": "vector", "shapes": 2, "contrast": 1.5, "imag": 0.0, "its": 4},
        # gradients of four problems of uneven, ragged size advanced together
        {"name": "batch 2D ragged", "kind": "batch", "sizes": "75,96,128,181", "txs": "24,32,17,40", "M": 128,
         "contrast": 0.1, "imag": 0.01, "its": 4},
        # the learned warm start of 32 transmitters that share one contrast image
        {"name": "fno forward 32", "kind": "fno", "B": 32, "per_sample": False, "grad": False},
        # loss and every parameter's gradient for a training batch of 32 samples
        {"name": "fno gradient 32", "kind": "fno", "B": 32, "per_sample": True, "grad": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same paths: sizes over the whole supported range, bounded by the listed cases' work."""
    kind = rng.choice(["matvec", "matvec", "matvec", "sensing", "prox", "grad", "grad", "step", "batch", "fno", "fno"])
    dim = rng.choice([2, 2, 3])
    if kind == "fno":
        return {"kind": "fno", "B": rng.randint(1, 32), "per_sample": rng.random() < 0.5, "grad": rng.random() < 0.5}
    if kind == "prox":
        return {"kind": "prox", "dim": dim, "n": _log(rng, 8, 256) if dim == 2 else _log(rng, 8, 64),
                "iters": rng.randint(1, 30), "complex_f": rng.random() < 0.5, "aniso": rng.random() < 0.3}
    if kind == "matvec":
        n = _log(rng, 8, 256) if dim == 2 else _log(rng, 8, 72)
        most = 64 if dim == 2 else (48 if n <= 64 else 6)
        c = {"kind": "matvec", "dim": dim, "n": n, "T": _log(rng, 1, most), "adjoint": rng.random() < 0.5,
             "complex_f": rng.random() < 0.5}
        if dim == 3 and n <= 32 and rng.random() < 0.4:
            c["tx"] = "vector"
        return c
    if kind == "sensing":
        n = _log(rng, 16, 256) if dim == 2 else _log(rng, 12, 64)
        return {"kind": "sensing", "dim": dim, "n": n, "T": _log(rng, 1, 64 if dim == 2 else 48),
                "M": _log(rng, 8, 512 if dim == 2 else 700), "complex_f": rng.random() < 0.5}
    if kind == "batch":
        k = rng.randint(2, 4)
        return {"kind": "batch", "sizes": ",".join(str(_log(rng, 32, 180)) for _ in range(k)),
                "txs": ",".join(str(_log(rng, 4, 40)) for _ in range(k)), "M": rng.randint(32, 128),
                "contrast": 0.1, "imag": rng.choice([0.0, 0.01]), "its": 4}
    cplx = rng.random() < 0.5
    c = {"kind": kind, "dim": dim, "complex_f": cplx, "imag": 0.02 if cplx else 0.0, "its": 5}
    if dim == 2:
        c["n"], c["T"], c["M"] = _log(rng, 24, 256), _log(rng, 2, 64), _log(rng, 16, 360)
        c["tx"] = rng.choice(["plane", "point"])
        side = rng.uniform(1.0, 4.0)
    else:
        c["tx"] = rng.choice(["plane", "plane", "vector"])
        c["n"] = _log(rng, 12, 60 if c["tx"] == "plane" else 32)
        c["T"], c["M"] = _log(rng, 2, 32), _log(rng, 16, 400)
        side = rng.uniform(1.0, 4.0)
    c["delta"] = side / c["n"]
    c["shapes"], c["contrast"] = rng.randint(2, 6), round(0.6 / side, 3)
    return c


# --------------------------------------------------------------------------- geometry and inputs
def _delta(case):
    return float(case.get("delta", 0.125 if case["dim"] == 2 else 1.0 / 6))


def _geometry(case):
    """(transmitters, receivers, mask) of a case: plane waves or sources around the grid, receivers outside it."""
    dim, n, T, M = case["dim"], case["n"], case.get("T", 1), case.get("M", 16)
    side = n * _delta(case)
    tx = case.get("tx", "plane")
    if dim == 2:
        if tx == "point":
            src, rx = synth.circle_sources(T, 4.8 * side), synth.circle_receivers(M, 5.07 * side)
            return src, rx, synth.angular_mask(src, rx, 60.0)
        return synth.plane_wave_angles(T), synth.circle_receivers(M, 0.75 * side), None
    i = np.arange(T) + 0.5  # directions spread over the upper hemisphere
    cz, ph = 1.0 - 0.95 * i / T, math.pi * (3.0 - math.sqrt(5.0)) * i
    sz = np.sqrt(1.0 - cz * cz)
    d = np.stack([sz * np.cos(ph), sz * np.sin(ph), cz], 1)
    if tx == "vector":  # polar unit vector as polarisation; receivers on a circle in the azimuth plane
        pol = np.stack([cz * np.cos(ph), cz * np.sin(ph), -sz], 1)
        rx2 = synth.circle_receivers(M, 10.0 * side)
        return np.concatenate([d, pol], 1), np.concatenate([rx2, np.zeros((M, 1))], 1), synth.angular_mask(d[:, :2], rx2, 50.0)
    w = math.ceil(math.sqrt(M))
    return d, synth.planar_receivers(w, 0.5, 0.75 * side)[:M], None


def _context(case, tuned):
    tx, rx, mask = _geometry(case)
    kind = case.get("tx", "plane")
    ctx = cisor.Cisor(case["n"], _delta(case), tx, rx, complex_f=case["complex_f"], dim=case["dim"],
                      tx_kind="point" if kind == "point" else 0, vectorial=kind == "vector")
    if mask is not None:
        ctx.set_rx_mask(mask)
    if tuned:  # what the benchmark and every long-running program do once per geometry
        ctx.autotune(reps=3)
    return ctx


def _phantom(dim, n, shapes, contrast, imag, seed):
    draw_ = synth.sphere_phantom if dim == 3 else synth.ellipse_phantom
    return draw_(n, shapes, (0.3 * contrast, contrast), seed, imag).astype(np.complex64)


def _randn(seed, *shape):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return torch.randn(*shape, dtype=C64, device=DEV, generator=g)


def _contrast_of(case, seed):
    """The phantom at which a single operator is applied."""
    f = _phantom(case["dim"], case["n"], 5, 0.8, 0.05 if case["complex_f"] else 0.0, seed)
    return torch.from_numpy(f).to(DEV)


def _born_data(model, f, seed):
    """Measurements of the phantom in the first Born approximation plus 40 dB of noise."""
    y = model.sense(f.to(C128), model.incident())
    y = y + 0.01 * float(y.abs().square().mean().sqrt()) * _randn(seed + 7, *y.shape).to(C128)
    return y.to(C64)


def _solve_inputs(case, seed):
    """Point at which the gradient is taken, and data of the true object."""
    f = _phantom(case["dim"], case["n"], case["shapes"], case["contrast"], case["imag"], seed)
    f = torch.from_numpy(f).to(DEV)
    y = _born_data(_Model(case), f, seed)
    return (0.9 * f).to(C64), y


def _batch_cases(case):
    sizes, txs = [int(v) for v in case["sizes"].split(",")], [int(v) for v in case["txs"].split(",")]
    return [{"dim": 2, "n": n, "T": t, "M": case["M"], "delta": 0.125, "complex_f": case["imag"] > 0, "tx": "plane",
             "shapes": 4, "contrast": case["contrast"], "imag": case["imag"]} for n, t in zip(sizes, txs)]


def _gamma(case):
    """Step size of the order of the inverse Born curvature: receivers see every pixel with about |H_mn|^2."""
    _, rx, _ = _geometry(case)
    k, d = 2.0 * math.pi, _delta(case)
    r = float(np.linalg.norm(rx, axis=1).mean())
    h = k * k * d ** case["dim"] * (0.25 * math.sqrt(2.0 / (math.pi * k * r)) if case["dim"] == 2 else 1.0 / (4.0 * math.pi * r))
    return 1.0 / (case["T"] * case["M"] * case["n"] ** case["dim"] * h * h)


def _fno_params(seed):
    """Flat parameters in the library's layout; weights are BF16 values, as its kernels read them."""
    g = torch.Generator(device="cpu").manual_seed(seed)

    def u(count, scale, bf=True):
        w = (torch.rand(count, generator=g) * 2 - 1) * scale
        return w.bfloat16().float() if bf else w

    parts = [u(FC * 8, 8 ** -0.5), u(FC, 0.1, False)]
    for _ in range(FL):
        parts += [u(2 * FM * FM * FC * FC * 2, 1.0 / FC), u(FC * FC, FC ** -0.5), u(FC, 0.1, False)]
    parts += [u(FH * FC, FC ** -0.5), u(FH, 0.1, False), u(2 * FH, FH ** -0.5), u(2, 0.1, False)]
    return torch.cat(parts)


def _fno_inputs(case, seed):
    B, nf = case["B"], case["B"] if case["per_sample"] else 1
    f = np.stack([synth.ellipse_phantom(FN, 3 + (seed + b) % 7, (0.0, 0.8), 100 * seed + b) for b in range(nf)])
    c = (np.arange(FN) - FN / 2 + 0.5) / 8
    a = 2 * np.pi * (np.arange(B) + 0.1 * (seed % 7)) / B
    u = np.exp(2j * np.pi * (np.cos(a)[:, None, None] * c[None, None, :] + np.sin(a)[:, None, None] * c[None, :, None]))
    lo = _randn(seed + 3, B, 2, 9, 9)  # smooth fields stand in for the demodulated scattered ones
    t = torch.nn.functional.interpolate(torch.view_as_real(lo[:, 0]).permute(0, 3, 1, 2), size=(FN, FN), mode="bicubic")
    t = torch.complex(t[:, 0].contiguous(), t[:, 1].contiguous())
    return torch.from_numpy(f.astype(np.complex64)).to(DEV), torch.from_numpy(u.astype(np.complex64)).to(DEV), 0.5 * t


# --------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    empty = lambda *shape: torch.empty(shape, dtype=C64, device=DEV)  # noqa: E731
    if kind == "fno":
        net = cisor.FNO(max_batch=max(32, case["B"]), seed=1)
        net.set_params(_fno_params(seed))
        f, u, t = _fno_inputs(case, seed)
        grad = torch.empty(net.num_params, dtype=torch.float32, device=DEV)
        return {"case": case, "net": net, "f": f, "u": u, "t": t, "out": torch.empty_like(u), "grad": grad}
    if kind == "batch":
        subs = _batch_cases(case)
        geoms = []
        for s in subs:
            tx, rx, _ = _geometry(s)
            geoms.append(dict(n=s["n"], delta=s["delta"], tx_angles=tx, rx_pos=rx, complex_f=s["complex_f"]))
        ins = [_solve_inputs(s, seed + i) for i, s in enumerate(subs)]
        return {"case": case, "batch": cisor.Batch(geoms, autotune=True), "f": [a for a, _ in ins],
                "y": [b for _, b in ins], "g": [torch.empty_like(a) for a, _ in ins]}
    ctx = _context(case, tuned=kind in ("grad", "step"))
    s = {"case": case, "ctx": ctx}
    if kind == "matvec":
        s.update(f=_contrast_of(case, seed), x=_randn(seed, ctx.T, ctx.Nf), y=empty(ctx.T, ctx.Nf))
    elif kind == "sensing":
        s.update(f=_contrast_of(case, seed), u=_randn(seed, ctx.T, ctx.Nf), w=_randn(seed + 1, ctx.T, ctx.M),
                 Z=empty(ctx.T, ctx.M), z=empty(ctx.T, ctx.Nf), b=empty(ctx.T, ctx.Nf))
    elif kind == "prox":
        z = _contrast_of(case, seed)
        s.update(z=z + 0.1 * _randn(seed, *z.shape), x=torch.empty_like(z))
    else:
        f, y = _solve_inputs(case, seed)
        s.update(f=f, y=y, g=torch.empty_like(f), fk=torch.empty_like(f), sk=torch.empty_like(f), gamma=_gamma(case))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "matvec":
        s["ctx"].apply_A(s["f"], s["x"], s["y"], adjoint=case["adjoint"])
        return {"y": s["y"]}
    if kind == "sensing":
        s["ctx"].sense(s["f"], s["u"], s["Z"])
        s["ctx"].sense_adjoint(s["f"], s["w"], s["z"], s["b"])
        return {"Z": s["Z"], "z": s["z"], "b": s["b"]}
    if kind == "prox":
        s["ctx"].tv_prox(s["z"], s["x"], TV, case["iters"], 0.0, 2.0, 0.0, 0.5, aniso=case["aniso"])
        return {"x": s["x"]}
    if kind == "grad":
        D, _, _ = s["ctx"].grad(s["f"], s["y"], s["g"], tol=TOL)
        return {"D": D, "g": s["g"]}
    if kind == "step":  # one relaxed-FISTA iteration from the same state each time
        s["fk"].copy_(s["f"])
        s["sk"].copy_(s["f"])
        st = s["ctx"].new_state(s["fk"], s["sk"], 0.96, s["gamma"], TV / s["gamma"], 20)
        st.t = 2.0  # past the first iteration, where the momentum is not zero
        s["ctx"].step(st, s["y"], tol=TOL, x0_mode=0)
        return {"D": st.D, "f": s["fk"], "s": s["sk"]}
    if kind == "batch":
        D, _, _ = s["batch"].grad(s["f"], s["y"], s["g"], tol=TOL)
        return {"D": D, "g": s["g"]}
    if case["grad"]:
        loss = s["net"].loss_grad(s["f"], s["u"], s["t"], s["grad"], f_per_sample=case["per_sample"])
        return {"loss": loss, "grad": s["grad"]}
    s["net"].forward(s["f"], s["u"], s["out"], f_per_sample=case["per_sample"])
    return {"out": s["out"]}


TOL = 1e-4   # relative residual of the field solves
TV = 5e-3    # gamma tau of the prox


# --------------------------------------------------------------------------- least work of a pass
def work(case):
    kind = case["kind"]
    if kind == "fno":
        B, px = case["B"], FN * FN
        nf = B if case["per_sample"] else 1
        weights = 2 * (FL * 2 * FM * FM * FC * FC * 2 + FL * FC * FC + FH * FC)
        layer = 2 * FC * FC * px + 2 * 8.0 * FC * (FN * FN * FM + FN * 2 * FM * FM) / 2 + 8.0 * FC * FC * 2 * FM * FM
        flops = B * (2 * 8 * FC * px + FL * layer + 2 * FC * FH * px + 4 * FH * px)
        if case["grad"]:
            return {"bytes": 8.0 * px * (nf + 2 * B) + weights + 2 * weights, "flops": 3.0 * flops}
        return {"bytes": 8.0 * px * (nf + 2 * B) + weights, "flops": flops}
    if kind == "batch":
        parts = [_solve_work(s, case["its"]) for s in _batch_cases(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    N = float(case["n"] ** case["dim"])
    if kind == "prox":
        planes = 2 if case["complex_f"] else 1
        return {"bytes": 16.0 * N, "flops": 12.0 * case["dim"] * planes * N * case["iters"]}
    nc = 3 if case.get("tx") == "vector" else 1
    if kind == "matvec":
        return {"bytes": 8 * (2 * case["T"] * nc * N + N), "flops": case["T"] * nc * _fft_flops(case)}
    if kind == "sensing":
        H = case["M"] * nc * N
        return {"bytes": 8 * (2 * H + 3 * case["T"] * nc * N), "flops": 16.0 * case["T"] * H}
    b, f = _solve_work(case, case["its"])
    return {"bytes": b, "flops": f}


def _fft_flops(case):
    cells = (2.0 * case["n"]) ** case["dim"]
    return 2 * 5 * cells * math.log2(cells) + 6 * cells


def _solve_work(case, its):
    """Two solves of `its` iterations (two operator applications and one vector update each) and the sensing."""
    nc = 3 if case.get("tx") == "vector" else 1
    Nf = nc * float(case["n"] ** case["dim"])
    H = case["M"] * Nf
    passes = 2 * (2 * its + 2) + 1
    return (8 * case["T"] * Nf * (2 * passes + 2 * 5 * its) + 16 * H,
            case["T"] * (nc * passes * _fft_flops(case) + 2 * its * 40 * Nf) + 16.0 * case["T"] * H)


# --------------------------------------------------------------------------- the same paths in 64 bits
def _hankel(order, x):
    """H^(1) of order 0 or 1 from its Laplace integral in t = s^2, by the trapezoidal rule (DLMF 10.9, error about
    exp(-2 pi sqrt(x) / h)); torch's own Bessel functions are good to 4e-7 only."""
    h = min(0.25, 0.19 * math.sqrt(float(x.min())))
    acc = torch.zeros(x.shape, dtype=C128, device=x.device)
    for j in range(int(6.2 / h) + 1):
        s2 = (j * h) ** 2
        root = torch.sqrt(torch.complex(torch.ones_like(x), s2 / (2 * x)))
        wt = h * math.exp(-s2) * (0.5 if j == 0 else 1.0)
        acc += 2 / math.sqrt(math.pi) * wt / root if order == 0 else 4 / math.sqrt(math.pi) * wt * s2 * root
    return torch.polar(torch.sqrt(2 / (math.pi * x)), x - (0.25 + 0.5 * order) * math.pi) * acc


class _Model:
    """Operators of one geometry in FP64: padded-FFT convolution with the Green's function, sensing, incident fields."""

    def __init__(self, case):
        self.case = case
        self.dim, self.n, self.T = case["dim"], case["n"], case["T"]
        self.vec = case.get("tx") == "vector"
        self.d, self.k = _delta(case), 2.0 * math.pi
        tx, rx, mask = _geometry(case)
        self.tx, self.rx = (torch.from_numpy(np.asarray(v, dtype=np.float64)).to(DEV) for v in (tx, rx))
        self.mask = None if mask is None else torch.from_numpy(mask).to(DEV).to(F64)
        c = (torch.arange(self.n, dtype=F64, device=DEV) - self.n / 2 + 0.5) * self.d
        g = torch.meshgrid(*[c] * self.dim, indexing="ij")
        self.pts = torch.stack([v.reshape(-1) for v in reversed(g)], 1)  # x first
        self.spec = None

    def green(self, r):
        if self.dim == 2:
            return 0.25j * _hankel(0, self.k * r)
        return torch.polar(1.0 / (4.0 * math.pi * r), self.k * r)

    def self_term(self):
        k, d = self.k, self.d
        if self.dim == 2:
            a = d / math.sqrt(math.pi)
            h1 = complex(_hankel(1, torch.tensor([k * a], dtype=F64, device=DEV))[0])
            return k * k * (1j * math.pi * a / (2 * k) * h1 - 1 / (k * k))
        a = d * (3.0 / (4.0 * math.pi)) ** (1.0 / 3.0)
        return (1 - 1j * k * a) * complex(math.cos(k * a), math.sin(k * a)) - 1

    def conv(self, x, adjoint=False):
        """G x (or G^H x) of [..., n(, n), n] fields."""
        P, n, dim = 2 * self.n, self.n, self.dim
        axes = tuple(range(-dim, 0))
        if self.spec is None:
            m = torch.arange(P, dtype=F64, device=DEV)
            m = torch.where(m < n, m, m - P)
            r = self.d * torch.sqrt(sum(v * v for v in torch.meshgrid(*[m] * dim, indexing="ij")))
            zero = (0,) * dim
            r[zero] = 1.0
            c = self.k ** 2 * self.d ** dim * self.green(r)
            c[zero] = self.self_term()
            for a in range(dim):  # the offset -n is not used
                c.select(a, n).zero_()
            self.spec = torch.fft.fftn(c, dim=axes)
        s = self.spec.conj() if adjoint else self.spec
        y = torch.fft.ifftn(s * torch.fft.fftn(x, s=(P,) * dim, dim=axes), dim=axes)
        for a in axes:
            y = y.narrow(a, 0, n)
        return y

    def grid(self, x):
        return x.reshape(x.shape[0], *([3] if self.vec else []), *[self.n] * self.dim)

    def graddiv(self, B):
        """Finite-difference grad div of [T, 3, z, y, x], zero outside the grid."""
        n, h = self.n, self.d
        Pd = torch.nn.functional.pad(B, (1, 1, 1, 1, 1, 1))

        def at(c, off):
            v = Pd[:, c]
            for comp in range(3):
                v = v.narrow(3 - comp, 1 + off.get(comp, 0), n)
            return v

        out = torch.empty_like(B)
        for c in range(3):
            acc = (at(c, {c: 1}) - 2 * at(c, {}) + at(c, {c: -1})) / h ** 2
            for j in range(3):
                if j != c:
                    acc = acc + (at(j, {c: -1, j: -1}) - at(j, {c: -1, j: 1}) - at(j, {c: 1, j: -1})
                                 + at(j, {c: 1, j: 1})) / (4 * h ** 2)
            out[:, c] = acc
        return out

    def apply(self, f, x, adjoint):
        """A x or A^H x for flat fields [T, Nf] and a flat contrast [N]."""
        out = torch.empty_like(x)
        fg = f.reshape(*[self.n] * self.dim)
        rows = max(1, int(2e8 // ((2 * self.n) ** self.dim * (3 if self.vec else 1))))
        for i in range(0, x.shape[0], rows):
            v = self.grid(x[i:i + rows])
            if adjoint:
                w = v + self.graddiv(v) / self.k ** 2 if self.vec else v
                y = v - fg.conj() * self.conv(w, True)
            else:
                c = self.conv(fg * v)
                y = v - c - (self.graddiv(c) / self.k ** 2 if self.vec else 0)
            out[i:i + rows] = y.reshape(y.shape[0], -1)
        return out

    def gz(self, z, v):
        out = torch.empty_like(z)
        rows = max(1, int(2e8 // ((2 * self.n) ** self.dim * (3 if self.vec else 1))))
        for i in range(0, z.shape[0], rows):
            w = self.grid(v[i:i + rows])
            w = w + self.graddiv(w) / self.k ** 2 if self.vec else w
            out[i:i + rows] = z[i:i + rows] + self.conv(w, True).reshape(w.shape[0], -1)
        return out

    def incident(self):
        k = self.k
        if self.case.get("tx", "plane") == "point":
            return self.green(torch.cdist(self.tx, self.pts, compute_mode="donot_use_mm_for_euclid_dist"))
        dirs = self.tx[:, :3] if self.dim == 3 else torch.stack([self.tx.cos(), self.tx.sin()], 1)
        u = torch.exp(1j * k * (dirs @ self.pts.T))
        if self.vec:
            u = (self.tx[:, 3:, None] * u[:, None]).reshape(self.T, -1)
        return u

    def rows(self):
        """Row blocks of the sensing matrix, as (first receiver, [m, Nf])."""
        step = max(1, int(3e7 // self.pts.shape[0]))
        for i in range(0, self.rx.shape[0], step):
            dv = self.rx[i:i + step, None, :] - self.pts[None]
            r = dv.square().sum(-1).sqrt()
            h = self.k ** 2 * self.d ** self.dim * self.green(r)
            if self.vec:
                kr = self.k * r
                a, b = 3 / kr ** 2 - 3j / kr - 1, 1 + 1j / kr - 1 / kr ** 2
                rh = dv / r[..., None]
                h = torch.cat([h * (a * rh[..., 2] * rh[..., c] + (b if c == 2 else 0)) for c in range(3)], 1)
            yield i, h

    def sense(self, f, u):
        fu = (f.reshape(-1).repeat(3 if self.vec else 1) * u).T.contiguous()
        return torch.cat([h @ fu for _, h in self.rows()], 0).T.contiguous()

    def sense_adjoint(self, w):
        return sum(w[:, i:i + h.shape[0]] @ h.conj() for i, h in self.rows())

    def solve(self, f, b, adjoint, x):
        """BiCGSTAB per transmitter from x to a true relative residual of TOL, restarted where the recurrence drifted."""
        dot = lambda a, c: (a.conj() * c).sum(1, keepdim=True)  # noqa: E731
        bn = b.norm(dim=1, keepdim=True)
        for _ in range(6):
            r = b - self.apply(f, x, adjoint)
            act = (r.norm(dim=1, keepdim=True) > TOL * bn)
            if not bool(act.any()):
                break
            rh, rho = r.clone(), dot(r, r)
            p = r.clone()
            for _ in range(500):
                v = self.apply(f, p, adjoint)
                alpha = rho / dot(rh, v)
                s = r - alpha * v
                t = self.apply(f, s, adjoint)
                omega = dot(t, s) / dot(t, t)
                x = torch.where(act, x + alpha * p + omega * s, x)
                r = torch.where(act, s - omega * t, r)
                act = act & (r.norm(dim=1, keepdim=True) > TOL * bn)
                if not bool(act.any()):
                    break
                new = dot(rh, r)
                p = r + (new / rho) * (alpha / omega) * (p - omega * v)
                rho = new
        return x

    def data_and_grad(self, f, y):
        f = f.reshape(-1)
        u_in = self.incident()
        u = self.solve(f, u_in, False, u_in.clone())
        w = self.sense(f, u) - y
        if self.mask is not None:
            w = w * self.mask
        z = self.sense_adjoint(w)
        fr = f.repeat(3 if self.vec else 1)
        v = self.solve(f, fr.conj() * z, True, torch.zeros_like(z))
        g = (u.conj() * self.gz(z, v)).sum(0)
        return 0.5 * float(w.abs().square().sum()), g.reshape(-1, f.numel()).sum(0)


def _diff(x, a):
    """Forward difference along axis a, zero at the last index."""
    d = torch.zeros_like(x)
    d.narrow(a, 0, x.shape[a] - 1).copy_(x.narrow(a, 1, x.shape[a] - 1) - x.narrow(a, 0, x.shape[a] - 1))
    return d


def _diff_t(p, a):
    """Adjoint of _diff."""
    out, m = torch.zeros_like(p), p.shape[a] - 1
    out.narrow(a, 0, m).sub_(p.narrow(a, 0, m))
    out.narrow(a, 1, m).add_(p.narrow(a, 0, m))
    return out


def _fgp(z, lam, iters, lo, hi):
    dim = z.dim()
    p, t = torch.zeros(dim, *z.shape, dtype=F64, device=z.device), 1.0
    r = p.clone()
    div = lambda q: sum(_diff_t(q[a], a) for a in range(dim))  # noqa: E731
    for _ in range(iters):
        x = (z - lam * div(r)).clamp(lo, hi)
        q = r + torch.stack([_diff(x, a) for a in range(dim)]) / (4 * dim * lam)
        q = q / q.square().sum(0).sqrt().clamp(min=1.0)
        tn = (1 + math.sqrt(1 + 4 * t * t)) / 2
        r, p, t = q + (t - 1) / tn * (q - p), q, tn
    return (z - lam * div(p)).clamp(lo, hi)


def _ppa(z, lam, iters, lo, hi):
    """Anisotropic TV: parallel proximal iteration over the even and odd pairs of every axis and the box."""
    dim, m = z.dim(), 2 * z.dim() + 1
    zs, x = [z.clone() for _ in range(m)], z
    for _ in range(iters):
        ps = []
        for j in range(2 * dim):
            a, first = j >> 1, j & 1
            q, pairs = zs[j].clone(), (z.shape[a] - first) // 2
            if pairs > 0:
                v = q.narrow(a, first, 2 * pairs).unflatten(a, (pairs, 2))
                lo_, hi_ = v.select(a + 1, 0).clone(), v.select(a + 1, 1).clone()
                dd = hi_ - lo_
                dd = torch.sign(dd) * (dd.abs() - 2 * m * lam).clamp(min=0)
                v.select(a + 1, 0).copy_(0.5 * (lo_ + hi_ - dd))
                v.select(a + 1, 1).copy_(0.5 * (lo_ + hi_ + dd))
            ps.append(q)
        ps.append(zs[-1].clamp(lo, hi))
        x = sum(ps) / m
        zs = [x + a - b for a, b in zip(zs, ps)]
    return x


def _prox64(z, iters, complex_f, aniso=False):
    fn = _ppa if aniso else _fgp
    re = fn(z.real.contiguous(), TV, iters, 0.0, 2.0)
    return torch.complex(re, fn(z.imag.contiguous(), TV, iters, 0.0, 0.5) if complex_f else torch.zeros_like(re))


def _fno64(flat, f, u, per_sample):
    """The network in FP64 with its parameters as one differentiable vector."""
    pos = 0

    def take(*shape):
        nonlocal pos
        count = math.prod(shape)
        pos += count
        return flat[pos - count:pos].reshape(shape)

    B = u.shape[0]
    f = f if per_sample else f.expand(B, FN, FN)
    up = torch.cat([u[:, :, :1], u, u[:, :, -1:]], 2)
    vx = (u.conj() * (up[:, :, 2:] - up[:, :, :-2])).imag
    up = torch.cat([u[:, :1], u, u[:, -1:]], 1)
    vy = (u.conj() * (up[:, 2:] - up[:, :-2])).imag
    nv = torch.sqrt(vx * vx + vy * vy)
    nv = torch.where(nv > 0, nv, torch.ones_like(nv))
    c = (torch.arange(FN, dtype=F64, device=DEV) + 0.5) / FN - 0.5
    X, Y = c[None, None, :].expand(B, FN, FN), c[None, :, None].expand(B, FN, FN)
    a = torch.stack([f.real, f.imag, u.real, u.imag, vx / nv, vy / nv, X, Y], 1)
    W0, b0 = take(FC, 8), take(FC)
    v = torch.einsum("oc,bcyx->boyx", W0, a) + b0[:, None, None]
    kx = torch.cat([torch.arange(FM), torch.arange(FN - FM, FN)]).to(DEV).to(F64)
    i = torch.arange(FN, dtype=F64, device=DEV)
    Fx = torch.exp(-2j * math.pi * torch.outer(kx, i) / FN)
    Fy = torch.exp(-2j * math.pi * torch.outer(i[:FM], i) / FN)
    wk = torch.full((FM,), 2.0, dtype=F64, device=DEV)
    wk[0] = 1.0
    gelu = lambda x: 0.5 * x * (1 + torch.erf(x / math.sqrt(2.0)))  # noqa: E731
    for l in range(FL):
        R = torch.view_as_complex(take(2 * FM, FM, FC, FC, 2))
        W, b = take(FC, FC), take(FC)
        S = Fx @ (v.to(C128) @ Fy.T)
        S = torch.einsum("klio,bikl->bokl", R, S) * (wk / FN ** 2)
        pre = (Fx.conj().T @ S @ Fy.conj()).real + torch.einsum("oi,biyx->boyx", W, v) + b[:, None, None]
        v = gelu(pre) if l < FL - 1 else pre
    P1, c1, P2, c2 = take(FH, FC), take(FH), take(2, FH), take(2)
    h = gelu(torch.einsum("hc,bcyx->bhyx", P1, v) + c1[:, None, None])
    o = torch.einsum("oh,bhyx->boyx", P2, h) + c2[:, None, None]
    return torch.complex(o[:, 0], o[:, 1])


def _fno_exact(case, seed):
    f, u, t = (v.to(C128) for v in _fno_inputs(case, seed))
    flat = _fno_params(seed).to(DEV).to(F64)
    nf, B = f.shape[0], u.shape[0]
    if not case["grad"]:
        outs = [_fno64(flat, f[i:i + 8] if nf == B else f, u[i:i + 8], nf == B) for i in range(0, B, 8)]
        return {"out": torch.cat(outs)}
    loss, grad = 0.0, torch.zeros_like(flat)
    for i in range(0, B, 8):
        p = flat.clone().requires_grad_(True)
        e = _fno64(p, f[i:i + 8] if nf == B else f, u[i:i + 8], nf == B) - t[i:i + 8]
        part = (e.abs().square().sum((1, 2)).sqrt() / t[i:i + 8].abs().square().sum((1, 2)).sqrt()).sum() / B
        part.backward()
        loss, grad = loss + float(part.detach()), grad + p.grad
    return {"loss": torch.tensor(loss, dtype=F64), "grad": grad}


def exact(case, seed):
    kind = case["kind"]
    if kind == "fno":
        return _fno_exact(case, seed)
    if kind == "batch":
        outs = []
        for i, s in enumerate(_batch_cases(case)):
            f, y = _solve_inputs(s, seed + i)
            D, g = _Model(s).data_and_grad(f.to(C128), y.to(C128))
            outs.append((D, g.reshape(f.shape)))
        return {"D": [torch.tensor(D, dtype=F64) for D, _ in outs], "g": [g for _, g in outs]}
    if kind == "prox":
        z = _contrast_of(case, seed)
        z = z + 0.1 * _randn(seed, *z.shape)
        return {"x": _prox64(z.to(C128), case["iters"], case["complex_f"], case["aniso"])}
    m = _Model(case)
    Nf = case["n"] ** case["dim"] * (3 if m.vec else 1)
    if kind == "matvec":
        f = _contrast_of(case, seed).to(C128).reshape(-1)
        return {"y": m.apply(f, _randn(seed, case["T"], Nf).to(C128), case["adjoint"])}
    if kind == "sensing":
        f = _contrast_of(case, seed).to(C128).reshape(-1)
        z = m.sense_adjoint(_randn(seed + 1, case["T"], case["M"]).to(C128))
        return {"Z": m.sense(f, _randn(seed, case["T"], Nf).to(C128)), "z": z, "b": f.conj().repeat(Nf // f.numel()) * z}
    f, y = _solve_inputs(case, seed)
    D, g = m.data_and_grad(f.to(C128), y.to(C128))
    D = torch.tensor(D, dtype=F64)
    if kind == "grad":
        return {"D": D, "g": g.reshape(f.shape)}
    s0 = f.to(C128)
    if not case["complex_f"]:
        g = g.real.to(C128)
    x = _prox64(s0 - _gamma(case) * g.reshape(f.shape), 20, case["complex_f"])
    beta = 0.96 * (2.0 - 1.0) / ((math.sqrt(4 * 2.0 ** 2 + 1) + 1) / 2)
    return {"D": D, "f": x, "s": x + beta * (x - s0)}
