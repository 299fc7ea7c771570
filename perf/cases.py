"""The calls of this library whose speed is measured, over the sizes they are used at.

A case is a dict of plain values with a ``kind``:

operator   lsw.apply_operator: the FFT operator, the product of every Krylov
           or series step and (adjoint) of every sketch.
precond    lsw.apply_precond: one product with a HODLR preconditioner.
solve      lsw.solve_series with a preconditioner the program already holds.
frequency  everything one frequency costs: Green table, contrast, sources,
           preconditioner, solve.
sweep      lsw.solve_sweep: several frequencies under the paper's rank policy.
train      one training step of the learned preconditioner (loss, gradients,
           Adam), at the end of the learning-rate decay.
learned    lsw.FNO.apply: the learned preconditioner on Krylov vectors.

Solves run to a residual of 1e-11 (the library's own checks against a direct
solution use 1e-10 and 1e-11), so that their fields are determined to far
below the comparison's resolution whatever the rounding inside the
preconditioner.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2005_01372_gb300 import lsw, media

PRECS = {"c128": lsw.C128, "c64": lsw.C64, "bf16": lsw.BF16, "mixed": lsw.MIXED}
MODES = {"forward": lsw.OP_FORWARD, "residual": lsw.OP_RESIDUAL, "plain": lsw.OP_PLAIN, "adjoint": lsw.OP_ADJOINT}
C0 = 2000.0
TOL = 1e-11


def listed():
    return [
        # One source on the smallest model of the paper's plain method: a
        # series step's operator call where launches and latency count.
        {"name": "operator-64x64-1", "kind": "operator", "nz": 64, "nx": 64, "h": 10.0, "freq": 10.0, "batch": 1,
         "prec": "c64", "mode": "forward"},
        # The residual of a 32-source problem, the ordinary Krylov step.
        {"name": "operator-256x256-32", "kind": "operator", "nz": 256, "nx": 256, "h": 10.0, "freq": 15.0,
         "batch": 32, "prec": "c64", "mode": "residual"},
        # The same at the largest benchmark model.
        {"name": "operator-1024x1024-16", "kind": "operator", "nz": 1024, "nx": 1024, "h": 5.0, "freq": 30.0,
         "batch": 16, "prec": "c64", "mode": "residual"},
        # The adjoint on a block of probes, as the sketches use it, on the
        # long embedded salt grid: non-square, a batch that is no power of two.
        {"name": "adjoint-256x1024-30", "kind": "operator", "nz": 256, "nx": 1024, "h": 10.0, "freq": 10.0,
         "batch": 30, "prec": "c64", "mode": "adjoint"},
        # The FP64 residual of iterative refinement.
        {"name": "operator-256x256-32-c128", "kind": "operator", "nz": 256, "nx": 256, "h": 10.0, "freq": 15.0,
         "batch": 32, "prec": "c128", "mode": "residual"},
        # H applied to the Krylov vectors of 32 sources, FP32 storage, at a low
        # frequency of the sweep (the start of the paper's ascending order).
        {"name": "precond-256x256-32", "kind": "precond", "nz": 256, "nx": 256, "h": 10.0, "freq": 2.0, "batch": 32,
         "prec": "c64", "levels": 6, "rank": 20, "over": 10},
        # The plain method in double precision: the preconditioned series on
        # the small inclusion, a few sources.
        {"name": "solve-64x64-3-c128", "kind": "solve", "nz": 64, "nx": 64, "h": 10.0, "freq": 10.0, "batch": 3,
         "prec": "c128", "hprec": "c128", "method": "series", "medium": "inclusion", "levels": 2, "rank": 20,
         "over": 10},
        # 16 sources against a BF16 preconditioner: FGMRES in FP32 inside FP64
        # refinement, the benchmark's solver at half its grid.
        {"name": "solve-512x512-16-bf16", "kind": "solve", "nz": 512, "nx": 512, "h": 5.0, "freq": 15.0, "batch": 16,
         "prec": "mixed", "hprec": "bf16", "method": "fgmres", "medium": "marmousi", "levels": 8, "rank": 40,
         "over": 10},
        # One frequency of the layered salt model, everything included.
        {"name": "frequency-256x256-32", "kind": "frequency", "nz": 256, "nx": 256, "h": 10.0, "freq": 15.0,
         "batch": 32, "prec": "mixed", "hprec": "c64", "method": "fgmres", "medium": "salt", "levels": 6, "rank": 20,
         "over": 10},
        # The paper's own experiment: ascending frequencies, one source, the
        # preconditioned series under the rank policy.
        {"name": "sweep-128x256-6", "kind": "sweep", "nz": 128, "nx": 256, "h": 15.0, "freq": 4.0, "nfreq": 6,
         "batch": 1, "prec": "mixed", "hprec": "c64", "method": "series", "medium": "subset", "levels": 5, "rank": 10,
         "over": 10},
        # A training step of the learned preconditioner at its full size.
        {"name": "train-256x256-32", "kind": "train", "nz": 256, "nx": 256, "width": 32, "modes": 16, "layers": 4,
         "batch": 32},
        # The learned preconditioner on the Krylov vectors of 8 sources.
        {"name": "learned-256x256-8", "kind": "learned", "nz": 256, "nx": 256, "h": 10.0, "freq": 15.0, "width": 32,
         "modes": 16, "layers": 4, "batch": 8, "prec": "c64"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["operator"] * 4 + ["precond", "solve", "frequency", "sweep", "train", "train", "learned"])
    if kind == "operator":
        # grid sides are powers of two; batches are whatever a program has
        nz, nx = 1 << rng.randint(4, 10), 1 << rng.randint(4, 10)
        most = max(1, min(200, (1 << 24) // (nz * nx)))
        prec = rng.choice(["c64", "c64", "c64", "c128"])
        if prec == "c128":
            most = max(1, most // 8)
        return {"kind": kind, "nz": nz, "nx": nx, "h": 10.0, "freq": round(rng.uniform(5.0, 15.0), 2),
                "batch": _log(rng, 1, most), "prec": prec, "mode": rng.choice(list(MODES))}
    if kind == "precond":
        lz, lx = rng.randint(6, 8), rng.randint(6, 8)
        return {"kind": kind, "nz": 1 << lz, "nx": 1 << lx, "h": 10.0, "freq": round(rng.uniform(1.0, 2.5), 2),
                "batch": _log(rng, 1, 40), "prec": "c64", "levels": lz + lx - 10 + rng.randint(0, 2),
                "rank": rng.randint(8, 24), "over": 10}
    if kind in ("solve", "frequency"):
        lz, lx = rng.randint(6, 8), rng.randint(6, 8)
        return {"kind": kind, "nz": 1 << lz, "nx": 1 << lx, "h": 10.0, "freq": round(rng.uniform(3.0, 10.0), 2),
                "batch": _log(rng, 1, 32), "prec": "mixed", "hprec": rng.choice(["c64", "bf16"]), "method": "fgmres",
                "medium": "random", "levels": lz + lx - 10 + rng.randint(0, 1), "rank": rng.randint(16, 24),
                "over": 10}
    if kind == "sweep":
        lz, lx = rng.randint(6, 7), rng.randint(6, 8)
        return {"kind": kind, "nz": 1 << lz, "nx": 1 << lx, "h": 10.0, "freq": round(rng.uniform(1.0, 3.0), 2),
                "nfreq": rng.randint(2, 4), "batch": rng.randint(1, 4), "prec": "mixed", "hprec": "c64",
                "method": "fgmres", "medium": "random", "levels": lz + lx - 10, "rank": 10, "over": 10}
    # the network runs on grids of any size
    nz, nx = _log(rng, 32, 256), _log(rng, 32, 256)
    width, modes, layers = rng.randint(4, 36), rng.randint(3, 16), rng.randint(1, 5)
    most = max(1, min(64, int(32 * 256 * 256 * 32 * 4 / (nz * nx * max(width, 8) * (layers + 1)))))
    case = {"kind": kind, "nz": nz, "nx": nx, "width": width, "modes": modes, "layers": layers,
            "batch": _log(rng, 1, most)}
    if kind == "learned":
        # applied on a problem's grid: powers of two
        case.update(nz=1 << rng.randint(5, 8), nx=1 << rng.randint(5, 8), h=10.0, freq=round(rng.uniform(10, 25), 2),
                    batch=min(case["batch"], 32), prec=rng.choice(["c64", "c128"]))
    return case


# --------------------------------------------------------------- inputs

def _velocity(case, seed):
    """A model (nx, nz) and one update of it: a smooth perturbation of up to
    1 % such as an inversion's iterations make."""
    nz, nx, h = case["nz"], case["nx"], case["h"]
    medium = case.get("medium", "random")
    if medium == "inclusion":
        c = media.gaussian_inclusion(nz, nx, h)
    elif medium == "marmousi":
        c = media.marmousi_like(np.random.default_rng(4), nz, nx, h)
    elif medium == "salt":
        rng = np.random.default_rng(2)
        c = media.salt_ellipse(rng, media.layered(rng, nz, nx, h), h)
    elif medium == "subset":
        c = media.marmousi_subset().velocity
    else:
        rng = np.random.default_rng(31)
        c = media.gaussian_anomalies(rng, media.layered(rng, nz, nx, h), h)
    rng = np.random.default_rng(seed)
    z, x = np.arange(nz)[None, :] / nz, np.arange(nx)[:, None] / nx
    d = np.zeros((nx, nz))
    for _ in range(4):
        kz, kx = rng.integers(1, 5, size=2)
        d += np.cos(2 * np.pi * (kz * z + rng.uniform())) * np.cos(2 * np.pi * (kx * x + rng.uniform()))
    if medium == "subset":
        d *= (c != C0)                  # the embedding keeps its zero contrast
    return c * (1.0 + 0.0025 * d)


def _sources(case, seed):
    rng = np.random.default_rng(seed + 7)
    ix = rng.choice(case["nx"], size=case["batch"], replace=case["batch"] > case["nx"])
    return [(0, int(i)) for i in np.sort(ix)]


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _fields(g, count, n, dtype):
    return torch.randn((count, n), generator=g, device="cuda", dtype=dtype)


def _smooth_fields(g, count, nz, nx):
    """Smooth complex fields of unit norm: residuals as a solve meets them."""
    f = torch.fft.fft2(torch.randn((count, nx, nz), generator=g, device="cuda", dtype=torch.complex64))
    kx = torch.fft.fftfreq(nx, device="cuda")[:, None]
    kz = torch.fft.fftfreq(nz, device="cuda")[None, :]
    f = torch.fft.ifft2(f * torch.exp(-60.0 * (kx * kx + kz * kz))).reshape(count, nx * nz)
    return f / f.norm(dim=1, keepdim=True)


def _network(case, seed):
    """Weights scaled like the library's own initial ones, biases included."""
    W, L, MM = case["width"], case["layers"], (2 * case["modes"]) ** 2
    g = _generator(seed + 3)

    def w(count, scale):
        return torch.randn(count, generator=g, device="cuda", dtype=torch.complex64) * scale
    parts = [w(2 * W, 2.0 ** -0.5), w(W, 0.01)]
    for _ in range(L):
        parts += [w(MM * W * W, 1.0 / W), w(W * W, W ** -0.5), w(W, 0.01)]
    parts += [w(W, W ** -0.5), w(1, 0.01)]
    return torch.cat(parts)


def _hparams(case, prec):
    return lsw.HParams(kind=lsw.H_HODLR, prec=PRECS[prec], levels=case["levels"], rank=case["rank"],
                       oversample=case["over"], seed=1002)


def _sparams(case):
    fgmres = case["method"] == "fgmres"
    return lsw.SolveParams(prec=PRECS[case["prec"]], method=lsw.FGMRES if fgmres else lsw.SERIES, tol=TOL,
                           inner_tol=1e-3, restart=30, max_iter=60, max_outer=16)


def _train_inputs(case, seed):
    nz, nx, B = case["nz"], case["nx"], case["batch"]
    g = _generator(seed)
    r = _smooth_fields(g, B, nz, nx)
    c = 1500.0 + 3000.0 * torch.rand((B, 1, nz), generator=g, device="cuda").expand(B, nx, nz).reshape(B, nx * nz)
    x1 = torch.complex((C0 / c) ** 2 - 1.0, torch.full_like(c, 2 * math.pi * 15.0 / C0 * 10.0))
    t = r + 0.5 * _smooth_fields(g, B, nz, nx)
    return torch.stack([r, x1], dim=1).contiguous(), t.contiguous()


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "train":
        s["net"] = lsw.FNO(case["nz"], case["nx"], case["width"], case["modes"], case["layers"], seed=1)
        s["net"].set(_network(case, seed))
        s["x"], s["t"] = _train_inputs(case, seed)
        s["step"] = 0
        return s
    vel = torch.from_numpy(np.ascontiguousarray(_velocity(case, seed).ravel())).cuda()
    if kind in ("frequency", "sweep"):
        s["velocity"], s["sources"] = vel, _sources(case, seed)
        return s
    s["G"] = lsw.build_green(case["nz"], case["nx"], case["h"], C0, case["freq"])
    s["chi"] = s["G"].contrast(vel)
    n = s["G"].n
    if kind == "solve":
        s["H"] = lsw.build_hmatrix(s["G"], s["chi"], _hparams(case, case["hprec"]))
        s["u0"] = s["G"].point_sources(_sources(case, seed), lsw.C128)
        return s
    g = _generator(seed)
    dtype = torch.complex128 if case["prec"] == "c128" else torch.complex64
    if kind == "learned":
        s["net"] = lsw.FNO(case["nz"], case["nx"], case["width"], case["modes"], case["layers"], seed=1)
        s["net"].set(_network(case, seed))
        s["v"] = (3.0 * _smooth_fields(g, case["batch"], case["nz"], case["nx"])).to(dtype)
        return s
    s["u"] = _fields(g, case["batch"], n, dtype)
    if kind == "operator":
        s["u0"] = _fields(g, case["batch"], n, dtype) if case["mode"] in ("forward", "residual") else None
    else:
        s["H"] = lsw.build_hmatrix(s["G"], s["chi"], _hparams(case, case["prec"]))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "operator":
        return lsw.apply_operator(s["G"], s["chi"], s["u"], s["u0"], MODES[case["mode"]])
    if kind == "precond":
        return lsw.apply_precond(s["H"], s["u"])
    if kind == "solve":
        return lsw.solve_series(s["G"], s["chi"], s["H"], s["u0"], sp=_sparams(case))[0]
    if kind == "frequency":
        G = lsw.build_green(case["nz"], case["nx"], case["h"], C0, case["freq"])
        chi = G.contrast(s["velocity"])
        u0 = G.point_sources(s["sources"], lsw.C128)
        H = lsw.build_hmatrix(G, chi, _hparams(case, case["hprec"]))
        return lsw.solve_series(G, chi, H, u0, sp=_sparams(case))[0]
    if kind == "sweep":
        freqs = [case["freq"] + i for i in range(case["nfreq"])]
        pol = lsw.SweepPolicy(rank0=case["rank"], rank_step=10, rank_max=50, raise_iters=20)
        return lsw.solve_sweep(case["nz"], case["nx"], case["h"], C0, s["velocity"], freqs, s["sources"],
                               _hparams(case, case["hprec"]), pol, _sparams(case))[0]
    if kind == "learned":
        return s["net"].apply(s["G"], s["chi"], s["v"])
    s["step"] += 1
    loss, grad = s["net"].loss_grad(s["x"], s["t"], want_grad=True)
    s["net"].adam_step(1e-5, s["step"])
    return {"loss": loss, "grad": grad, "weights": s["net"].get()}


def work(case):
    """Inputs read once, outputs written once; flops of the transforms and
    products one pass is made of (for a solve, of one iteration)."""
    nz, nx, B = case["nz"], case["nx"], case["batch"]
    n = nz * nx
    if case["kind"] in ("train", "learned"):
        W, MM, L = case["width"], (2 * case["modes"]) ** 2, case["layers"]
        weights = 3 * W + L * (MM * W * W + W * W + W) + W + 1
        # each activation is made once and (training) read once on the way back
        act = 8.0 * n * B * W * L
        m2 = 2 * case["modes"]
        layer = 8.0 * B * W * (2.0 * (m2 * nx * nz + m2 * m2 * nx) + n * W) + 8.0 * B * W * W * MM
        if case["kind"] == "train":
            return {"bytes": 8.0 * (3 * n * B + 10 * weights) + 2 * act, "flops": 3 * L * layer}
        return {"bytes": 8.0 * (2 * n * B + weights) + 8.0 * n, "flops": L * layer}
    pz, px = 2.0 * nz, 2.0 * nx
    op = B * (2 * nx * 5 * pz * math.log2(pz) + 2 * pz * 5 * px * math.log2(px) + 6 * pz * px)
    elem = 16.0 if case["prec"] in ("c128", "mixed") else 8.0
    grid = 8.0 * n + elem * (nz + 1) * (nx + 1)
    if case["kind"] == "operator":
        return {"bytes": elem * n * B * (3 if case["mode"] in ("forward", "residual") else 2) + grid, "flops": op}
    leaf = n >> case["levels"]
    entry = {"c128": 16.0, "c64": 8.0, "bf16": 4.0}[case["hprec" if "hprec" in case else "prec"]]
    entries = float(n) * leaf + 2.0 * n * case["rank"] * case["levels"]
    if case["kind"] == "precond":
        return {"bytes": entry * entries + 16.0 * n * B, "flops": 8.0 * entries * B}
    count = case.get("nfreq", 1)
    if case["kind"] == "solve":
        return {"bytes": entry * entries + 2 * elem * n * B + grid, "flops": 8.0 * entries * B + op}
    return {"bytes": 8.0 * n + count * elem * n * B, "flops": count * (8.0 * entries * B + op)}


# ---------------------------------------------------- the same in 64 bits

def _bessel(x):
    """J0, J1, Y0, Y1 of a tensor of positive numbers: Miller's backward
    recurrence normalised by 1 = J0 + 2 sum J_2k, Neumann's series for Y0 and
    the Wronskian for Y1."""
    top = 2 * ((int(float(x.max())) + 60 + 12 * int(float(x.max()) ** (1 / 3))) // 2)
    hi, lo = torch.zeros_like(x), torch.full_like(x, 1e-200)    # J_{n+1}, J_n up to a factor
    norm, y = torch.zeros_like(x), torch.zeros_like(x)
    one, small = torch.ones_like(x), torch.full_like(x, 1e-100)
    for n in range(top, 0, -1):
        if n % 2 == 0:
            norm += 2 * lo
            y += (1.0 if (n // 2) % 2 else -1.0) * lo / (n // 2)
        hi, lo = lo, (2.0 * n / x) * lo - hi
        scale = torch.where(lo.abs() > 1e100, small, one)
        hi, lo, norm, y = hi * scale, lo * scale, norm * scale, y * scale
    norm += lo
    j0, j1, y = lo / norm, hi / norm, y / norm
    y0 = 2 / math.pi * ((torch.log(x / 2) + 0.57721566490153286) * j0 + 2 * y)
    return j0, j1, y0, (j1 * y0 - 2 / (math.pi * x)) / j0


def _green(case):
    """The cell-integrated Green function at every offset, evenly extended."""
    nz, nx, h = case["nz"], case["nx"], case["h"]
    k = 2 * math.pi * case["freq"] / C0
    a = h / math.sqrt(math.pi)
    pre = math.pi * a / (2 * k)
    dz = torch.arange(nz + 1, dtype=torch.float64, device="cuda")[None, :]
    dx = torch.arange(nx + 1, dtype=torch.float64, device="cuda")[:, None]
    kr = k * h * torch.sqrt(dz * dz + dx * dx)
    kr[0, 0] = 1.0
    _, j1, _, y1 = (float(v) for v in _bessel(torch.tensor([k * a], dtype=torch.float64, device="cuda")))
    j0r, _, y0r, _ = _bessel(kr)
    t = torch.complex(-pre * j1 * y0r, pre * j1 * j0r)
    t[0, 0] = complex(-pre * y1 - 1.0 / (k * k), pre * j1)
    ix = torch.minimum(torch.arange(2 * nx), 2 * nx - torch.arange(2 * nx)).cuda()
    iz = torch.minimum(torch.arange(2 * nz), 2 * nz - torch.arange(2 * nz)).cuda()
    return t, torch.fft.fft2(t[ix][:, iz])


def _chi64(case, seed):
    c = torch.from_numpy(np.ascontiguousarray(_velocity(case, seed).ravel())).cuda()
    w = 2 * math.pi * case["freq"]
    return w * w * (1.0 / (c * c) - 1.0 / (C0 * C0))


def _convolve(case, spec, v):
    nz, nx = case["nz"], case["nx"]
    f = torch.fft.fft2(v.reshape(-1, nx, nz), s=(2 * nx, 2 * nz))
    return torch.fft.ifft2(f * spec)[:, :nx, :nz].reshape(v.shape[0], nx * nz)


def _exact_operator(case, seed):
    g = _generator(seed)
    dtype = torch.complex128 if case["prec"] == "c128" else torch.complex64
    n = case["nz"] * case["nx"]
    u = _fields(g, case["batch"], n, dtype).to(torch.complex128)
    u0 = _fields(g, case["batch"], n, dtype).to(torch.complex128) if case["mode"] in ("forward", "residual") else None
    chi, (_, spec) = _chi64(case, seed), _green(case)
    if case["mode"] == "adjoint":
        return chi * _convolve(case, spec, u.conj()).conj()
    y = torch.cat([_convolve(case, spec, chi * v) for v in u.split(4)])
    return u0 + y if case["mode"] == "forward" else u - y - u0 if case["mode"] == "residual" else y


def _exact_solve(case, seed):
    nz, nx, n = case["nz"], case["nx"], case["nz"] * case["nx"]
    chi, (table, _) = _chi64(case, seed), _green(case)
    i = torch.arange(n, device="cuda")
    ix, iz = i // nz, i % nz
    A = -table[(ix[:, None] - ix[None, :]).abs(), (iz[:, None] - iz[None, :]).abs()] * chi[None, :]
    A.diagonal().add_(1.0)
    b = torch.stack([table[(ix - x).abs(), (iz - z).abs()] for z, x in _sources(case, seed)], dim=1) / case["h"] ** 2
    return torch.linalg.solve(A, b).T.contiguous()


def _exact_network(case, p, x):
    """The network in complex128; p: the flat parameters."""
    nz, nx, W, m, L = case["nz"], case["nx"], case["width"], case["modes"], case["layers"]
    M, B = 2 * m, x.shape[0]
    at = [0]

    def take(*shape):
        count = math.prod(shape)
        at[0] += count
        return p[at[0] - count:at[0]].reshape(shape)

    def act(t):
        return torch.complex(torch.nn.functional.gelu(t.real), torch.nn.functional.gelu(t.imag))

    def rows(k, count):
        k = torch.cat([torch.arange(k), torch.arange(count - k, count)]).cuda().double()
        i = torch.arange(count, device="cuda").double()
        turn = torch.remainder(k[:, None] * i[None, :], count) * (-2 * math.pi / count)
        return torch.polar(torch.ones_like(turn), turn)

    Fz, Fx = rows(m, nz), rows(m, nx)
    v = torch.einsum("wc,bcn->bwn", take(W, 2), x) + take(W)[None, :, None]
    for layer in range(L):
        R = take(M, M, W, W)            # [kx][kz][in][out]
        WT, b = take(W, W), take(W)     # WT[out][in]
        f = v.reshape(B, W, nx, nz) @ Fz.T
        f = torch.einsum("ax,bwxk->bwak", Fx, f)
        f = torch.einsum("akio,biak->boak", R, f)
        f = torch.einsum("ax,boak->boxk", Fx.conj(), f) @ Fz.conj()
        z = f.reshape(B, W, nx * nz) / (nx * nz) + torch.einsum("oi,bin->bon", WT, v) + b[None, :, None]
        v = act(z) if layer < L - 1 else z
    Q, q = take(W), take(1)
    return x[:, 0] + torch.einsum("w,bwn->bn", Q, v) + q


def exact(case, seed):
    kind = case["kind"]
    if kind == "operator":
        return _exact_operator(case, seed)
    if kind == "solve" and case["nz"] * case["nx"] <= 8192:
        return _exact_solve(case, seed)
    if kind == "learned":
        g = _generator(seed)
        dtype = torch.complex128 if case["prec"] == "c128" else torch.complex64
        v = (3.0 * _smooth_fields(g, case["batch"], case["nz"], case["nx"])).to(dtype).to(torch.complex128)
        k = 2 * math.pi * case["freq"] / C0
        x1 = torch.complex(_chi64(case, seed) / (k * k), torch.full((v.shape[1],), k * case["h"], device="cuda",
                                                                    dtype=torch.float64))
        norm = v.norm(dim=1, keepdim=True)
        with torch.no_grad():
            return norm * _exact_network(case, _network(case, seed).to(torch.complex128),
                                         torch.stack([v / norm, x1.expand_as(v)], dim=1))
    if kind == "train":
        x, t = (a.to(torch.complex128) for a in _train_inputs(case, seed))
        p = _network(case, seed).to(torch.complex128).requires_grad_()
        total = 0.0
        for i in range(0, x.shape[0], 4):       # the mean over all samples, four at a time
            d = _exact_network(case, p, x[i:i + 4]) - t[i:i + 4]
            loss = (d.real.square() + d.imag.square()).sum() / t.numel()
            loss.backward()
            total += float(loss)
        grad, w, lr = p.grad, p.detach(), 1e-5
        # Adam's first step on real and imaginary parts
        gr, wr = torch.view_as_real(grad), torch.view_as_real(w)
        new = torch.view_as_complex((wr - lr * gr / (gr.abs() + 1e-8)).contiguous())
        return {"loss": total, "grad": grad, "weights": new}
    # no plain 64-bit counterpart: H itself is the approximation, and the
    # larger systems' direct solutions are out of reach
    return None
