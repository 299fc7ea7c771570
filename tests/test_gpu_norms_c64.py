"""Norms of complex64 fields to FP64's accuracy, read off a solver's decisions.

A series solve of no steps without H reports convergence exactly if
||a|| / ||u0|| <= tol, a = u0 - G0 V u0 - u0 in complex64; bisecting tol over the
doubles gives the ratio the library formed.  It is compared with the exact sums
(math.fsum of exact squares in FP64) of the same a and u0.

Tolerance: every addition on the way of a term rounds at 2^-53: two per group of
eight entries and group of a thread, 5 + 8 across a block's lanes and warps, one
per chunk of 4096 entries (and one for each squared norm's last rounding); half
of both norms' sum for the square roots of the ratio, one more for the division,
one for the root and one for fsum's."""
import math

import numpy as np
import pytest

from paper_2005_01372_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# 16 parts of one group of eight entries whose rounding errors, summed in FP32
# alone, are 8e-14 of the sum of squares
CANCELLING = """0x1.6fb5c8p+0 0x1.e81ed2p+0 0x1.22e724p-1 0x1.8029e8p+0 0x1.052b92p+0 0x1.0b5bd8p-1 0x1.366d48p+0
0x1.3c61aep+0 0x1.48bd06p+0 0x1.556c8ep+0 0x1.1247dep-1 0x1.2934b4p-1 0x1.1a5a64p-1 0x1.062b5cp-1 0x1.0561dcp-1
0x1.014c42p-1""".split()


def squares(x):
    x = x.view(np.float32).astype(np.float64)       # squares of FP32 numbers are exact in FP64
    return math.fsum(x * x)


def field(kind, rng, n):
    u = (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)
    if kind == "one group":
        u[:] = 0
        u[5:5 + 8 * 256:256] = np.array([float.fromhex(h) for h in CANCELLING], np.float32).view(np.complex64)
    elif kind == "far apart":
        u[::3] *= np.float32(1e-9)
        u[1::7] *= np.float32(3e4)
    elif kind == "tiny":
        u *= np.float32(1e-25)
    elif kind == "large":
        u *= np.float32(1e25)
    return u


@pytest.mark.parametrize("nz,nx,kind", [(64, 64, "one group"), (8, 8, "far apart"), (32, 64, "far apart"), (64, 32, "tiny"),
                                        (64, 256, "large"), (128, 128, "far apart")])
def test_norm_ratio(nz, nx, kind):
    from paper_2005_01372_gb300 import lsw
    n = nz * nx
    rng = np.random.default_rng(nx)
    G = lsw.build_green(nz, nx, 10.0, media.C0, 8.0)
    chi = G.contrast(torch.from_numpy(media.random_field(rng, nz, nx).ravel().copy()).cuda())
    u0 = torch.from_numpy(field(kind, rng, n)).cuda()[None]
    a = lsw.apply_operator(G, chi, u0, u0, lsw.OP_RESIDUAL)
    want = math.sqrt(squares(a.cpu().numpy().ravel()) / squares(u0.cpu().numpy().ravel()))

    def within(tol):
        sp = lsw.SolveParams(prec=lsw.C64, method=lsw.SERIES, tol=tol, max_iter=0)
        return lsw.solve_series(G, chi, None, u0, sp=sp)[1][0].status == 0

    lo, hi = want * (1 - 1e-6), want * (1 + 1e-6)
    assert within(hi) and not within(lo)
    while np.nextafter(lo, hi) < hi:
        mid = 0.5 * (lo + hi)
        mid = np.nextafter(lo, hi) if not lo < mid < hi else mid
        lo, hi = (lo, mid) if within(mid) else (mid, hi)
    groups, chunks = -(-min(n, 4096) // 2048), -(-n // 4096)
    each = 2 * groups + 13 + chunks + 1
    first = 6 if kind == "one group" else each      # sums with zeros do not round
    assert abs(hi / want - 1) <= (0.5 * (each + first) + 3) * 2.0 ** -53
