"""The batched Gauss-Jordan inverses of H's leaves by leaf size: up to 160
rows in shared memory; beyond, one or more
strips of 64 columns, panels by blocks of 256, 512 and 1024 threads.

The contrast is confined to one leaf's cells.  The blocks that couple into that
leaf are then exactly zero, so H restricted to it is the inverse of the leaf's
own matrix, whatever the sketches of the others; strong contrasts make the
pivots leave the diagonal.  Tolerance: 1e-10 in FP64 and max(1e-5,
16 kappa 2^-24) in FP32, the bounds for an inverse of condition number kappa."""
import numpy as np
import pytest

from oracle import operator as oop
from paper_2005_01372_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lsw():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_01372_gb300 import lsw as L
    L.lib()
    return L


@pytest.mark.parametrize("nz,nx", [(4, 8), (8, 8), (8, 16), (16, 16), (8, 32), (16, 32), (32, 32), (32, 64)])
@pytest.mark.parametrize("prec", ["C128", "C64"])
def test_leaf_sizes(lsw, nz, nx, prec):
    rng = np.random.default_rng(nz + nx)
    c = np.full((nx, nz), 2000.0)
    c[: nx // 2] = rng.uniform(700.0, 3000.0, (nx // 2, nz))
    P = oop.Problem(nz, nx, 10.0, 2000.0, 25.0, c)
    G = lsw.build_green(nz, nx, P.h, P.c0, P.freq_hz)
    chi = torch.from_numpy(P.chi.copy()).cuda()
    H = lsw.build_hmatrix(G, chi, lsw.HParams(kind=lsw.H_HODLR, prec=getattr(lsw, prec), levels=1, rank=8,
                                              oversample=4, seed=31))
    n = P.n // 2
    D = P.dense_A()[:n, :n]
    x = media.complex_field(rng, (3, P.n))
    if prec == "C64":
        x = x.astype(np.complex64)
    y = lsw.apply_precond(H, torch.from_numpy(x).cuda()).cpu().numpy()[:, :n]
    want = np.linalg.solve(D, x[:, :n].T.astype(np.complex128)).T
    tol = 1e-10 if prec == "C128" else max(1e-5, 16.0 * 2.0 ** -24 * np.linalg.cond(D))
    assert np.linalg.norm(y - want) <= tol * np.linalg.norm(want)
