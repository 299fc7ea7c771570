"""Products with H by few vectors: every count of vectors that has a kernel
form of its own, at ranks and block sizes on either side of the kernels'
limits, against the same H applied to 40 vectors in one call.

The products are sums without solves, so two orders of summation in a
precision of unit roundoff u differ by about sqrt(n) u of the terms' size: with
n <= 32768 and terms a few times the result, 1e-5 in FP32 and 1e-12 in FP64.
On BF16 storage both orders read the same stored values, and the vectors enter
as BF16 pairs hi + lo (2^-17 each): 5e-5."""
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


@pytest.mark.parametrize("prec", ["C128", "C64", "BF16"])
@pytest.mark.parametrize("nz,nx,L,rank", [(32, 32, 2, 4), (64, 64, 2, 9), (64, 64, 5, 8), (64, 128, 3, 16),
                                          (128, 128, 7, 17), (128, 128, 6, 20), (256, 128, 7, 40)])
def test_few_vectors_equal_many(lsw, nz, nx, L, rank, prec):
    rng = np.random.default_rng(nz + nx + L + rank)
    P = oop.Problem(nz, nx, 10.0, media.C0, 8.0, media.random_field(rng, nz, nx))
    G = lsw.build_green(nz, nx, P.h, P.c0, P.freq_hz)
    chi = torch.from_numpy(P.chi.copy()).cuda()
    H = lsw.build_hmatrix(G, chi, lsw.HParams(kind=lsw.H_HODLR, prec=getattr(lsw, prec), levels=L, rank=rank,
                                              oversample=4, seed=5))
    x = torch.from_numpy(media.complex_field(rng, (40, P.n))).cuda()
    x = x if prec == "C128" else x.to(torch.complex64)
    y = torch.empty_like(x)
    lsw.apply_precond(H, x, y)
    tol = {"C128": 1e-12, "C64": 1e-5, "BF16": 5e-5}[prec]
    for k in (1, 2, 3, 4, 5, 7, 8, 9, 16, 17, 32):
        z = torch.empty_like(x[:k])
        lsw.apply_precond(H, x[:k].contiguous(), z)
        d = (z - y[:k]).abs().pow(2).sum(1).sqrt() / y[:k].abs().pow(2).sum(1).sqrt()
        assert float(d.max()) <= tol, (k, float(d.max()))
