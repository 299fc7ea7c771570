"""The eigenvectors that truncate complex64 sketches (one-sided Jacobi on the
FP64 Cholesky factor), through whole sketches: probe counts at the edges of the
kernel's variants (1, odd, 32, 33, 64 columns), blocks of lower rank than the
probes (floored pivots), and the complex128 sketch of the same probes as the
reference.  Tolerance 1e-5, the library's bound for complex64 sketches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _products(lsw, G, chi, rows, cols, rank, over, prec):
    U, W = lsw.sketch_range(G, chi, rows, cols, rank, over, 0, 77, stream_id=3, prec=prec)
    U, W = U.to(torch.complex128), W.to(torch.complex128)
    return (U.T @ W.conj()).cpu().numpy()


@pytest.mark.parametrize("rank,over", [(1, 0), (2, 1), (7, 2), (20, 12), (20, 13), (33, 0), (40, 23), (60, 4)])
@pytest.mark.parametrize("medium", ["random", "rank7"])
def test_truncation_matches_fp64(rank, over, medium):
    from paper_2005_01372_gb300 import lsw, media
    n = 32
    rng = np.random.default_rng(rank + 100 * over)
    c = media.random_field(rng, n, n)
    if medium == "rank7":               # chi on seven cells of the columns' box
        c = np.full((n, n), 2000.0)
        c.ravel()[512 + rng.choice(512, size=7, replace=False)] = rng.uniform(1500, 4500, size=7)
    G = lsw.build_green(n, n, 10.0, media.C0, 15.0)
    chi = G.contrast(torch.from_numpy(c.ravel().copy()).cuda())
    rows, cols = (0, n, 0, n // 2), (0, n, n // 2, n)
    got = _products(lsw, G, chi, rows, cols, rank, over, lsw.C64)
    want = _products(lsw, G, chi, rows, cols, rank, over, lsw.C128)
    assert np.all(np.isfinite(got))
    assert np.linalg.norm(got - want) / np.linalg.norm(want) < 1e-5
