"""The first residual of a solve that starts from zero fields (formed from one
field for several sources): a contrast that is not finite is reported before
any iteration, as by the full residual, and finite ones converge."""
import numpy as np
import pytest

from paper_2005_01372_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [1, 3])
@pytest.mark.parametrize("prec", ["C128", "C64", "MIXED"])
@pytest.mark.parametrize("bad", [None, float("nan"), float("inf")])
def test_first_residual(nb, prec, bad):
    from paper_2005_01372_gb300 import lsw
    n = 32
    c = media.random_field(np.random.default_rng(4), n, n)
    G = lsw.build_green(n, n, 10.0, media.C0, 5.0)
    chi = G.contrast(torch.from_numpy(np.ascontiguousarray(c.ravel())).cuda())
    if bad is not None:
        chi[n * n // 3] = bad
    u0 = G.point_sources([(0, 4 + 9 * s) for s in range(nb)], lsw.C64 if prec == "C64" else lsw.C128)
    tol = 1e-4 if prec == "C64" else 1e-9
    sp = lsw.SolveParams(prec=getattr(lsw, prec), tol=tol, method=lsw.FGMRES, max_iter=200)
    u, infos = lsw.solve_series(G, chi, None, u0, sp=sp)
    for i in infos:
        if bad is None:
            assert i.status == 0 and i.rel_residual <= 2 * tol
        else:
            assert i.status == 7 and i.iterations == 0
