"""lsw_solve_batched with seven problems at a time, again and again: workers capture
solver steps as graphs while others release preconditioners and Green handles, calls
that wait for the whole device and fail during a capture.  Every call succeeds, and
every solution is the one the problem has alone."""
import numpy as np
import pytest

from paper_2005_01372_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_many_problems_at_a_time():
    from paper_2005_01372_gb300 import lsw
    problems = []
    for i in range(28):
        n = (32, 64, 32, 16)[i % 4]
        c = media.random_field(np.random.default_rng(i), n, n)
        problems.append(dict(nz=n, nx=n, h=10.0, c0=media.C0, freq_hz=4.0 + 0.25 * i,
                             velocity=torch.from_numpy(c.ravel().copy()).cuda(), sources=[(0, 1 + 2 * s) for s in range(3)]))
    hp = lsw.HParams(kind=lsw.H_HODLR, prec=lsw.C64, levels=2, rank=8, oversample=4, seed=3)
    sp = lsw.SolveParams(prec=lsw.MIXED, method=lsw.FGMRES, tol=1e-8, max_iter=60, restart=30, max_outer=12)
    want, infos = lsw.solve_batched(problems, hp, sp, 1)
    assert all(i.status == 0 for per in infos for i in per)
    for _ in range(12):
        got, infos = lsw.solve_batched(problems, hp, sp, 7)
        assert all(i.status == 0 for per in infos for i in per)
        for a, b in zip(got, want):
            assert torch.equal(a, b)
