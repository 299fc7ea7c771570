"""The scaling of Krylov vectors in complex64 solves: rounded as the FP64 product,
inside the range of scales where FP32 parts do the work and outside of it.

FGMRES without H is exactly homogeneous under powers of two as long as nothing
underflows: a right-hand side times 2^k has the same Krylov vectors, so its
solution is 2^k times the solution, bit for bit, and its iterations and residuals
are the same.  2^-78 and 2^60 put the first vector's scale (one over a norm) above
1e20 and below 1e-20, where every entry takes the FP64 product; 1 and 2^-20 are
inside.  Equality, no tolerance.  Solves of one step on the large grid compare 3e8
parts of first vectors: roundings off in one of 2^26 would show."""
import numpy as np
import pytest

from paper_2005_01372_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nb,steps,repeats", [(64, 3, 12, 1), (1024, 4, 1, 36)])
def test_solve_is_homogeneous(n, nb, steps, repeats):
    from paper_2005_01372_gb300 import lsw
    G = lsw.build_green(n, n, 10.0, media.C0, 6.0)
    chi = G.contrast(torch.from_numpy(media.random_field(np.random.default_rng(n), n, n).ravel().copy()).cuda())
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    sp = lsw.SolveParams(prec=lsw.C64, method=lsw.FGMRES, tol=1e-12, max_iter=steps, restart=steps)
    for _ in range(repeats):
        u0 = torch.randn((nb, n * n), generator=g, device="cuda", dtype=torch.complex64)
        # no entry so small that its products underflow
        u0 += torch.complex(torch.sign(u0.real), torch.sign(u0.imag)) * 1e-3
        got = {}
        for k in (0, -20, -78, 60):
            u, infos = lsw.solve_series(G, chi, None, u0 * 2.0 ** k, sp=sp)
            got[k] = (u, [(i.iterations, i.status, i.rel_residual) for i in infos])
        ref, info = got[0]
        assert torch.isfinite(torch.view_as_real(ref)).all() and all(i[0] == steps for i in info)
        for k in (-20, -78, 60):
            assert got[k][1] == info, k
            assert torch.equal(got[k][0] * 2.0 ** -k, ref), k
