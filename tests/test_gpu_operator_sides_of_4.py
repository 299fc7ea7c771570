"""The operator on boxes of four cells along an axis, the shortest register
transforms: one launch and three passes, both precisions, against the FP64 oracle.

Tolerances (relative 2-norm) as for the other line lengths: 1e-10 in FP64, 1e-5 in
FP32."""
import numpy as np
import pytest

from oracle import operator as oop
from paper_2005_01372_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("nz,nx,nb", [(4, 4, 1), (4, 4, 37), (4, 64, 3), (64, 4, 2), (4, 128, 70), (128, 4, 1), (4, 256, 5),
                                      (512, 4, 3), (4, 1024, 2), (1024, 4, 9), (4, 2, 3), (2, 4, 2), (4, 4, 2100)])
def test_against_oracle(nz, nx, nb, prec):
    from paper_2005_01372_gb300 import lsw
    rng = np.random.default_rng(nz + 5 * nx)
    P = oop.Problem(nz, nx, 10.0, media.C0, 15.0, media.random_field(rng, nz, nx))
    G = lsw.build_green(nz, nx, P.h, P.c0, P.freq_hz)
    chi = torch.from_numpy(P.chi).cuda()
    dt = torch.complex128 if prec == "c128" else torch.complex64
    u = torch.from_numpy(media.complex_field(rng, (nb, P.n))).to(dt)
    u0 = torch.from_numpy(media.complex_field(rng, (nb, P.n))).to(dt)
    un, u0n = (v.numpy().astype(np.complex128).T for v in (u, u0))
    for mode in (lsw.OP_FORWARD, lsw.OP_RESIDUAL, lsw.OP_PLAIN, lsw.OP_ADJOINT):
        y = lsw.apply_operator(G, chi, u.cuda(), u0.cuda(), mode).cpu().numpy()
        ref = oop.apply(mode, P.spec, P.chi, un, u0n, nz, nx).T
        assert np.linalg.norm(y - ref) <= (1e-10 if prec == "c128" else 1e-5) * np.linalg.norm(ref), mode
