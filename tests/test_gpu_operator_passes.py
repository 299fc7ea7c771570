"""The operator's register-FFT passes over their line lengths (8 to 1024 on
either axis, both precisions), and the one-launch form for small fields.

Tolerances (relative 2-norm against the FP64 oracle): 1e-10 for the FP64 path,
1e-5 for the FP32 path."""
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


def _setup(lsw, nz, nx, nb, prec, seed):
    rng = np.random.default_rng(seed)
    P = oop.Problem(nz, nx, 10.0, media.C0, 15.0, media.random_field(rng, nz, nx))
    G = lsw.build_green(nz, nx, P.h, P.c0, P.freq_hz)
    dt = torch.complex128 if prec == "c128" else torch.complex64
    u = torch.from_numpy(media.complex_field(rng, (nb, P.n))).to(dt)
    u0 = torch.from_numpy(media.complex_field(rng, (nb, P.n))).to(dt)
    return P, G, torch.from_numpy(P.chi).cuda(), u, u0


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("nz,nx,nb", [
    (8, 8, 1), (8, 16, 5), (16, 8, 3), (32, 32, 1), (8, 256, 2), (256, 8, 2), (128, 256, 1), (256, 128, 1),
    (64, 128, 3), (256, 64, 3), (8, 512, 2), (512, 8, 2), (16, 1024, 1), (1024, 16, 1), (32, 1024, 2), (512, 32, 9)])
def test_line_lengths(lsw, nz, nx, nb, prec):
    P, G, chi, u, u0 = _setup(lsw, nz, nx, nb, prec, 31 * nz + nx)
    un, u0n = (v.numpy().astype(np.complex128).T for v in (u, u0))
    for mode in (lsw.OP_FORWARD, lsw.OP_RESIDUAL, lsw.OP_PLAIN, lsw.OP_ADJOINT):
        y = lsw.apply_operator(G, chi, u.cuda(), u0.cuda(), mode).cpu().numpy()
        ref = oop.apply(mode, P.spec, P.chi, un, u0n, nz, nx).T
        assert np.linalg.norm(y - ref) <= (1e-10 if prec == "c128" else 1e-5) * np.linalg.norm(ref), mode


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("nz,nx,nb", [(8, 8, 600), (32, 16, 70), (64, 64, 40), (128, 32, 33), (128, 256, 3),
                                      (256, 256, 9)])
def test_field_alone_equals_field_in_batch(lsw, nz, nx, nb, prec):
    """A field's result does not depend on how many fields the call has, on
    either side of the sizes that take one launch."""
    P, G, chi, u, u0 = _setup(lsw, nz, nx, nb, prec, nz + nx + nb)
    u, u0 = u.cuda(), u0.cuda()
    for mode in (lsw.OP_RESIDUAL, lsw.OP_ADJOINT):
        y = lsw.apply_operator(G, chi, u, u0, mode)
        for b in (0, nb // 2, nb - 1):
            one = lsw.apply_operator(G, chi, u[b:b + 1].contiguous(), u0[b:b + 1].contiguous(), mode)
            assert torch.equal(one, y[b:b + 1])
