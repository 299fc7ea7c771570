"""Rounding of the complex64 operator: its distance to the FP64 operator on the same
fields is no larger than that of radix-8 passes with products by (cos, sin), the
library's first register passes, measured on these inputs (FORMER, relative
2-norms).  Inputs are fixed and the kernels are deterministic, so no tolerance."""
import numpy as np
import pytest

from paper_2005_01372_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FORMER = {
    (8, 8): (1.18496e-07, 1.18627e-07), (8, 64): (1.33987e-07, 1.35327e-07),
    (16, 16): (1.41662e-07, 1.43472e-07), (16, 64): (1.50518e-07, 1.50329e-07),
    (16, 1024): (1.66099e-07, 1.68970e-07), (32, 32): (1.41675e-07, 1.43136e-07),
    (32, 128): (1.66186e-07, 1.63995e-07), (64, 64): (1.71547e-07, 1.72232e-07),
    (64, 16): (1.45837e-07, 1.45401e-07), (128, 32): (1.59828e-07, 1.61131e-07),
    (128, 128): (1.78347e-07, 1.80313e-07), (128, 256): (1.89810e-07, 1.85761e-07),
    (256, 16): (1.52244e-07, 1.52998e-07), (256, 256): (1.96934e-07, 1.91962e-07),
    (256, 1024): (2.00570e-07, 2.04874e-07), (512, 64): (1.84434e-07, 1.83211e-07),
    (512, 512): (2.08549e-07, 2.10502e-07), (1024, 16): (1.63286e-07, 1.63673e-07),
    (1024, 128): (1.97667e-07, 1.91393e-07), (1024, 1024): (2.20423e-07, 2.13889e-07),
}


def errors(nz, nx):
    """The distances of PLAIN and ADJOINT on about 2^20 cells of noise."""
    from paper_2005_01372_gb300 import lsw
    G = lsw.build_green(nz, nx, 10.0, media.C0, 9.0)
    rng = np.random.default_rng(nz + 3 * nx)
    chi = G.contrast(torch.from_numpy(media.random_field(rng, nz, nx).ravel().copy()).cuda())
    nb = max(1, min(512, (1 << 20) // (nz * nx)))
    u = (rng.standard_normal((nb, nz * nx)) + 1j * rng.standard_normal((nb, nz * nx))).astype(np.complex64)
    u = torch.from_numpy(u).cuda()
    out = []
    for mode in (lsw.OP_PLAIN, lsw.OP_ADJOINT):
        ref = lsw.apply_operator(G, chi, u.to(torch.complex128), None, mode)
        y = lsw.apply_operator(G, chi, u, None, mode)
        out.append(float((y.to(torch.complex128) - ref).norm() / ref.norm()))
    return out


@pytest.mark.parametrize("size", sorted(FORMER))
def test_no_larger_than_before(size):
    for got, former in zip(errors(*size), FORMER[size]):
        assert got <= former
