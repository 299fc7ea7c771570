"""complex128 operators on few fields: the rule by which the passes start early, on
both sides of its lines (a field alone and the same field among others, bit for bit),
and that few fields do not wait for each other on part of the GPU: a quarter of the
fields takes less than half the time (0.3 of it; two thirds when early starts
crowded them)."""
import numpy as np
import pytest

from paper_2005_01372_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def setup(nz, nx, nb):
    from paper_2005_01372_gb300 import lsw
    rng = np.random.default_rng(nz + nb)
    G = lsw.build_green(nz, nx, 10.0, media.C0, 9.0)
    chi = G.contrast(torch.from_numpy(media.random_field(rng, nz, nx).ravel().copy()).cuda())
    return lsw, G, chi, torch.from_numpy(media.complex_field(rng, (nb, nz * nx))).cuda()


@pytest.mark.parametrize("nz,nx,nb", [(16, 1024, 16), (1024, 16, 31), (512, 32, 32), (256, 64, 31), (64, 256, 16),
                                      (128, 128, 31), (256, 256, 8), (128, 512, 8), (512, 512, 2), (1024, 256, 2), (8, 256, 130)])
def test_alone_equals_among_others(nz, nx, nb):
    lsw, G, chi, u = setup(nz, nx, nb)
    for mode in (lsw.OP_RESIDUAL, lsw.OP_ADJOINT):
        y = lsw.apply_operator(G, chi, u, u, mode)
        for k in (1, nb // 2 + 1):
            part = lsw.apply_operator(G, chi, u[nb - k:].contiguous(), u[nb - k:].contiguous(), mode)
            assert torch.equal(part, y[nb - k:])


def time_of(lsw, G, chi, u):
    y = torch.empty_like(u)
    best = float("inf")
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(10):
            lsw.apply_operator(G, chi, u, None, lsw.OP_PLAIN, y=y)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("nz,nx,nb", [(128, 128, 32), (1024, 16, 32), (256, 256, 8)])
def test_few_fields_take_their_share(nz, nx, nb):
    lsw, G, chi, u = setup(nz, nx, nb)
    assert time_of(lsw, G, chi, u[:nb // 4].contiguous()) < 0.5 * time_of(lsw, G, chi, u)
