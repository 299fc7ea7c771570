"""FP32 field norms over FP32's whole range: squares of entries around 1e-30 or
1e30 leave FP32 (and are summed in FP32 parts), so a field times a power of two
must have its norm times exactly that power.  The network's apply divides by
the norm and multiplies by it again, which makes it homogeneous of degree one.
Tolerance 1e-6: FP32 rounding of the scaled products (2^-24 each), no more."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(32, 1), (64, 3)])
@pytest.mark.parametrize("power", [-100, -62, 62, 90])
def test_apply_is_homogeneous_over_the_range(n, batch, power):
    from paper_2005_01372_gb300 import lsw, media
    G = lsw.build_green(n, n, 10.0, media.C0, 12.0)
    rng = np.random.default_rng(n + power + 200)
    chi = G.contrast(torch.from_numpy(media.random_field(rng, n, n).ravel().copy()).cuda())
    net = lsw.FNO(n, n, 4, 3, 2, seed=2)
    v = torch.from_numpy(media.complex_field(rng, (batch, n * n)).astype(np.complex64)).cuda()
    v[:, ::5] *= 1e-12                  # entries far below the largest of their group
    z = net.apply(G, chi, v).cpu().numpy().astype(np.complex128)
    zs = net.apply(G, chi, v * 2.0 ** power).cpu().numpy().astype(np.complex128) / 2.0 ** power
    assert np.all(np.isfinite(zs))
    assert np.linalg.norm(zs - z) / np.linalg.norm(z) < 1e-6
