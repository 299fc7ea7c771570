"""The network's apply on complex128 vectors is fixed to its last digit: its
arithmetic is FP32, but results leave as complex128 and are compared as such.
The golden file holds 48 entries per case, taken from the library when this
type's order of operations was fixed.  Cases: register-transform sizes, one
whose first transform splits its inner dimension, mode counts and channel
counts of the dense products, more vectors than a tile is wide.

Tolerance 1e-9, what complex128 results are held to elsewhere; one FP32 rounding
that falls the other way shows as 1e-8 or more."""
import os

import numpy as np
import pytest

from paper_2005_01372_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fno_apply_c128.txt")
# nz, nx, width, modes, layers, vectors
CASES = [(64, 64, 16, 8, 3, 2), (256, 64, 4, 4, 2, 1), (32, 64, 9, 5, 5, 3), (64, 32, 35, 16, 2, 2), (32, 32, 5, 4, 1, 70)]


def sampled(nz, nx, W, m, L, B):
    from paper_2005_01372_gb300 import lsw
    rng = np.random.default_rng(nz + 10 * W)
    G = lsw.build_green(nz, nx, 10.0, media.C0, 15.0)
    chi = G.contrast(torch.from_numpy(media.random_field(rng, nz, nx).ravel().copy()).cuda())
    net = lsw.FNO(nz, nx, W, m, L, seed=3)
    w = net.get().cpu().numpy()
    w += (0.01 * (rng.standard_normal(w.size) + 1j * rng.standard_normal(w.size))).astype(np.complex64)
    net.set(torch.from_numpy(w).cuda())
    v = 3.0 * (rng.standard_normal((B, nz * nx)) + 1j * rng.standard_normal((B, nz * nx)))
    z = net.apply(G, chi, torch.from_numpy(v).cuda()).cpu().numpy().ravel()
    return z[np.linspace(0, z.size - 1, 48).astype(np.int64)]


@pytest.mark.parametrize("row", range(len(CASES)))
def test_apply_repeats_to_the_last_digit(row):
    with open(GOLDEN) as f:
        lines = [line.split() for line in f if not line.startswith("#")]
    ref = np.array([complex(float(r), float(i)) for k, r, i in lines if int(k) == row])
    z = sampled(*CASES[row])
    assert ref.size == z.size
    assert np.linalg.norm(z - ref) <= 1e-9 * np.linalg.norm(ref)
