"""The network's fused passes at the edges of their dispatch, against the FP64
oracle: register transforms (2m = 8, 16, 32 and sides of 2m times a power of
two up to 2m) with one column, many columns or no whole column per tile, the
dense transforms, channel counts that fill no group of eight, take 512 threads
or the largest size, and fields of an odd number of cells.

Tolerance 1e-4 per tensor, as for the other FP32 network checks: sums of at
most n products rounded at 2^-24 each."""
import numpy as np
import pytest

import test_gpu_fno as base
from oracle import fno as ofno

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
lsw = base.lsw

# nz, nx, W, m, L, batch
SHAPES = [(64, 64, 16, 8, 2, 3), (64, 8, 5, 4, 2, 2), (256, 32, 33, 16, 1, 1), (1024, 32, 3, 16, 1, 1),
          (512, 32, 20, 16, 2, 1), (128, 32, 9, 4, 2, 1), (33, 47, 7, 5, 2, 3), (32, 32, 64, 4, 2, 2),
          (32, 64, 1, 16, 2, 5)]


@pytest.mark.parametrize("nz,nx,W,m,L,B", SHAPES)
def test_passes_match_oracle(lsw, nz, nx, W, m, L, B):
    params, net = base._net(lsw, nz, nx, W, m, L, seed=2 * nz + W)
    xs, ts, xg, tg = base._inputs(nz, nx, B, seed=13)
    y = net.forward(xg).cpu().numpy()
    loss, g = net.loss_grad(xg, tg, want_grad=True)
    ref_loss, ref = 0.0, {}
    for b in range(B):
        x64 = xs[b].astype(np.complex64).astype(np.complex128)
        t64 = ts[b].astype(np.complex64).astype(np.complex128)
        assert base._rel(base.from_flat(y[b], nz, nx), ofno.forward(params, x64, nz, nx, m)) < 1e-4
        lb, gb = ofno.loss_and_grad(params, x64, t64, nz, nx, m)
        ref_loss += lb / B
        for k, v in gb.items():
            ref[k] = ref.get(k, 0.0) + v / B
    assert loss == pytest.approx(ref_loss, rel=1e-4)
    got = base._unflat_grads(g.cpu().numpy().astype(np.complex128), params, L)
    for k, v in ref.items():
        assert base._rel(got[k], v) < 1e-4, k
