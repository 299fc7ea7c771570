"""Products with BF16 leaves on the CUDA cores (tensor cores switched off) against
the tensor-core products of the same H: leaves stored column by column (64) and as
operand tiles (128 and more), one vector, a few, and more than a block of 32.  Both
read the same stored values, and the tensor cores take a vector as BF16 parts hi + lo
(2^-17 each): 5e-5, as for the other products of this storage.  The steps the kernel
takes through a row of tiles are checked against fac_index on the host."""
import os
import subprocess

import numpy as np
import pytest

import test_fac_layout as layout
from paper_2005_01372_gb300 import media

PROGRAM = r"""
#include <cstdio>
#include "lsw_internal.cuh"
using namespace lsw;
int main() {
    for (int nL : {128, 256, 1024})
        for (int b = 0; b < 3; ++b)
            for (int i = 0; i < nL; ++i) {
                const long long d = fac_index(FAC_TILE_A, nL, nL, nL, b, i, 0);
                if (d % 4) return 1;            // 16-byte loads
                for (int t = 0; t < nL; ++t)
                    if (fac_index(FAC_TILE_A, nL, nL, nL, b, i, t) != d + t / 8 * 1024 + t % 8 / 4 * 32 + t % 4) return 2;
            }
    return 0;
}
"""


def test_steps_through_a_row(tmp_path):
    nvcc = layout._nvcc()
    if not nvcc:
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "steps.cu", tmp_path / "steps"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", os.path.join(layout.ROOT, "include"),
                        "-I", os.path.join(layout.ROOT, "paper_2005_01372_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    assert subprocess.run([str(exe)]).returncode == 0


@pytest.mark.gpu
@pytest.mark.parametrize("nz,nx,L", [(64, 64, 6), (64, 64, 5), (64, 128, 5), (128, 64, 3)])
def test_cuda_cores_equal_tensor_cores(nz, nx, L):
    torch = pytest.importorskip("torch")
    from paper_2005_01372_gb300 import lsw
    rng = np.random.default_rng(nz + L)
    G = lsw.build_green(nz, nx, 10.0, media.C0, 5.0)
    chi = G.contrast(torch.from_numpy(media.random_field(rng, nz, nx).ravel().copy()).cuda())
    H = lsw.build_hmatrix(G, chi, lsw.HParams(kind=lsw.H_HODLR, prec=lsw.BF16, levels=L, rank=12, oversample=4, seed=5))
    for k in (1, 6, 35):
        x = torch.from_numpy(media.complex_field(rng, (k, nz * nx)).astype(np.complex64)).cuda()
        on, off = torch.empty_like(x), torch.empty_like(x)
        lsw.apply_precond(H, x, on)
        lsw.set_tensor_cores(False)
        try:
            lsw.apply_precond(H, x, off)
        finally:
            lsw.set_tensor_cores(True)
        d = (on - off).abs().pow(2).sum(1).sqrt() / on.abs().pow(2).sum(1).sqrt()
        assert float(d.max()) <= 5e-5, k
