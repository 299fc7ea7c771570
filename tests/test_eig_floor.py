"""What the truncation's eigenvectors lose where a pivot of the Gram matrix's
factorisation is floored (small64.cu): a NumPy model of the sorted, floored
square-root-free Cholesky factorisation.  With p floored pivots, v^H G v is at most
(p + 1) v^H G' v for the matrix G' that is factored, so the weight of G outside the
leading r eigenvectors of G' is at most (p + 1) times that of G'.  Columns nearly equal
to earlier ones come ahead of independent columns of the same norm, the order in which
the dropped entries are largest.  Allowance: 1e-13 for the rounding of FP64 sums of
trace 1 (64 terms, some hundred operations)."""
import numpy as np
import pytest

TINY = 1e-15


def floored_factor(G):
    """W with W W^H = G' for G scaled to trace 1, and the number of floored pivots."""
    k = G.shape[0]
    key = np.floor(np.log2(np.maximum(np.diag(G).real, 1e-300)) / 10)
    order = np.argsort(-key, kind="stable")
    A = G[np.ix_(order, order)].copy()
    W, floored = np.zeros_like(A), 0
    for j in range(k):
        d = A[j, j].real
        if d > TINY:
            W[j:, j] = A[j:, j] / np.sqrt(d)
            A[j + 1:, j + 1:] -= np.outer(A[j + 1:, j], A[j + 1:, j].conj()) / d
        else:
            W[j, j] = np.sqrt(TINY)
            floored += 1
    out = np.empty_like(W)
    out[order] = W
    return out, floored


@pytest.mark.parametrize("k,dup,eps", [(3, 1, 1e-9), (12, 4, 1e-8), (30, 10, 1e-9), (30, 14, 1e-12), (50, 20, 3e-8)])
def test_floored_pivots_keep_the_weights(k, dup, eps):
    rng = np.random.default_rng(k + dup)
    Y = rng.standard_normal((400, k)) + 1j * rng.standard_normal((400, k))
    Y /= np.linalg.norm(Y, axis=0)
    for j in range(1, dup + 1):         # near copies of the first column, pointing into later ones
        Y[:, j] = Y[:, 0] + eps * Y[:, dup + 1 + j % (k - dup - 1)]
        Y[:, j] /= np.linalg.norm(Y[:, j])
    G = Y.conj().T @ Y
    G /= np.trace(G).real
    W, p = floored_factor(G)
    assert p >= 1
    Gp = W @ W.conj().T
    low = np.linalg.eigvalsh((p + 1) * Gp - G)
    assert low[0] >= -1e-13
    lam, V = np.linalg.eigh(Gp)
    for r in (1, k // 3, k - dup - 1, k - 1):
        out = V[:, :k - r]
        assert np.trace(out.conj().T @ G @ out).real <= (p + 1) * lam[:k - r].sum() + 1e-13
    # the kept part is a best one to FP32's accuracy: G's own leading weights
    r = k - dup
    assert lam[::-1][:r].sum() == pytest.approx(np.linalg.eigvalsh(G)[::-1][:r].sum(), abs=3e-8)
