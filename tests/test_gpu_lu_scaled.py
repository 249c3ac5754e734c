"""Complex128 LU of matrices whose blocks, rows or columns differ by many orders and couple
weakly or sparsely, where the factors' largest entries do not meet in the products."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _matrix(kind, n, rng):
    def g(*s):
        return rng.standard_normal(s) + 1j * rng.standard_normal(s)

    def scale():
        return 10.0 ** rng.uniform(-8, 8, n)

    def sparse(d):
        return g(n, n) * (rng.random((n, n)) < d) + np.diag(3 * g(n))
    pr, pc = rng.permutation(n), rng.permutation(n)
    if kind == "sparse columns":
        return sparse(0.05) * scale()[None]
    if kind == "sparse rows and columns":
        return sparse(0.05) * scale()[None] * scale()[:, None]
    if kind == "very sparse":
        return sparse(0.01) * scale()[None] * scale()[:, None]
    if kind == "weakly coupled blocks":
        A = 1e-11 * g(n, n)
        for b in range(0, n, 16):
            e = min(n, b + 16)
            A[b:e, b:e] += g(e - b, e - b) * 10.0 ** rng.uniform(-8, 8)
        return A[pr][:, pr]
    A = g(n, n)                                              # upper triangle of blocks, large columns
    A[n // 2:, :n // 2] = 0.0
    A[:, :n // 2] *= 1e8
    return A[pr][:, pc]


@pytest.mark.parametrize("kind", ["sparse columns", "sparse rows and columns", "very sparse", "weakly coupled blocks",
                                  "block upper"])
@pytest.mark.parametrize("n", [97, 200, 290])
def test_residual_by_columns(kind, n):
    """P A - L U relative to each column's largest entry of A or U.  |l| <= 1, so a column takes
    n products of at most that, rounded or sliced to 2^-53 a few times (8 n 2^-53), and at most
    16 updates by digits, each off by 2^-55 of a bound up to 2^8 times it."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as mb
    A = _matrix(kind, n, np.random.default_rng(n))
    F = torch.tensor(np.ascontiguousarray(A.T)[None], device=DEV)
    piv = torch.zeros((1, n), dtype=torch.int32, device=DEV)
    info = torch.zeros(1, dtype=torch.int32, device=DEV)
    mb.lu_batched(F, piv, info)
    F, P = F.cpu().numpy()[0].T, np.arange(n)
    assert not info.any()
    for k, p in enumerate(piv.cpu().numpy()[0]):
        P[[k, p]] = P[[p, k]]
    L, U = np.tril(F, -1) + np.eye(n), np.triu(F)
    R = np.abs(A[P].astype(np.clongdouble) - L.astype(np.clongdouble) @ U.astype(np.clongdouble)).max(0)
    size = np.maximum(np.abs(A).max(0), np.abs(U).max(0))
    assert (R <= (8 * n * 2.0 ** -53 + 16 * 2.0 ** -47) * size).all(), float((R / size).max())
