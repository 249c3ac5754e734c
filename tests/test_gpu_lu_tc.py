"""Complex128 LU with tensor-core products: sizes at the edges of panels, blocks
and tiles, graded rows, non-finite entries, several matrices."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def mb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as m
    return m


def _lu(mb, A):
    """A [batch, n, n] (math layout) -> L U packed, pivots, info."""
    B, n = A.shape[:2]
    F = torch.tensor(np.ascontiguousarray(A.transpose(0, 2, 1)), device=DEV)
    piv = torch.zeros((B, n), dtype=torch.int32, device=DEV)
    info = torch.zeros(B, dtype=torch.int32, device=DEV)
    mb.lu_batched(F, piv, info)
    return F.cpu().numpy().transpose(0, 2, 1), piv.cpu().numpy(), info.cpu().numpy()


def _matrix(rng, n, grade):
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return A * 10.0 ** (grade * rng.uniform(-1, 1, n))[:, None]


@pytest.mark.parametrize("n", [31, 33, 64, 97, 128, 129, 160, 161, 255, 257, 289, 385])
@pytest.mark.parametrize("grade", [0, 11])
def test_factors_reproduce_rows(mb, n, grade):
    """P A = L U entry by entry, rows spread over 22 orders for grade 11.  With
    d_k the largest entry of row k of U, every product of the factorization is
    at most rmax_i cmax_j, rmax_i = max_k |l_ik| d_k, cmax_j = max_k |u_kj| / d_k;
    n of them, each rounded or sliced to 2^-53 of that bound a few times
    (slicing and joining 2^-55, product and sum 2^-53, the block row's inverse):
    |P A - L U| <= 8 n 2^-53 rmax_i cmax_j."""
    rng = np.random.default_rng(n + grade)
    A = np.stack([_matrix(rng, n, grade) for _ in range(2)])
    F, piv, info = _lu(mb, A)
    assert not info.any()
    for b in range(2):
        P = np.arange(n)
        for k, p in enumerate(piv[b]):
            assert k <= p < n
            P[[k, p]] = P[[p, k]]
        L, U = np.tril(F[b], -1) + np.eye(n), np.triu(F[b])
        assert np.abs(L).max() <= 1 + 1e-12                       # partial pivoting
        d = np.abs(U).max(1)
        bound = 8 * n * 2.0 ** -53 * (np.abs(L) * d).max(1)[:, None] * (np.abs(U) / d[:, None]).max(0)[None, :]
        R = A[b][P].astype(np.clongdouble) - L.astype(np.clongdouble) @ U.astype(np.clongdouble)
        assert (np.abs(R) <= bound).all(), float((np.abs(R) / bound).max())


def test_non_finite_entries_stay(mb):
    """A NaN or infinity reaches the factors of its matrix and no other."""
    rng = np.random.default_rng(4)
    A = np.stack([_matrix(rng, 300, 0) for _ in range(3)])
    good, gp, _ = _lu(mb, A[1:2])
    A[0, 290, 5] = np.nan
    A[2, 7, 250] = np.inf
    F, piv, _ = _lu(mb, A)
    assert np.array_equal(F[1], good[0]) and np.array_equal(piv[1], gp[0])
    for b in (0, 2):
        assert not np.isfinite(F[b]).all()
        assert not np.isfinite(F[b][-1, -1])
