"""Complex128 LU with less workspace than its matrices want (groups that share one
matrix's) and with none (FP64 pipe), and matrices of several orders in one call."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W

DEV = "cuda:0"


@pytest.fixture(scope="module")
def mb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as m
    return m


@pytest.mark.parametrize("pool", ["", "lu_pool_one", "lu_pool_none"])
@pytest.mark.parametrize("n", [33, 129, 300])
def test_factors_reproduce_the_matrix(mb, monkeypatch, pool, n):
    """P A = L U of five Gaussian matrices: n products an entry, each rounded or sliced a
    few times to 2^-53 of at most max |l| max |u|, |l| <= 1: 8 n 2^-53 max |u|."""
    monkeypatch.setenv("MUELLER_FAULT_INJECT", pool)
    rng = np.random.default_rng(n)
    A = rng.standard_normal((5, n, n)) + 1j * rng.standard_normal((5, n, n))
    F = torch.tensor(np.ascontiguousarray(A.transpose(0, 2, 1)), device=DEV)
    piv = torch.zeros((5, n), dtype=torch.int32, device=DEV)
    info = torch.zeros(5, dtype=torch.int32, device=DEV)
    mb.lu_batched(F, piv, info)
    F, piv = F.cpu().numpy().transpose(0, 2, 1), piv.cpu().numpy()
    assert not info.any()
    for b in range(5):
        P = np.arange(n)
        for k, q in enumerate(piv[b]):
            P[[k, q]] = P[[q, k]]
        L, U = np.tril(F[b], -1) + np.eye(n), np.triu(F[b])
        R = A[b][P].astype(np.clongdouble) - L.astype(np.clongdouble) @ U.astype(np.clongdouble)
        assert float(np.abs(R).max()) <= 8 * n * 2.0 ** -53 * np.abs(U).max()


@pytest.mark.parametrize("pool", ["", "lu_pool_one", "lu_pool_none"])
def test_bodies_of_several_orders(mb, monkeypatch, pool):
    """Orders 64 to 576, whose ends fall inside and between the blocks of 128: the currents
    of bodies factored together and alone satisfy the same systems, whose condition numbers
    are below 1e4: 1e-11 of the largest."""
    bodies = [(W.random_body(p, seed=p), W.Media.from_k(1.0 + 0.1 * p, 1.5), 2 + p) for p in (1, 2, 3, 5, 9)]
    opts = mb.Options(n_phi=64, precision=0)
    w = [W.plane_wave([0.3, 0.4, 1.0], [1.0, 0.0, 0.0])]

    def currents(ctx, M, N):
        rhs = torch.zeros((2 * M + 1, 1, 4 * N), dtype=torch.complex128, device=DEV)
        x = torch.zeros_like(rhs)
        ctx.rhs_planewave([v.d for v in w], [v.e for v in w], rhs)
        ctx.solve(rhs, x)
        ctx.close()
        return x

    alone = [currents(mb.build(c, m, M, opts), M, c.N) for c, m, M in bodies]
    monkeypatch.setenv("MUELLER_FAULT_INJECT", pool)
    for ctx, (c, _, M), x in zip(mb.build_many(bodies, opts), bodies, alone):
        assert float((currents(ctx, M, c.N) - x).abs().max()) <= 1e-11 * float(x.abs().max()), c.N
