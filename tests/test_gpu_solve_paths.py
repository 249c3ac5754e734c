"""Block-step solves at the edges of their shapes: one to five 64-column blocks
(odd and even counts: half tiles), every vector group (4, 8, 16, 32) full and
ragged, both precisions, interchanged rows."""
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


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("panels,nrhs", [(1, 1), (1, 17), (2, 2), (3, 3), (3, 8), (4, 5), (5, 9), (5, 33)])
def test_solution_satisfies_the_system(mb, panels, nrhs, precision):
    """||A'y - b'||_inf <= tol (||A'||_inf ||y||_inf + ||b'||_inf) per vector, modes -M..M,
    with the assembled weighted matrices: complex128 LU and substitution round
    each of n products a few times, growth below 8 here: tol = 64 n 2^-53; the
    mixed paths stop at 1e-14 (their residual's own rounding on top: 2e-14)."""
    M = 3
    curve, media = W.random_body(panels, seed=panels), W.Media.from_k(1.0, 1.5)
    opts = mb.Options(n_phi=64, precision=precision)
    ctx = mb.build(curve, media, M, opts)
    n = 4 * curve.N
    A = torch.zeros((M + 1, n, n), dtype=torch.complex128, device=DEV)
    mb.assemble(curve, media, M, A, opts)
    A = A.cpu().numpy().transpose(0, 2, 1)
    rng = np.random.default_rng(nrhs)
    rhs = rng.standard_normal((2 * M + 1, nrhs, n)) + 1j * rng.standard_normal((2 * M + 1, nrhs, n))
    x = torch.zeros(rhs.shape, dtype=torch.complex128, device=DEV)
    ctx.solve(torch.tensor(rhs, device=DEV), x)
    x = x.cpu().numpy()
    ctx.close()
    sp = np.hypot(curve.dr, curve.dz)
    sw = np.repeat(np.sqrt(np.tile(np.polynomial.legendre.leggauss(16)[1], panels) * sp), 4)
    Dr, Dc = np.tile([-1.0, 1, 1, -1], curve.N), np.tile([1.0, -1, -1, 1], curve.N)
    tol = 64 * n * 2.0 ** -53 if precision == 0 else 2e-14
    for m in range(-M, M + 1):
        Am = A[abs(m)] if m >= 0 else Dr[:, None] * A[-m] * Dc[None, :]
        y, b = x[m + M].T * sw[:, None], rhs[m + M].T * sw[:, None]
        r = np.abs(Am @ y - b).max(0)
        assert (r <= tol * (np.abs(Am).sum(1).max() * np.abs(y).max(0) + np.abs(b).max(0))).all(), m
