"""Complex64 substitution in groups of 32 and 64 vectors, which calls with many vectors
over all modes take: full and ragged groups, one block and several."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W

DEV = "cuda:0"


@pytest.mark.parametrize("panels,M,nrhs", [(1, 40, 20), (3, 30, 30), (2, 30, 70), (5, 40, 52)])
def test_solution_satisfies_the_system(panels, M, nrhs):
    """||A'y - b'||_inf <= 2e-14 (||A'||_inf ||y||_inf + ||b'||_inf) per vector: the
    refinement stops at 1e-14 and its residual's rounding adds at most as much."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as mb
    assert 2 * nrhs > 32 and (2 * M + 1) * nrhs > 1600
    curve, media = W.random_body(panels, seed=panels), W.Media.from_k(1.0, 1.5)
    opts = mb.Options(n_phi=128, precision=1)
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
    for m in (0, 1, -1, -7, M, -M):
        Am = A[abs(m)] if m >= 0 else Dr[:, None] * A[-m] * Dc[None, :]
        y, b = x[m + M].T * sw[:, None], rhs[m + M].T * sw[:, None]
        r = np.abs(Am @ y - b).max(0)
        assert (r <= 2e-14 * (np.abs(Am).sum(1).max() * np.abs(y).max(0) + np.abs(b).max(0))).all(), m
