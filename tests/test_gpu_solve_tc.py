"""Complex64 substitution on the tensor cores (groups of 16, 32 and 64 vectors of a
mode): one block (no product), full and half tiles, ragged last groups down to
two vectors, and mode 0 with half the vectors."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W

DEV = "cuda:0"


@pytest.mark.parametrize("panels,nrhs", [(1, 64), (2, 7), (2, 17), (3, 13), (3, 32), (4, 33), (5, 65)])
def test_solution_satisfies_the_system(panels, nrhs):
    """||A'y - b'||_inf <= tol (||A'||_inf ||y||_inf + ||b'||_inf) per vector, modes -M..M:
    the refinement stops at 1e-14 and its residual's rounding adds at most as much
    (tol = 2e-14).  One correction in FP32 precision leaves about n 2^-24 of the
    error (n = 320: 2e-5), so from FP64's 1 the bound is met after three; four are
    allowed."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as mb
    M = 3
    curve, media = W.random_body(panels, seed=panels), W.Media.from_k(1.0, 1.5)
    opts = mb.Options(n_phi=64, precision=1)
    ctx = mb.build(curve, media, M, opts)
    n = 4 * curve.N
    A = torch.zeros((M + 1, n, n), dtype=torch.complex128, device=DEV)
    mb.assemble(curve, media, M, A, opts)
    A = A.cpu().numpy().transpose(0, 2, 1)
    rng = np.random.default_rng(nrhs)
    rhs = rng.standard_normal((2 * M + 1, nrhs, n)) + 1j * rng.standard_normal((2 * M + 1, nrhs, n))
    x = torch.zeros(rhs.shape, dtype=torch.complex128, device=DEV)
    ctx.solve(torch.tensor(rhs, device=DEV), x)
    iters = ctx.stats()["refine_iters"]
    x = x.cpu().numpy()
    ctx.close()
    sp = np.hypot(curve.dr, curve.dz)
    sw = np.repeat(np.sqrt(np.tile(np.polynomial.legendre.leggauss(16)[1], panels) * sp), 4)
    Dr, Dc = np.tile([-1.0, 1, 1, -1], curve.N), np.tile([1.0, -1, -1, 1], curve.N)
    for m in range(-M, M + 1):
        Am = A[abs(m)] if m >= 0 else Dr[:, None] * A[-m] * Dc[None, :]
        y, b = x[m + M].T * sw[:, None], rhs[m + M].T * sw[:, None]
        r = np.abs(Am @ y - b).max(0)
        assert (r <= 2e-14 * (np.abs(Am).sum(1).max() * np.abs(y).max(0) + np.abs(b).max(0))).all(), m
    assert iters <= 4
