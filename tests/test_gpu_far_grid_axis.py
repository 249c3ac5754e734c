"""Far field on a grid of currents that live near the axis alone, where the nodes' weights
are many orders below the largest."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W

DEV = "cuda:0"


@pytest.mark.parametrize("nodes", [1, 4, 40])
def test_currents_near_the_axis(nodes):
    """One mode a side on the nodes nearest the axis: eight sides together (tensor cores)
    against one at a time (FP64 pipe).  Both sum terms of at most w_j |X_j| whose factor
    b_a is known to some ten roundings of 1: 1e-14 of the sides' own weighted currents
    (times k0 / 4 pi), whatever the weights elsewhere."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as mb
    curve, M, k0, npol = W.sphere(16), 12, 3.0, 120
    assert 24 * 60 * curve.N * (2 * M + 1) < 2e7 <= 8 * 24 * 60 * curve.N * (2 * M + 1)
    ctx = mb.build(curve, W.Media.from_k(k0, 4.5), M, mb.Options(n_phi=64, precision=1))
    rng = np.random.default_rng(nodes)
    weight = 2 * np.pi * curve.r * np.tile(np.polynomial.legendre.leggauss(16)[1], 16) * np.hypot(curve.dr, curve.dz)
    near = np.argsort(curve.r)[:nodes]
    x = np.zeros((2 * M + 1, 8, curve.N, 4), dtype=complex)
    for side, m in enumerate((0, 1, -1, 2, -3, 5, 12, -12)):
        x[M + m, side, near] = rng.standard_normal((nodes, 4)) + 1j * rng.standard_normal((nodes, 4))
    size = (np.abs(x).sum(-1) * weight).sum((0, 2)) * k0 / (4 * np.pi)
    X = torch.tensor(x.reshape(2 * M + 1, 8, -1), device=DEV)
    E = torch.zeros((8, npol, 3, 3), dtype=torch.complex128, device=DEV)
    ctx.far_field_grid(X, E)
    one = torch.zeros((1, npol, 3, 3), dtype=torch.complex128, device=DEV)
    for side in range(8):
        ctx.far_field_grid(X[:, side:side + 1].contiguous(), one)
        assert float((E[side] - one[0]).abs().max()) <= 1e-14 * size[side], side
    ctx.close()
