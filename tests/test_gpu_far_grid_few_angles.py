"""Far field on a grid of at most four polar angles (FP64 pipe): tiles of two angles and
every number of sides a block takes, nodes that leave a part of a block's share."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W

DEV = "cuda:0"


@pytest.mark.parametrize("panels,M,nrhs,npol", [(1, 0, 1, 1), (3, 2, 1, 2), (5, 3, 2, 3), (7, 10, 5, 7), (3, 20, 9, 8),
                                                (5, 60, 3, 5), (2, 80, 17, 6)])
def test_few_angles(panels, M, nrhs, npol):
    """Against the direct quadrature over directions of the same library: a few hundred
    rounded terms of size 1, <= 1e-13 of the largest component."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as mb
    curve = W.random_body(panels, seed=panels)
    assert (npol + 1) // 2 <= 4 and 24 * ((npol + 1) // 2) * curve.N * (2 * M + 1) * nrhs < 2e7
    ctx = mb.build(curve, W.Media.from_k(1.0, 1.5), M, mb.Options(n_phi=64, precision=1))
    rng = np.random.default_rng(nrhs)
    x = rng.standard_normal((2 * M + 1, nrhs, 4 * curve.N)) + 1j * rng.standard_normal((2 * M + 1, nrhs, 4 * curve.N))
    x = torch.tensor(x * 2.0 ** -np.abs(np.arange(-M, M + 1))[:, None, None], device=DEV)
    naz = 5
    E = torch.zeros((nrhs, npol, naz, 3), dtype=torch.complex128, device=DEV)
    ctx.far_field_grid(x, E)
    T, P = np.meshgrid((np.arange(npol) + 0.5) * np.pi / npol, 2 * np.pi * np.arange(naz) / naz, indexing="ij")
    dirs = np.stack([np.sin(T) * np.cos(P), np.sin(T) * np.sin(P), np.cos(T)], -1).reshape(-1, 3)
    ref = torch.zeros((nrhs, npol * naz, 3), dtype=torch.complex128, device=DEV)
    ctx.far_field(x, torch.tensor(dirs, device=DEV), ref)
    assert float((E - ref.reshape(E.shape)).abs().max()) <= 1e-13 * float(ref.abs().max())
    ctx.close()
