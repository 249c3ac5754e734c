"""Far field on a grid by the tensor-core sums at the edges of their tiles: half a
chunk of nodes and one node tile beyond a chunk, row tiles of angles with a
remainder, full and ragged column tiles, mode 0 alone."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W

DEV = "cuda:0"


@pytest.mark.parametrize("panels,M,nrhs,npol", [(3, 20, 17, 64), (17, 9, 3, 131), (4, 0, 48, 600), (32, 33, 1, 60)])
def test_far_field_grid_products(panels, M, nrhs, npol):
    """Against the direct quadrature over directions of the same library (its own
    kernel) at every grid direction: both sums carry a few hundred rounded terms of
    size 1, <= 1e-13 of the largest component.  A side with a NaN current has no
    finite field and leaves the others' bits alone."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as mb
    assert 24 * ((npol + 1) // 2) * 16 * panels * (2 * M + 1) * nrhs >= 2e7  # the tensor-core form is taken
    curve, media = W.random_body(panels, seed=panels), W.Media.from_k(1.0, 1.5)
    ctx = mb.build(curve, media, M, mb.Options(n_phi=64))
    rng = np.random.default_rng(nrhs)
    x = rng.standard_normal((2 * M + 1, nrhs, 4 * curve.N)) + 1j * rng.standard_normal((2 * M + 1, nrhs, 4 * curve.N))
    x *= 2.0 ** -np.abs(np.arange(-M, M + 1))[:, None, None]
    x, naz = torch.tensor(x, device=DEV), 3
    E = torch.zeros((nrhs, npol, naz, 3), dtype=torch.complex128, device=DEV)
    ctx.far_field_grid(x, E)
    T, P = np.meshgrid((np.arange(npol) + 0.5) * np.pi / npol, 2 * np.pi * np.arange(naz) / naz, indexing="ij")
    dirs = np.stack([np.sin(T) * np.cos(P), np.sin(T) * np.sin(P), np.cos(T)], -1).reshape(-1, 3)
    ref = torch.zeros((nrhs, npol * naz, 3), dtype=torch.complex128, device=DEV)
    ctx.far_field(x, torch.tensor(dirs, device=DEV), ref)
    ref = ref.reshape(E.shape)
    assert float((E - ref).abs().max()) <= 1e-13 * float(ref.abs().max())
    x[M, nrhs - 1, 5] = float("nan")
    E2 = torch.zeros_like(E)
    ctx.far_field_grid(x, E2)
    assert bool(torch.isnan(E2[-1].abs()).any(-1).all())
    assert torch.equal(E2[:-1], E[:-1])
    ctx.close()
