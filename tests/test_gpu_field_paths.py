"""The field kernels at the edges of their tilings: right-hand-side groups,
polar angles below and above a tile, odd grids, mirrored angles, axial waves,
splits of the ring points."""
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


def _ctx(mb, M=5, k1=1.5, panels=3, k0=1.0):
    curve, media = W.random_body(panels, seed=3), W.Media.from_k(k0, k1)
    return curve, media, mb.build(curve, media, M, mb.Options(n_phi=64))


def _currents(seed, M, nrhs, N):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((2 * M + 1, nrhs, 4 * N)) + 1j * rng.standard_normal((2 * M + 1, nrhs, 4 * N))
    return x * 4.0 ** -np.abs(np.arange(-M, M + 1))[:, None, None]


@pytest.mark.parametrize("M,nrhs,npol,naz", [(5, 1, 1, 1), (5, 2, 2, 3), (4, 3, 33, 10), (5, 9, 31, 7), (0, 4, 36, 2)])
def test_far_field_grid_tiles(mb, M, nrhs, npol, naz):
    """The grid far field against the direct quadrature over directions of the
    same library (its own kernel) at every grid direction: both sums carry
    a few hundred rounded terms of size 1, <= 1e-13 of the largest component."""
    curve, media, ctx = _ctx(mb, M)
    x = torch.tensor(_currents(1, M, nrhs, curve.N), device=DEV)
    E = torch.zeros((nrhs, npol, naz, 3), dtype=torch.complex128, device=DEV)
    ctx.far_field_grid(x, E)
    T, P = np.meshgrid((np.arange(npol) + 0.5) * np.pi / npol, 2 * np.pi * np.arange(naz) / naz, indexing="ij")
    dirs = np.stack([np.sin(T) * np.cos(P), np.sin(T) * np.sin(P), np.cos(T)], -1).reshape(-1, 3)
    ref = torch.zeros((nrhs, npol * naz, 3), dtype=torch.complex128, device=DEV)
    ctx.far_field(x, torch.tensor(dirs, device=DEV), ref)
    ref = ref.reshape(E.shape)
    assert float((E - ref).abs().max()) <= 1e-13 * float(ref.abs().max())
    ctx.close()


@pytest.mark.parametrize("M,nrhs,k0", [(0, 1, 1.0), (1, 3, 0.5), (6, 9, 4.0), (33, 2, 2.0)])
def test_rhs_planewave_rings(mb, M, nrhs, k0):
    """Plane-wave data against the oracle's trapezoid of the sampled traces:
    axial, equatorial and oblique waves, <= 1e-14 of the largest entry times
    the phase |k0| r (below 5) they both round."""
    from oracle import fields
    curve, media, ctx = _ctx(mb, M, k1=1.5 * k0, k0=k0)
    rng = np.random.default_rng(5)
    dirs = [[0.0, 0.0, 1.0], [0.0, 1.0, 0.0], [1e-160, 0.0, -1.0]] + list(rng.standard_normal((nrhs, 3)))
    first = 3 if M == 0 else 0  # an axial wave has the modes +-1 alone
    waves = [W.plane_wave(d, [1.0, 0.3, 0.2]) for d in dirs[first:first + nrhs]]
    rhs = torch.zeros((2 * M + 1, nrhs, 4 * curve.N), dtype=torch.complex128, device=DEV)
    ctx.rhs_planewave([w.d for w in waves], [w.e for w in waves], rhs)
    ref = fields.modal_rhs(curve, media, M, waves).transpose(0, 2, 1)
    assert np.abs(rhs.cpu().numpy() - ref).max() <= 5e-14 * np.abs(ref).max()
    ctx.close()


@pytest.mark.parametrize("nrhs,nt,region,k1", [(1, 1, 0, 1.5), (2, 7, 1, 1.5 + 0.1j), (3, 700, 0, 1.5), (5, 2, 1, 1.5)])
def test_eval_splits(mb, nrhs, nt, region, k1):
    """Fields at points against the oracle's direct sum on the same nodes (the
    points are farther than 1.5 panel lengths, where panels are not split and
    the oracle's upsampling, a finer rule, is off), with one and many splits of
    the ring points and right-hand sides that leave half a group: <= 1e-12 of
    the largest component."""
    from oracle import fields
    M = 4
    curve, media, ctx = _ctx(mb, M, k1=k1, panels=8)
    x = _currents(2, M, nrhs, curve.N)
    rng = np.random.default_rng(9)
    d = rng.standard_normal((nt, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    P = d * rng.uniform(3.0, 4.0, (nt, 1)) if region == 0 else 0.02 * d
    out = torch.zeros((nrhs, nt, 6), dtype=torch.complex128, device=DEV)
    ctx.eval(torch.tensor(x, device=DEV), P, region, out)
    sub = slice(0, min(nt, 9))
    E, H = fields.near_field(curve, media, M, x.transpose(0, 2, 1), P[sub], region, formulation=0, upsample=1)
    ref = np.concatenate([E, H], -1)
    assert np.abs(out.cpu().numpy()[:, sub] - ref).max() <= 1e-12 * np.abs(ref).max()
    ctx.close()
