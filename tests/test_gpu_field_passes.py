"""Field products cut into many passes (angles, blocks of ring integrals, indices, sides,
ring points, waves) against the same calls in one pass."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W

DEV = "cuda:0"


@pytest.fixture()
def body():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as mb
    M = 24
    curve = W.random_body(16, seed=5)
    ctx = mb.build(curve, W.Media.from_k(4.0, 6.0 + 0.1j), M, mb.Options(n_phi=64, precision=1))
    rng = np.random.default_rng(8)
    x = rng.standard_normal((2 * M + 1, 7, 4 * curve.N)) + 1j * rng.standard_normal((2 * M + 1, 7, 4 * curve.N))
    yield ctx, M, curve, rng, torch.tensor(x, device=DEV)
    ctx.close()


def _both(monkeypatch, call, out):
    """A pass sums the same digits in the same order as the whole call does: equal bits."""
    call(out)
    whole = out.clone()
    out.zero_()
    monkeypatch.setenv("MUELLER_FAULT_INJECT", "small_passes")
    call(out)
    assert torch.equal(out, whole)
    assert float(whole.abs().max()) > 0.0


@pytest.mark.parametrize("npol,naz", [(181, 90), (40, 7), (2, 33)])
def test_far_field_grid(body, monkeypatch, npol, naz):
    ctx, M, curve, rng, x = body
    x = x if npol > 2 else x.repeat(1, 10, 1)
    assert 24 * ((npol + 1) // 2) * curve.N * (2 * M + 1) * x.shape[1] >= 2e7  # the tensor-core form is taken
    _both(monkeypatch, lambda E: ctx.far_field_grid(x, E),
          torch.zeros((x.shape[1], npol, naz, 3), dtype=torch.complex128, device=DEV))


def test_points(body, monkeypatch):
    ctx, M, curve, rng, x = body
    d = rng.standard_normal((60, 3))
    P = 3.0 * d / np.linalg.norm(d, axis=1, keepdims=True)
    _both(monkeypatch, lambda out: ctx.eval(x, P, 0, out), torch.zeros((7, 60, 6), dtype=torch.complex128, device=DEV))


def test_plane_waves(body, monkeypatch):
    ctx, M, curve, rng, x = body
    waves = [W.plane_wave(d, [1.0, 0.3, 0.2]) for d in rng.standard_normal((600, 3))]
    _both(monkeypatch, lambda rhs: ctx.rhs_planewave([w.d for w in waves], [w.e for w in waves], rhs),
          torch.zeros((2 * M + 1, 600, 4 * curve.N), dtype=torch.complex128, device=DEV))
