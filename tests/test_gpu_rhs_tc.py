"""Plane-wave data with the ring integrals on the tensor cores (many waves) against
the same waves one at a time, whose integrals run on the FP64 pipe: whole and ragged
row tiles."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W

DEV = "cuda:0"


@pytest.mark.parametrize("panels,M,nrhs", [(16, 64, 130), (3, 64, 700), (9, 95, 140)])
def test_many_waves_like_one(panels, M, nrhs):
    """Both paths share the argument of every sample; their sums round at most n / 4 =
    M + 2 terms of the ring average, so entries agree to 2e-14 of the largest."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as mb
    curve, media = W.random_body(panels, seed=panels), W.Media.from_k(2.0, 3.0)
    ctx = mb.build(curve, media, M, mb.Options(n_phi=256, precision=1))
    n = 4 * curve.N
    rng = np.random.default_rng(panels)
    dirs = rng.standard_normal((nrhs, 3))
    dirs[0] = [0.0, 0.0, 1.0]
    waves = [W.plane_wave(d, [1.0, 0.3, 0.2]) for d in dirs]
    rhs = torch.zeros((2 * M + 1, nrhs, n), dtype=torch.complex128, device=DEV)
    ctx.rhs_planewave([w.d for w in waves], [w.e for w in waves], rhs)
    one = torch.zeros((2 * M + 1, 1, n), dtype=torch.complex128, device=DEV)
    for i in (0, 1, nrhs // 2, nrhs - 1):
        ctx.rhs_planewave([waves[i].d], [waves[i].e], one)
        assert float((rhs[:, i] - one[:, 0]).abs().max()) <= 2e-14 * float(one.abs().max()), i
    ctx.close()
