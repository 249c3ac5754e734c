"""Plane-wave data of more waves than one table holds (1024): each wave as by itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W

DEV = "cuda:0"


@pytest.mark.parametrize("panels,M,nrhs", [(8, 64, 1100), (4, 40, 2200)])
def test_waves_beyond_one_table(panels, M, nrhs):
    """The samples' arguments are the same on both paths and the sums round at most
    n / 4 terms of the ring average: entries agree to 2e-14 of the largest."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as mb
    curve, media = W.random_body(panels, seed=panels), W.Media.from_k(2.0, 3.0)
    ctx = mb.build(curve, media, M, mb.Options(n_phi=256, precision=1))
    rng = np.random.default_rng(panels)
    waves = [W.plane_wave(d, [1.0, 0.3, 0.2]) for d in rng.standard_normal((nrhs, 3))]
    rhs = torch.zeros((2 * M + 1, nrhs, 4 * curve.N), dtype=torch.complex128, device=DEV)
    ctx.rhs_planewave([w.d for w in waves], [w.e for w in waves], rhs)
    one = torch.zeros((2 * M + 1, 1, 4 * curve.N), dtype=torch.complex128, device=DEV)
    for i in (0, 1023, 1024, nrhs - 1):
        ctx.rhs_planewave([waves[i].d], [waves[i].e], one)
        assert float((rhs[:, i] - one[:, 0]).abs().max()) <= 2e-14 * float(one.abs().max()), i
    ctx.close()
