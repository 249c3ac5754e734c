"""Fields at many points by products on the tensor cores against the same points a few
at a time, whose sums run on the FP64 pipe: ring points that leave a part of the last
index, row tiles with a remainder, one to three column tiles, a lossy interior."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W

DEV = "cuda:0"


@pytest.mark.parametrize("panels,nrhs,nt,region,k1", [(6, 1, 130, 0, 1.5), (7, 3, 121, 1, 1.5 + 0.2j), (6, 7, 150, 0, 1.5)])
def test_many_points_like_few(panels, nrhs, nt, region, k1):
    """Both paths round a few thousand terms below 1e-2 of the largest sum's bound of
    their absolute values; the terms of a point far from the surface cancel little:
    components agree to 1e-13 of the largest."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as mb
    M = 5
    curve, media = W.random_body(panels, seed=panels), W.Media.from_k(1.0, k1)
    ctx = mb.build(curve, media, M, mb.Options(n_phi=64))
    rng = np.random.default_rng(panels)
    x = rng.standard_normal((2 * M + 1, nrhs, 4 * curve.N)) + 1j * rng.standard_normal((2 * M + 1, nrhs, 4 * curve.N))
    x = torch.tensor(x * 4.0 ** -np.abs(np.arange(-M, M + 1))[:, None, None], device=DEV)
    d = rng.standard_normal((nt, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    P = d * rng.uniform(3.0, 4.0, (nt, 1)) if region == 0 else 0.02 * d
    out = torch.zeros((nrhs, nt, 6), dtype=torch.complex128, device=DEV)
    ctx.eval(x, P, region, out)
    few = torch.zeros((nrhs, 5, 6), dtype=torch.complex128, device=DEV)
    for i in (0, 7, nt - 5):
        ctx.eval(x, P[i:i + 5], region, few)
        assert float((out[:, i:i + 5] - few).abs().max()) <= 1e-13 * float(few.abs().max()), i
    ctx.close()
