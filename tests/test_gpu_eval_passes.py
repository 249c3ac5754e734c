"""Fields close to the surface: more ring points and sides than one pass of the
tensor-core products holds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W

DEV = "cuda:0"


@pytest.mark.parametrize("d,nrhs", [(0.006, 12), (0.02, 3)])
def test_close_points_in_passes(d, nrhs):
    """Nine copies of one point (two row tiles) against the point alone and one side at a
    time (the FP64 pipe), over the same ring points.  Digits keep 2^-57 of the largest
    kernel among 512 ring points (3.5e-15 for all of them), FP64 terms 2^-52 each, and
    close to the surface the terms add up to about a hundred times the field: 1e-12 of
    the largest component.  Copies get the same bits."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_07067_gb300 as mb
    M = 4
    curve, media = W.random_body(4, seed=4), W.Media.from_k(1.0, 1.5)
    ctx = mb.build(curve, media, M, mb.Options(n_phi=64))
    rng = np.random.default_rng(nrhs)
    x = rng.standard_normal((2 * M + 1, nrhs, 4 * curve.N)) + 1j * rng.standard_normal((2 * M + 1, nrhs, 4 * curve.N))
    x = torch.tensor(x * 4.0 ** -np.abs(np.arange(-M, M + 1))[:, None, None], device=DEV)
    j = curve.N // 2
    sp = np.hypot(curve.dr[j], curve.dz[j])
    r, z = curve.r[j] + d * curve.dz[j] / sp, curve.z[j] - d * curve.dr[j] / sp
    P = np.tile([[r * np.cos(1.1), r * np.sin(1.1), z]], (9, 1))
    out = torch.zeros((nrhs, 9, 6), dtype=torch.complex128, device=DEV)
    ctx.eval(x, P, 0, out)
    assert torch.equal(out, out[:, :1].expand_as(out))
    one = torch.zeros((1, 1, 6), dtype=torch.complex128, device=DEV)
    for w in (0, nrhs - 1):
        ctx.eval(x[:, w:w + 1].contiguous(), P[:1], 0, one)
        for h in (0, 3):
            assert float((out[w, 0, h:h + 3] - one[0, 0, h:h + 3]).abs().max()) <= \
                1e-12 * float(one[0, 0, h:h + 3].abs().max()), w
    ctx.close()
