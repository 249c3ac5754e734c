"""The library's cache of device blocks: bounded, given back, and reused without
one call's values reaching another (several sizes, threads and streams)."""
import threading

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


def _solve(mb, panels, M, seed, stream=None):
    curve, media = W.random_body(panels, seed=seed), W.Media.from_k(1.0 + 0.1 * seed, 1.5)
    with torch.cuda.stream(stream or torch.cuda.current_stream()):
        ctx = mb.build(curve, media, M, mb.Options(n_phi=64, precision=seed % 2))
        rhs = torch.zeros((2 * M + 1, 2, 4 * curve.N), dtype=torch.complex128, device=DEV)
        w = [W.plane_wave([0.3, 0.4, 1.0], [1.0, 0.0, 0.0]), W.plane_wave([0.0, 1.0, 0.2], [1.0, 0.0, 1.0])]
        ctx.rhs_planewave([v.d for v in w], [v.e for v in w], rhs)
        x = torch.zeros_like(rhs)
        ctx.solve(rhs, x)
        out = x.cpu().numpy()
        ctx.close()
    return out


def test_bounded_and_given_back(mb):
    old = mb.cache_limit(256 << 20)
    try:
        for panels in (3, 9, 5):
            _solve(mb, panels, 20, 1)
            assert mb.cache_bytes() <= (256 << 20) * 2          # the cap, and the small blocks' own
        mb.cache_trim()
        assert mb.cache_bytes() == 0
        mb.cache_limit(0)
        _solve(mb, 3, 6, 0)
        assert mb.cache_bytes() == 0                            # nothing kept when the cap is 0
    finally:
        mb.cache_limit(old)


def test_reused_blocks_carry_nothing_over(mb):
    """Bodies of different sizes alone with empty caches, then interleaved on three
    threads and streams sharing the cache: bitwise the same currents."""
    jobs = [(3, 6, 0), (4, 9, 1), (6, 5, 2), (5, 12, 3)]
    alone = []
    for j in jobs:
        mb.cache_trim()
        alone.append(_solve(mb, *j))
    got, errors = {}, []

    def work(t):
        try:
            s = torch.cuda.Stream()
            for rep in range(3):
                for k in range(len(jobs)):
                    q = (k + t) % len(jobs)
                    got[(t, rep, q)] = _solve(mb, *jobs[q], stream=s)
        except BaseException as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert len(got) == 36
    for (t, rep, q), x in got.items():
        assert np.array_equal(x, alone[q]), (t, rep, q)
