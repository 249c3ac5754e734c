"""Workspace plans of the tensor-core field products (csrc/fields_plan.cuh, compiled for
the CPU): what the kernels of every pass write, counted here from their tiles, ends
inside the block that the plan asks for."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
MB = 1 << 20


def _up(a, b):
    return -(-a // b)


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("plan") / "fields_plan_check")
    subprocess.run(["nvcc", "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "native", "fields_plan_check.cu")],
                   check=True, capture_output=True, timeout=300)

    def run(op, cases, small=False):
        env = dict(os.environ, MUELLER_FAULT_INJECT="small_passes" if small else "")
        lines = "".join(op + " " + " ".join(str(v) for v in c) + "\n" for c in cases)
        out = subprocess.run([exe], input=lines, capture_output=True, text=True, timeout=300, env=env)
        assert out.returncode == 0, out.stderr
        rows = [[int(v) for v in line.split()] for line in out.stdout.strip().split("\n")]
        assert len(rows) == len(cases)
        return rows

    return run


def test_plane_wave_passes_stay_inside(plan):
    """Bodies of 16 to 4096 nodes, 1 to 65535 waves; launches take at most 1024 of them."""
    rng = np.random.default_rng(11)
    cases = [(64, 10, 96, 2200), (128, 32, 144, 1500), (160, 20, 112, 2000), (256, 32, 144, 1500), (128, 64, 208, 1100)]
    for N in (16, 32, 64, 128, 256, 512, 1024, 4096):
        for nrhs in (1, 2, 1023, 1024, 1025, 2048, 65535):
            M = int(rng.integers(0, 560))
            cases.append((N, M, (2 * M + 64 + int(rng.integers(0, 400)) + 15) // 16 * 16, nrhs))
    for (N, M, n, nrhs), (nkt, nct, waves, a, table, cost, coef, nbytes) in zip(cases, plan("rhs", cases)):
        assert nkt == _up(n // 4 + 1, 16) and nct * 32 > (M + 1) // 2
        assert 1 <= waves <= min(nrhs, 1024)
        rows = _up(waves * N, 128) * 128                     # of the fullest pass
        assert a == 0 and a + 2 * nkt * rows * 16 * 8 * 2 <= table          # two parities, 8 digits of 2 bytes
        assert table + 2 * nkt * nct * 32 * 16 * 8 * 2 <= cost
        assert cost + nkt * 16 * 8 <= coef
        assert coef + 2 * nct * 32 * rows * 8 <= nbytes
        assert waves == 1 or 2 * nkt * rows * 256 <= 512 * MB
        assert all(v % 256 == 0 for v in (table, cost, coef))


def test_field_passes_stay_inside_and_bounded(plan):
    """From 16 ring points to those of 4096 sub-nodes at 8192 azimuths, 1 to 1e5 points, up
    to 65535 sides: every pass inside its parts, no part above 512 MB."""
    rng = np.random.default_rng(12)
    cases = [(t, nt, w) for t in (16, 512, 528, 46080, 262144, 262160, 1024 * 8192, 4096 * 8192)
             for nt in (1, 7, 8, 100, 100000) for w in (1, 2, 10, 11, 100, 65535)]
    cases += [(16 * int(rng.integers(1, 1 << 20)), int(rng.integers(1, 3000)), int(rng.integers(1, 3000)))
              for _ in range(200)]
    for (total, nt, nrhs), row in zip(cases, plan("nf", cases)):
        na, nap, npt, nrt, nw, nct, groups, passes, a, r, b, c, y, s, group, nbytes = row
        assert na == _up(total, 512) and 1 <= nap <= na and 1 <= npt <= nt and 1 <= nw <= nrhs and groups >= 1 and passes >= 1
        assert 18 * npt <= 128 * nrt and 12 * nw <= 32 * nct
        rows, cols = 128 * nrt, 32 * nct                     # of the fullest product, 8 digits of 2 bytes each
        assert a == 0 and a + nap * rows * 512 * 8 * 2 <= r and r + nap * rows * 8 <= b
        assert b + nap * cols * 512 * 8 * 2 <= c and c + nap * cols * 8 <= y
        assert y + nap * cols * rows * 8 <= s
        assert group >= cols * rows and s + ((passes * groups - 1) * group + cols * rows) * 8 <= nbytes
        assert max(r, c - b, s - y, nbytes - s) <= 512 * MB + 256 and nbytes <= 2200 * 10 ** 6
        assert all(v % 256 == 0 for v in (r, b, c, y, s))
        if na <= 512 and 18 * nt <= 128 * (512 // na):
            assert nap == na and npt == nt                   # nothing is cut that fits whole


def test_far_field_grid_passes_stay_inside_and_bounded(plan):
    """16 to 4096 nodes, modes up to 568, 1 to 3600 polar angles, up to 14000 azimuths and
    65535 sides: every pass inside its parts, none of them above 512 MB; nothing is cut
    that fits whole."""
    rng = np.random.default_rng(13)
    cases = [(N, M, npol, naz, (2 * M + 64 + 15) // 16 * 16, w) for N in (16, 512, 1024, 4096) for M in (0, 64, 128, 568)
             for npol, naz in ((1, 1), (2, 8), (180, 360), (3600, 7200)) for w in (1, 8, 1000)]
    cases += [(16 * int(rng.integers(1, 257)), M, int(rng.integers(1, 2000)), int(rng.integers(1, 14001)),
               (2 * M + int(rng.integers(64, 1000)) + 15) // 16 * 16, int(rng.integers(1, 65536)))
              for M in rng.integers(0, 569, 200).tolist()]
    for small in (False, True):
        for (N, M, npol, naz, n, nrhs), row in zip(cases, plan("grid", cases, small)):
            (P2, rkt, rct, np_, nrt, nps, nap, nw, nct, skt, sct, swp, nkt,
             phase, a, r, b, c, y, table, cost, coef, block, nbytes) = row
            na = M + 2
            assert P2 == (npol + 1) // 2 and nkt == N // 16 and rkt == _up(n // 4 + 1, 16) and rct * 32 > (M + 1) // 2
            assert 1 <= nps <= np_ <= P2 and 2 * np_ <= 128 * nrt and 1 <= nap <= na and 1 <= nw <= nrhs
            assert 24 * nw <= 32 * nct and skt * 16 > M and sct * 32 > naz // 2 and 1 <= swp <= nrhs * npol
            rows, cols, rrows, srows = 128 * nrt, 32 * nct, 128 * _up(nps * N, 128), 128 * _up(6 * swp, 128)
            assert phase == 0 and N * (P2 * 16 + 24) <= a
            parts = dict(a=max(nap * rows * nkt, 2 * rrows * rkt, 2 * srows * skt) * 16 * 8 * 2,
                         r=max(nap * rows, 2 * srows) * 8, b=max(nap * cols * nkt, 2 * sct * 32 * skt) * 16 * 8 * 2,
                         c=nap * cols * 8, y=max(na * cols * rows, 2 * sct * 32 * srows) * 8,
                         table=2 * rkt * rct * 32 * 16 * 8 * 2, cost=rkt * 16 * 8,
                         coef=(_up(np_, nps) - 1) * block + 2 * rct * 32 * rrows * 8)
            for (_, size), lo, hi in zip(parts.items(), (a, r, b, c, y, table, cost, coef),
                                         (r, b, c, y, table, cost, coef, nbytes)):
                assert lo % 256 == 0 and lo + size <= hi
            if not small:
                assert max(parts["a"], parts["b"], parts["y"], nbytes - coef) <= 512 * MB + rrows * rct * 512
            if not small and na * nkt * 128 * _up(2 * P2, 128) * 256 <= 512 * MB and npol <= 180 and N <= 1024:
                assert np_ == P2 and nap == na
