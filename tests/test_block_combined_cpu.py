"""The far-pair assembly's two-step block (csrc/block.cuh, compiled for the CPU)
against the oracle's Lemma 1 and modal N and K operators: both forms, real and
lossy interior, non-unit vacuum parameters (K factors other than +-1), modes 0,
1 and the highest.  Each entry is a sum of a few dozen products, rounded a few
times each: 2e-14 of the block's largest entry."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import system
from workloads.configs import Media

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _c(z):
    z = complex(z)
    return f"{z.real!r} {z.imag!r}"


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
def test_two_step_block_matches_oracle(tmp_path):
    exe = str(tmp_path / "block_combined_check")
    subprocess.run(["nvcc", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-o", exe,
                    os.path.join(HERE, "native", "block_combined_check.cu")], check=True, capture_output=True,
                   timeout=300)
    rng = np.random.default_rng(77)
    cases, lines = [], []
    for q in range(180):
        form = q % 2
        k0 = float(rng.uniform(0.5, 20.0))
        k1 = complex(k0 * rng.uniform(1.1, 2.0), rng.uniform(1e-3, 0.5) if q % 3 == 2 else 0.0)
        med = Media.from_k(k0, k1)
        if q % 5 == 4:
            med = Media(k0, 1.3, 0.7, complex(med.eps1), complex(1.1, 0.01 if q % 3 == 2 else 0.0))
        kk0, kk1 = system.wavenumbers(med)
        M = int(rng.integers(2, 40))
        m = [0, 1, M, int(rng.integers(0, M + 1))][q % 4]
        rt, rs = (float(v) for v in rng.uniform(0.05, 2.0, 2))
        a_t, a_s = rng.uniform(0, 2 * np.pi, 2)
        geo = [float(v) for v in (rt, np.cos(a_t), np.sin(a_t), rs, np.cos(a_s), np.sin(a_s))]
        F = (rng.standard_normal((9, M + 2)) + 1j * rng.standard_normal((9, M + 2))) * 10.0 ** rng.uniform(-3, 3, (9, 1))
        cases.append((form, med, kk0, kk1, m, geo, F))
        lines.append(f"{form} {med.omega!r} {_c(kk0)} {_c(kk1)} {_c(med.eps0)} {_c(med.mu0)} {_c(med.eps1)} "
                     f"{_c(med.mu1)} {M} {m} " + " ".join(repr(v) for v in geo) + " " +
                     " ".join(_c(v) for v in F.reshape(-1)))
    out = subprocess.run([exe], input=f"{len(cases)}\n" + "\n".join(lines) + "\n", capture_output=True, text=True,
                         timeout=300)
    assert out.returncode == 0, out.stderr
    vals, pos, n_simple = out.stdout.split(), 0, 0
    for form, med, kk0, kk1, m, (rt, rpt, zpt, rs, rps, zps), F in cases:
        n_simple += int(vals[pos])
        got = np.array([float(v) for v in vals[pos + 1:pos + 65]]).reshape(2, 4, 4, 2)
        pos += 65
        N0, N1, KD = system.operator_blocks(F[None], np.array([rs]), np.array([rps]), np.array([zps]), rt, rpt, zpt,
                                            kk0, kk1, np.array([m]))
        co = system.coefficients(med, form)
        x0, x1 = co["x"]; y0, y1 = co["y"]
        ref = np.zeros((4, 4), dtype=complex)
        ref[0:2, 0:2] = co["aEJ"] * KD[0, 0]
        ref[0:2, 2:4] = -1j * med.omega * (x0 * N0[0, 0] - x1 * N1[0, 0])
        ref[2:4, 0:2] = -1j * med.omega * (y0 * N0[0, 0] - y1 * N1[0, 0])
        ref[2:4, 2:4] = co["aHM"] * KD[0, 0]
        for v in range(2):
            assert np.abs(got[v, ..., 0] + 1j * got[v, ..., 1] - ref).max() <= 2e-14 * np.abs(ref).max(), (form, m, v)
    assert 40 <= n_simple < len(cases)
