"""The functions behind the kernel samples (csrc/special.cuh, sample_series and
sample_closed on the CPU) against mpmath from their definitions in x: small x,
both sides of the switch at |x| = 2, large x, real and complex.  Sizes to
compare with: 1 for c and sinc, the size of the closed form's terms (1/|x|^2,
1/|x|^3, 1/|x|, 1/(4 |x|^2) times cosh Im x) or the value at 0 if smaller; a
dozen roundings each: 3e-15."""
import os
import shutil
import subprocess

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _exact(x):
    x = mp.mpc(x)
    s, c = mp.sin(x), mp.cos(x)
    C = (3 - x * x) * c + 3 * x * s - 3
    return [c, s / x, (x * c - s) / x ** 3, ((3 - x * x) * s - 3 * x * c) / x ** 5, (1 - c - x * s) / x ** 2,
            (C / x ** 2 - mp.mpf(1) / 2) / (4 * x * x)]


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
def test_sample_functions(tmp_path):
    exe = str(tmp_path / "sample_fun_check")
    subprocess.run(["nvcc", "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "native", "sample_fun_check.cu")],
                   check=True, capture_output=True, timeout=300)
    rng = np.random.default_rng(3)
    xs = [10.0 ** rng.uniform(-3, 0.3) for _ in range(60)] + list(rng.uniform(1.9, 2.1, 40)) + list(rng.uniform(2, 60, 40))
    xs = [complex(x, x * f) for x in xs for f in (0.0, 0.002, 0.1)]
    out = subprocess.run([exe], input="\n".join(f"{x.real!r} {x.imag!r}" for x in xs), capture_output=True, text=True,
                         timeout=120)
    assert out.returncode == 0
    at0 = [1.0, 1.0, 1 / 3, 1 / 15, 0.5, 1 / 32]
    with mp.workdps(60):
        for x, line in zip(xs, out.stdout.splitlines()):
            v = np.array([float(t) for t in line.split()]).reshape(2, 6, 2)
            v = v[..., 0] + 1j * v[..., 1]
            for row, arg in ((0, x), (1, x.real)):
                r, g = abs(arg), np.cosh(complex(arg).imag)
                size = [g, min(1.0, g), min(1 / 3, g / r ** 2), min(1 / 15, g / r ** 3), min(0.5, g / r),
                        min(1 / 32, g / (4 * r * r))]
                size = [max(s, 1e-3 * z) if r < 2 else s for s, z in zip(size, at0)]
                for q, ref in enumerate(_exact(arg)):
                    assert abs(v[row, q] - complex(ref)) <= 3e-15 * size[q], (arg, q)
