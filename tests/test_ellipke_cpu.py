"""K and E from the complementary modulus (csrc/special.cuh, compiled for the CPU), which the
split pairs' coefficients start from, against mpmath at 60 digits."""
import os
import shutil
import subprocess

import numpy as np
import pytest

mpmath = pytest.importorskip("mpmath")

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
def test_ellipke_against_mpmath(tmp_path):
    """Moduli kc from 1e-12 to 1 and close to 1.  At most seven steps of sums of positive
    terms, some four roundings each: 28 x 2^-53 = 3.1e-15, relative."""
    exe = str(tmp_path / "ellipke_check")
    subprocess.run(["nvcc", "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "native", "ellipke_check.cu")],
                   check=True, capture_output=True, timeout=300)
    kcs = np.concatenate([np.geomspace(1e-12, 1.0, 80), 1.0 - np.geomspace(1e-15, 0.5, 40)])
    out = subprocess.run([exe], input="\n".join(repr(float(k)) for k in kcs) + "\n", capture_output=True, text=True,
                         timeout=60)
    assert out.returncode == 0, out.stderr
    with mpmath.workdps(60):
        for kc, line in zip(kcs, out.stdout.strip().split("\n")):
            m = 1 - mpmath.mpf(float(kc)) ** 2
            for got, want in zip(line.split(), (mpmath.ellipk(m), mpmath.ellipe(m))):
                assert abs((mpmath.mpf(float(got)) - want) / want) <= 3.1e-15, kc
