"""The one-dimensional basis of the axis-by-axis L2P (host compiler, no GPU): each value is the exact
one rounded to FP32, like the entries of the interpolation tables that it stands for."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2112_10059_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"
PROBE = r'''
#include "sph_kernels.cuh"
#include <cstdio>
int main() {
    const sph::CellBasis B = sph::cheb_cell_basis();
    for (int k = 0; k < 5; ++k)
        for (int i = 0; i < 4; ++i) printf("%.9g\n", B.v[k][i]);
    return 0;
}
'''


def test_cell_basis_is_the_lagrange_basis_rounded_once(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("host compiler or CUDA headers missing")
    (tmp_path / "p.cpp").write_text(PROBE)
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CUDA_INC, "-I", CSRC, str(tmp_path / "p.cpp"), "-o", str(tmp_path / "p")],
                   check=True, capture_output=True, timeout=120)
    out = subprocess.run([str(tmp_path / "p")], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    got = np.array(out, np.float32).reshape(5, 4)
    # Fractions: only the nodes' own FP64 rounding (1e-16) is left
    t = [Fraction(float(np.cos((2 * k + 1) * np.pi / 10))) for k in range(5)]
    for k in range(5):
        for i in range(4):
            x, v = Fraction(2 * i - 3, 4), Fraction(1)
            for j in range(5):
                if j != k:
                    v *= (x - t[j]) / (t[k] - t[j])
            ulp = float(np.spacing(np.float32(float(v))))
            assert abs(float(Fraction(float(got[k, i])) - v)) <= abs(ulp) * (0.5 + 1e-6), (k, i)
    # a constant is reproduced
    assert np.max(np.abs(got.astype(np.float64).sum(axis=0) - 1)) < 5 * 2.0 ** -25
