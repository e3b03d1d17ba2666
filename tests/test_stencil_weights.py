"""The FP32 second-derivative weights of the 3D kernels against the exact Taylor weights in
64 bits: the relative error of the symbol sum 2 w_j (cos(j k h) - 1), a run's phase error.
The y = 2 kernels take the set whose rounding errors cancel for smooth waves."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_03345_gb300", "csrc")

PROGRAM = r"""
#define __device__
#define __forceinline__ inline
#include "stencil3d.cuh"
#include <cstdio>
int main() {
  for (int j = 1; j <= 4; ++j) printf("%.17g %.17g\n", (double)fwi::w2c<4>(j), (double)fwi::w2s<4>(j));
  for (int j = 1; j <= 5; ++j) printf("%.17g %.17g\n", (double)fwi::w2c<5>(j), (double)fwi::w2s<5>(j));
}
"""
EXACT = {8: [8 / 5, -1 / 5, 8 / 315, -1 / 560], 10: [5 / 3, -5 / 21, 5 / 126, -5 / 1008, 1 / 3150]}


@pytest.fixture(scope="module")
def weights(tmp_path_factory):
    d = tmp_path_factory.mktemp("w")
    (d / "w.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "w.cpp"), "-o", str(d / "w")], check=True)
    w = np.array([line.split() for line in subprocess.check_output([str(d / "w")], text=True).splitlines()], float)
    return {8: w[:4].T, 10: w[4:].T}


@pytest.mark.parametrize("order", [8, 10])
def test_symbol(weights, order):
    kh = np.linspace(0.02, 1.3, 200)
    sym = lambda w: sum(2 * a * (np.cos((j + 1) * kh) - 1) for j, a in enumerate(w))  # noqa: E731
    nearest, smooth = (np.abs(sym(w) / sym(EXACT[order]) - 1) for w in weights[order])
    assert np.array_equal(weights[order][0], np.float32(EXACT[order]).astype(float))
    w = np.float32(weights[order][0])
    assert all(b in (a, np.nextafter(a, np.float32(9)), np.nextafter(a, np.float32(-9)))
               for a, b in zip(w, np.float32(weights[order][1])))
    assert smooth[kh <= 0.5].max() < 6e-9 and nearest[kh <= 0.5].max() > 1.4e-8
    assert smooth.max() < 3e-8
