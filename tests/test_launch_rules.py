"""The rules that choose kernels and launch shapes from sizes, compiled alone, against times
measured on a GB300."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_03345_gb300", "csrc")

PROGRAM = r"""
#include "launch_rules.h"
#include <cstdio>
#include <cstring>
int main() {
  char what[32];
  double a[12];
  while (scanf("%31s", what) == 1) {
    auto read = [&](int n) { for (int i = 0; i < n; ++i) if (scanf("%lf", &a[i]) != 1) return false; return true; };
    if (!strcmp(what, "flags") && read(4))
      printf("%d\n", (int)fwi::density_flags_pay((long long)a[0], (int)a[1], a[2] != 0, a[3] != 0));
    else return 1;
  }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "r.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(d / "r.cpp"), "-o", str(d / "r")], check=True)

    def ask(rows):
        text = "\n".join(" ".join(str(v) for v in r) for r in rows)
        return [float(v) for v in subprocess.check_output([str(d / "r")], input=text, text=True).split()]

    return ask


# grid, PML, forward: cost of the flags and gain per step, gradient: the same (us)
FLAGS = [((40, 44, 48), 0, 39.2, 0.12, 53.4, -0.04), ((64, 64, 64), 0, 40.0, -0.60, 51.8, -0.49),
         ((100, 100, 100), 0, 53.2, -0.38, 58.8, -1.82), ((128, 128, 128), 0, 50.7, -0.19, 61.7, -1.30),
         ((152, 160, 176), 0, 65.1, -0.05, 78.1, -0.40), ((300, 64, 64), 0, 41.5, 0.15, 45.9, 1.11),
         ((192, 180, 200), 0, 91.7, 2.48, 97.6, 11.78), ((256, 256, 256), 0, 163.3, 8.44, 163.8, 20.56),
         ((384, 384, 384), 0, 426.3, 52.66, 315.5, 118.27), ((64, 64, 64), 1, 45.3, -0.19, 50.0, -0.12),
         ((128, 128, 128), 1, 43.8, 4.24, 52.7, 5.90), ((152, 160, 176), 1, 70.2, 5.75, 70.2, 7.62),
         ((300, 64, 64), 1, 32.8, 2.25, 40.8, 5.75), ((192, 180, 200), 1, 88.7, 11.59, 70.2, 40.70),
         ((256, 256, 256), 1, 153.2, 17.46, 122.1, 55.66), ((384, 384, 384), 1, 425.9, 59.39, 250.8, 240.87)]


def test_density_flags(rules):
    """Where the flags are made they win more than they cost, and no call of hundreds of
    steps on a large grid goes without them."""
    rows, want = [], []
    for shape, pml, fc, fg, gc, gg in FLAGS:
        for grad, cost, gain in ((0, fc, fg), (1, gc, gg)):
            for nt in (2, 3, 9, 10, 20, 40, 41, 100, 1000):
                rows.append(("flags", shape[0] * shape[1] * shape[2], nt, grad, pml))
                want.append((gain * nt - cost, nt, shape[0] * shape[1] * shape[2] > 5e6))
    for r, on, (net, nt, large) in zip(rows, rules(rows), want):
        if on:
            assert net > -20, r
        else:
            assert not (large and nt >= 100), r
