"""The constants of the mixed pair sums over boxes of all sizes: the one ratio that
cannot be exact in single precision is within 3e-9 (the first 1e-9 among 256
scattered candidates; all of them further off than 3e-9 has a chance of 1e-8), and
the scales that take the free factor out again are exact to the rounding of their
FP64 and split forms."""
import os
import subprocess

import numpy as np

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "re_internal.h"
int main() {
  double L;
  while (std::scanf("%lf", &L) == 1) {
    re::StepConst k{};
    k.lam32 = L * 0x1.0p-32;
    re::set_pair_constants(k);
    std::printf("%.17g %.9g %.9g %.9g %.9g %.9g %.17g\n", L, k.cs, k.c1, k.c3, k.eu, k.eul, k.f24);
  }
}
"""


def test_constants(tmp_path):
    from paper_0812_1633_gb300 import build
    src = tmp_path / "c.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "c"
    subprocess.check_call([build._nvcc(), *build.ARCH, "-std=c++17", "-I" + build.CSRC, str(src), "-o", str(exe)])
    L = np.concatenate([(np.array([256, 500, 864, 987, 1372, 2048, 2916, 4000]) / 0.8442) ** (1 / 3),
                        2.0 ** np.arange(2, 8), np.exp(np.random.default_rng(1).uniform(np.log(6), np.log(200), 500))])
    out = subprocess.run([str(exe)], input="\n".join("%.17g" % v for v in L), capture_output=True, text=True, check=True)
    rows = np.array([[float(w) for w in line.split()] for line in out.stdout.splitlines()])
    assert len(rows) == len(L)
    L, f24 = rows[:, 0], rows[:, 6]
    cs, c1, c3, eu, eul = rows[:, 1:6].astype(np.float32).astype(np.float64).T  # nine digits name a float
    inv2 = (2.0 ** 32 / L) ** 2
    kappa = inv2 / -cs
    assert ((kappa >= 0.5) & (kappa < 1)).all() and (np.log2(-cs) % 1 == 0).all()
    assert ((c1 >= 0.5) & (c1 < 1)).all()
    assert np.abs(c3 / c1 / (2 * kappa ** 3) - 1).max() < 3e-9
    assert np.abs((eu + eul) * c1 * c1 - 1).max() < 1e-14
    assert np.abs(f24 * c1 / (24 * kappa ** 4) - 1).max() < 1e-14
