"""The mixed form's mesh fractions (double-float arithmetic, compiled for the
host from the kernels' own header) against exact rational arithmetic."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2503_07526_gb300 import build_lib, synth

MAIN = r"""
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include "common.cuh"
int main() {
  int num, den;
  float oh, ol, kh, kl;
  while (std::scanf("%d %d %a %a %a %a", &num, &den, &oh, &ol, &kh, &kl) == 6) {
    int base;
    const float f = otf::df_fraction(num, den, otf::dfloat{oh, ol}, otf::dfloat{kh, kl}, base);
    std::printf("%d %a\n", base, f);
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = build_lib._nvcc()
    if not (os.path.exists(nvcc) or shutil.which(nvcc)):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("df")
    (d / "main.cu").write_text(MAIN)
    subprocess.run([nvcc, *build_lib.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-ffp-contract=off",
                    "-I" + build_lib.INCLUDE, "-I" + build_lib.CSRC, "-o", str(d / "main"), str(d / "main.cu")],
                   check=True)
    return str(d / "main")


def words(x):
    h = np.float32(x)
    return h, np.float32(x - float(h))


@pytest.mark.parametrize("K", [8, 16, 48, 128, 512])
@pytest.mark.parametrize("nc", [3, 7, 14, 100, 1023])
def test_fractions_are_rounded_once(program, K, nc):
    """Half an ulp of a number below one, 2^-25, and 1e-12 for the double-float
    coordinate (at most 512 / 3 mesh points of an offset, 2^-46 relative)."""
    u = synth.uniform01(K + nc, 800)
    L = 3.3 * nc
    kl = K / L
    kh, kw = words(kl)
    lines, want = [], []
    for c, x in zip((u[:400] * nc).astype(int), 1.1 * u[400:] - 0.55):
        oh, ol = words(x * L / nc)
        num = (2 * int(c) + 1) * K
        lines.append(f"{num} {2 * nc} {float(oh).hex()} {float(ol).hex()} {float(kh).hex()} {float(kw).hex()}")
        want.append(Fraction(num, 2 * nc) + (Fraction(float(oh)) + Fraction(float(ol))) * Fraction(kl))
    out = subprocess.run([program], input="\n".join(lines), capture_output=True, text=True, check=True).stdout.split()
    worst = max(abs(int(b) + Fraction(float.fromhex(f)) - w) for b, f, w in zip(out[::2], out[1::2], want))
    assert len(out) == 2 * len(want) and all(0.0 <= float.fromhex(f) <= 1.0 for f in out[1::2])
    assert float(worst) <= 2.0 ** -25 + 1e-12
