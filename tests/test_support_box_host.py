"""CPU check of the local force's box: the grid indices around an atom outside which its Gaussian is
negligible, for every positive width (the widest overflowed the box's integers)."""
import os
import subprocess

from paper_2106_03872_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cmath>
#include "common.h"
int main() {
  for (int N : {8, 54, 128})
    for (double width : {1e-300, 1e-3, 0.3, 0.8, 5.0, 1e3, 1e7, 4e7, 1e11, 1e300, (double)INFINITY}) {
      const double h = 0.3125;
      const int half = ks::gaussian_half_box(width, h, N);
      // no index beyond the half box of at least half a period carries 1e-20 of the Gaussian
      const double d = half * h;
      const bool covered = half >= N || std::exp(-d * d / (2 * width * width)) <= 1.000001e-20;
      const bool tight = half <= 1 || std::exp(-(d - h) * (d - h) / (2 * width * width)) > 0.999e-20;
      std::printf("%d\n", half >= 0 && half <= N && covered && tight);
    }
  return 0;
}
"""


def test_gaussian_half_box(tmp_path):
    if not os.path.exists(build.LIB):
        build.build()
    src, exe = str(tmp_path / "box.cu"), str(tmp_path / "box")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, src, build.LIB, "-Xlinker",
                    "-rpath=" + os.path.dirname(build.LIB), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == ["1"] * 33
