"""The FP32 pairs that stand for step coefficients (csrc/fg_kernels.h), compiled
for the host: products near the coefficient, by the C++ that the library uses."""

import pathlib
import shutil
import subprocess

import pytest

HEADER = pathlib.Path(__file__).resolve().parent.parent / "paper_0910_2950_gb300" / "csrc" / "fg_kernels.h"

MAIN = r"""
#include <cmath>
#include <cstdio>
#include <limits>
%s
int main() {
  double worst = 0.0, extra = 0.0;
  for (int i = 1; i <= 3000; ++i) {
    const double k = (i & 1 ? 1 : -1) * std::exp(0.7 * std::sin(1.7 * i)) / (3.0 + i %% 97);
    KickPair p = kick_pair(k);
    if (p.w != 0.0f) return 1;
    worst = std::fmax(worst, std::fabs((double)p.a * p.b / k - 1.0));
    const double c = k * (0.2 + i %% 11);
    if (i <= 300) {
      p = kick_pair(k, c);
      extra = std::fmax(extra, std::fabs((double)p.a * p.b / k - 1.0));
      extra = std::fmax(extra, std::fabs((double)p.w * p.b / c - 1.0));
      p = kick_pair(0.0, c);   // beta = 0
      if (p.a != 0.0f) return 2;
      extra = std::fmax(extra, std::fabs((double)p.w * p.b / c - 1.0));
    }
  }
  const KickPair none = kick_pair(0.0), big = kick_pair(1e39);
  if (none.a != 0.0f || none.b != 0.0f || none.w != 0.0f) return 3;
  if (std::isfinite(big.a * big.b)) return 4;   // beyond FP32: the product says so
  std::printf("%%g %%g\n", worst, extra);
  return worst <= std::ldexp(1.0, -26) && extra <= std::ldexp(1.0, -25) ? 0 : 5;
}
"""


def test_products_are_the_coefficients(tmp_path):
    """Twice as near as FP32 numbers lie at the least, four times without an extra force."""
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    text = HEADER.read_text()
    part = text[text.index("struct KickPair {"):text.index("// FP32 drifts by exp(i c P) likewise")]
    src = tmp_path / "pairs.cpp"
    src.write_text(MAIN % part)
    subprocess.run([gxx, "-O1", "-std=c++17", str(src), "-o", str(tmp_path / "pairs")], check=True)
    assert subprocess.run([str(tmp_path / "pairs")]).returncode == 0
