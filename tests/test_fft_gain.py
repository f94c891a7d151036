"""The gain of the register transforms (csrc/fft_reg.cuh, compiled for the host): what the rounding
of their constants does to every element alike, which no sum averages out. With every constant
rounded by itself to FP32 the compiled grid edges have gain errors of up to 2.3e-8 (48 points)."""
import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]
LENGTHS = (3, 4, 5, 8, 9, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 60)

SOURCE = r"""
#include <math.h>
#include <cstdio>
#include <random>
#include "fft_reg.cuh"
// sum |X|^2 / (N sum |x|^2), 1 for an exact transform (Parseval)
template <int N, int SIGN> double energy() {
  std::mt19937 g(7);
  std::normal_distribution<double> d;
  double a = 0, b = 0;
  for (int v = 0; v < 400000 / N; ++v) {
    float re[N], im[N];
    for (int i = 0; i < N; ++i) {
      re[i] = float(d(g)); im[i] = float(d(g));
      a += double(re[i]) * re[i] + double(im[i]) * im[i];
    }
    occri::fft::pfa<N, SIGN>(re, im);
    for (int i = 0; i < N; ++i) b += double(re[i]) * re[i] + double(im[i]) * im[i];
  }
  return b / (N * a);
}
template <int N> void row() {
  printf("%d %.17g %.17g\n", N, energy<N, -1>() - 1, energy<N, 1>() - 1);
}
int main() { ROWS }
"""


@pytest.fixture(scope="module")
def gains(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("fft")
    (d / "gain.cc").write_text(SOURCE.replace("ROWS", " ".join(f"row<{n}>();" for n in LENGTHS)))
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", str(ROOT / "paper_2207_09028_gb300/csrc"),
                    str(d / "gain.cc"), "-o", str(d / "gain")], check=True)
    out = subprocess.run([str(d / "gain")], check=True, capture_output=True, text=True).stdout
    return {int(r.split()[0]): [float(x) for x in r.split()[1:]] for r in out.splitlines()}


@pytest.mark.parametrize("n", LENGTHS)
def test_gain(gains, n):
    # in the amplitude; the rounding of 400,000 random elements leaves about 6e-8 / sqrt(4e5) = 1e-10
    for energy in gains[n]:
        assert abs(energy) / 2 <= 2.3e-8 + 2e-10
