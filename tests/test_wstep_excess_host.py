"""Host check of the excess ratios 1 - rho2 / u of the W-step pivots u (no GPU needed).

wstep_excess (compiled here for the host) against the pivots of the run blocks
of K_{mu rho2} taken exactly in rational arithmetic, up to rho2 = 1e12, where
1 - rho2 inv formed in FP64 keeps only ten digits.  Tolerance: a step of the
recurrence has four roundings and damps the error of the step before it, so
some ten units of 2^-53."""
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2005_09838_gb300 import build

PROG = r'''
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "tc_kernels.cuh"
int main(int argc, char** argv) {
  const int n2 = std::atoi(argv[1]);
  std::vector<double> h(2 * (size_t)n2);
  tc::wstep_excess<double>(h.data(), n2, std::atof(argv[2]), std::atof(argv[3]));
  for (double v : h) std::printf("%.17g\n", v);
  return 0;
}
'''


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("wexc")
    src, exe = d / "wexc.cu", d / "wexc"
    src.write_text(PROG)
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.INCLUDE,
                    "-I", build.CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("n2", [2, 9, 33])
@pytest.mark.parametrize("mu,rho2", [(1e-3, 1e-1), (0.0, 1e6), (0.5, 1e12)])
def test_excess_ratios_against_exact_pivots(prog, n2, mu, rho2):
    out = subprocess.run([str(prog), str(n2), repr(mu), repr(rho2)], check=True, capture_output=True, text=True)
    h = np.array([float(v) for v in out.stdout.split()]).reshape(2, n2)
    m, p = Fraction(mu), Fraction(rho2)
    for b, first in enumerate((1 + m + p, 1 + m + 2 * p)):
        u = first
        for q in range(n2):
            exact = 1 - p / u
            assert abs(Fraction(float(h[b, q])) - exact) <= Fraction(2) ** -49 * exact, (b, q)
            u = 1 + m + 2 * p - p * p / u
