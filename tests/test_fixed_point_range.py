"""Range of the integer stencil formulas (csrc/mg_fixed.cuh), on the CPU.

The formulas are compiled over a type that holds, instead of a number, the coefficients of
the inputs it is a sum of.  With every input at the largest magnitude it can have and the
worst of all signs, the size of an intermediate is the sum of its coefficients' magnitudes
times the inputs'.  No intermediate may reach 2^63.
"""

import json
import subprocess

import pytest

PROGRAM = r"""
#include <cmath>
#include <cstdio>

#include "mg_fixed.cuh"

static double worst;  // largest intermediate, in units of 2^59

struct Lin {
  double c[4];  // coefficients times the inputs' largest magnitude, in units of 2^59
  double size() const { return std::fabs(c[0]) + std::fabs(c[1]) + std::fabs(c[2]) + std::fabs(c[3]); }
};
static Lin input(int q, double range) {
  Lin l{};
  l.c[q] = range;
  return l;
}
static Lin seen(Lin l) {
  worst = std::fmax(worst, l.size());
  return l;
}
static Lin mix(Lin a, double fa, Lin b, double fb) {
  Lin o;
  for (int q = 0; q < 4; ++q) o.c[q] = fa * a.c[q] + fb * b.c[q];
  return seen(o);
}
Lin operator+(Lin a, Lin b) { return mix(a, 1, b, 1); }
Lin operator-(Lin a, Lin b) { return mix(a, 1, b, -1); }
Lin operator*(int f, Lin a) { return mix(a, f, a, 0); }
Lin operator>>(Lin a, int n) { return mix(a, std::ldexp(1.0, -n), a, 0); }

template <int ORDER>
void order() {
  // sums of 6 neighbours at each distance, sums or differences of 2
  const Lin six[3] = {input(0, 6), input(1, 6), input(2, 6)};
  const Lin two[3] = {input(0, 2), input(1, 2), input(2, 2)};
  const Lin c = input(3, 1);
  worst = 0;
  seen(mgk::fx_weighted<ORDER>(six) + mgk::fx_centre<ORDER>(c));
  const double lap = worst;
  worst = 0;
  seen(mgk::fx_second<ORDER>(two, c));
  const double second = worst;
  worst = 0;
  const double b = seen(mgk::fx_first<ORDER>(two)).size();
  const double first = worst;
  // differences of two first derivatives
  const Lin again[3] = {input(0, 2 * b), input(1, 2 * b), input(2, 2 * b)};
  worst = 0;
  seen(mgk::fx_first<ORDER>(again));
  printf("\"%d\": {\"laplacian\": %.4f, \"second\": %.4f, \"first\": %.4f, \"mixed\": %.4f}", ORDER,
         lap, second, first, worst);
}

int main() {
  printf("{");
  order<2>();
  printf(", ");
  order<4>();
  printf(", ");
  order<6>();
  printf("}\n");
  return 0;
}
"""


@pytest.fixture(scope="module")
def sizes(tmp_path_factory):
    from paper_1103_6031_gb300 import build as b
    d = tmp_path_factory.mktemp("range")
    src, exe = str(d / "range.cu"), str(d / "range")
    with open(src, "w") as f:
        f.write(PROGRAM)
    cmd = [b._nvcc()] + b.ARCH + ["-std=c++17", "-diag-suppress=20011,20014", "-I", b.INCLUDE, "-I",
                                  b.CSRC, src, "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    return json.loads(subprocess.run([exe], capture_output=True, text=True, check=True).stdout)


@pytest.mark.parametrize("what", ("laplacian", "second", "first", "mixed"))
@pytest.mark.parametrize("order", ("2", "4", "6"))
def test_no_intermediate_overflows(sizes, order, what):
    # 16 units are 2^63; the low bits that the shifts drop stay below 2^-50 of a unit
    assert sizes[order][what] < 15.99, sizes[order]
