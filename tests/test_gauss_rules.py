"""The quadrature rules of the coefficients (csrc/gauss_rules.h), compiled for the host: every node and weight is the
nearest double, and a process's first plan hardly pays for them (the extended type is software arithmetic on some
hosts, some 16 ns an operation: 10 000 of them are 0.16 ms).
"""
import decimal
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_02718_gb300", "csrc")
ORDERS = (4, 5, 8, 14, 20, 32)

PROGRAM = r"""
#include <cstdio>
#include "gauss_rules.h"
static long ops = 0;
struct R {
  long double v;
  R() : v(0) {}
  explicit R(double a) : v(a) {}
  explicit R(int a) : v(a) {}
  R(long double a, bool) : v(a) {}
  explicit operator double() const { return (double)v; }
};
static R made(long double v) { ++ops; return R(v, true); }
R operator+(R a, R b) { return made(a.v + b.v); }
R operator-(R a, R b) { return made(a.v - b.v); }
R operator*(R a, R b) { return made(a.v * b.v); }
R operator/(R a, R b) { return made(a.v / b.v); }
int main() {
  const frlap::GaussRules g = frlap::make_gauss_rules<R>();
  std::printf("%ld\n", ops);
  for (int i = 0; i < frlap::kQTotal; ++i) std::printf("%a %a\n", g.x[i], g.w[i]);
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, exe = str(d / "rules.cpp"), str(d / "rules")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, src, "-o", exe], check=True)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    return int(lines[0]), [tuple(float.fromhex(t) for t in ln.split()) for ln in lines[1:] if ln]


def _reference(q):
    """Nodes and weights on [0, 1] in 50 digits, first node first."""
    D = decimal.Decimal
    out = []
    with decimal.localcontext() as ctx:
        ctx.prec = 50
        import math
        for i in range(q):
            x = D(math.cos(math.pi * (i + 0.75) / (q + 0.5)))
            for _ in range(8):
                p0, p1 = D(1), x
                for k in range(2, q + 1):
                    p0, p1 = p1, ((2 * k - 1) * x * p1 - (k - 1) * p0) / k
                dp = q * (x * p1 - p0) / (x * x - 1)
                x -= p1 / dp
            out.append(((1 - x) / 2, 1 / ((1 - x * x) * dp * dp)))
    return out


def test_nodes_and_weights_are_the_nearest_doubles(rules):
    _, got = rules
    want = [pair for q in ORDERS for pair in _reference(q)]
    assert len(got) == len(want)
    assert got == [(float(x), float(w)) for x, w in want]


def test_few_operations_in_the_extended_type(rules):
    assert rules[0] <= 10000
