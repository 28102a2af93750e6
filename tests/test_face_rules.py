"""The S-point rules of the tent matrix's face integrals and their tables
(tp::face_rule), computed by the host code compiled on its own and checked in
exact rational arithmetic, against the moments of a simplex and against the
front rule, for every dimension and degree that has one:

* points inside, weights positive, exact to degree 2p;
* to_points takes front values of a polynomial of degree p to sqrt(w) times its
  values at the rule's points, to_front takes those back to the front;
* a constant passes with an error far below one rounding, so that a table used
  by every tent of a sweep does not add up its roundings.

Every tolerance is a bound on the roundings of the stored values, u = 2^-53 for
binary64 and 2^-47 for the float-float pairs.  A table's row is rounded entry
after entry, each taking the error so far: entry k is off by its own rounding
and by that of the entry before, u |t_k| + u max_j(|t_j| w_j) / w_k with the
weights w of the constant's sum."""
import itertools
import os
import subprocess
from fractions import Fraction
from math import factorial

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1907_02367_gb300", "csrc")
DEGREES = [(2, p) for p in range(1, 6)] + [(3, p) for p in range(1, 4)]
U, UFF = Fraction(1, 2 ** 53), Fraction(1, 2 ** 47)
UBASIS = Fraction(1, 2 ** 56)   # orthonormal bases in 64-bit mantissas

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "tp_internal.h"
int main(int, char** v) {
  const int n = std::atoi(v[1]), p = std::atoi(v[2]);
  const tp::SimplexRule q = tp::simplex_rule(n, p + 1);
  const tp::FaceRule& r = tp::face_rule(n, p, q);
  std::printf("%d %d %d\n", q.Q, r.S, r.stride);
  auto row = [](const auto& a) { for (double x : a) std::printf("%a ", x); std::printf("\n"); };
  row(q.bary); row(q.w); row(r.bary); row(r.sqw); row(r.to_points); row(r.to_front); row(r.to_points_ff); row(r.to_front_ff);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("face_rules")
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "rules")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC, str(d / "main.cpp"),
                    os.path.join(CSRC, "tp_host.cpp"), "-o", exe], check=True)
    return exe


def _rules(program, n, p):
    lines = subprocess.run([program, str(n), str(p)], check=True, capture_output=True, text=True).stdout.splitlines()
    Q, S, stride = map(int, lines[0].split())
    num = [[Fraction(float.fromhex(x)) for x in ln.split()] for ln in lines[1:]]
    pts = lambda a: [a[i:i + n + 1] for i in range(0, len(a), n + 1)]
    table = lambda a: [a[i * stride:i * stride + Q] for i in range(S)]
    pair = lambda a: [a[2 * i] + a[2 * i + 1] for i in range(len(a) // 2)]
    return dict(Q=Q, S=S, xq=pts(num[0]), wq=num[1], xs=pts(num[2]), sqw=num[3], to_points=table(num[4]), to_front=table(num[5]),
                to_points_ff=table(pair(num[6])), to_front_ff=table(pair(num[7])))


def _exponents(n, deg):
    return [a for a in itertools.product(range(deg + 1), repeat=n + 1) if sum(a) <= deg]


def _power(lam, a):
    t = Fraction(1)
    for x, k in zip(lam, a):
        t *= x ** k
    return t


def _moment(n, a):   # over the reference simplex
    t = 1
    for k in a:
        t *= factorial(k)
    return Fraction(t, factorial(sum(a) + n))


@pytest.mark.parametrize("n,p", DEGREES)
def test_exact_to_twice_the_degree(program, n, p):
    r = _rules(program, n, p)
    assert 0 < r["S"] < r["Q"] == (p + 1) ** n
    assert all(x > 0 for lam in r["xs"] for x in lam) and all(w > 0 for w in r["sqw"])
    assert all(abs(sum(lam) - 1) <= (n + 1) * U for lam in r["xs"])
    for a in _exponents(n, 2 * p):
        got = sum(s * s * _power(lam, a) for s, lam in zip(r["sqw"], r["xs"]))
        # every coordinate is off by at most 2 u, every weight by 3 u of itself
        down = sum(k * _moment(n, a[:i] + (k - 1,) + a[i + 1:]) for i, k in enumerate(a) if k)
        assert abs(got - _moment(n, a)) <= 2 * (2 * U * down + 3 * U * _moment(n, a)), a


@pytest.mark.parametrize("n,p", DEGREES)
def test_tables_carry_polynomials(program, n, p):
    r = _rules(program, n, p)
    rng = np.random.default_rng(10 * n + p)
    exps = [a for a in _exponents(n, p) if a[0] == 0]   # (the stored coordinates sum to 1 only to rounding)
    polys = [[(a, Fraction(1))] for a in exps] + [[(a, Fraction(float(c))) for a, c in zip(exps, rng.normal(size=len(exps)))]
                                                  for _ in range(3)]
    for f in polys:
        val = lambda lam: sum(c * _power(lam, a) for a, c in f)
        fq, fs = [val(x) for x in r["xq"]], [s * val(x) for s, x in zip(r["sqw"], r["xs"])]

        def check(row, data, want, weight, u):
            carried = max(abs(t) * w for t, w in zip(row, weight))
            bound = sum(abs(v) * u * (abs(t) + carried / w) for t, v, w in zip(row, data, weight))
            assert abs(sum(t * v for t, v in zip(row, data)) - want) <= bound + UBASIS * sum(abs(t * v) for t, v in zip(row, data))

        for name, u in (("to_points", U), ("to_points_ff", UFF)):
            for i, row in enumerate(r[name]):
                check(row, fq, fs[i], [Fraction(1)] * r["Q"], u)
        for name, u in (("to_front", U), ("to_front_ff", UFF)):
            for q in range(r["Q"]):
                check([row[q] for row in r[name]], fs, fq[q], r["sqw"], u)


@pytest.mark.parametrize("n,p", DEGREES)
def test_a_constant_passes(program, n, p):
    """What is left of a row is the rounding of its smallest entry, and of the
    entries' own computation in 64-bit mantissas."""
    r = _rules(program, n, p)
    for name, u in (("to_points", U), ("to_points_ff", UFF)):
        for i, row in enumerate(r[name]):
            left = u * min(map(abs, row)) + r["Q"] * UBASIS / 16 * max(map(abs, row))
            assert abs(sum(row) - r["sqw"][i]) <= left
    big = max(r["sqw"])
    for name, u in (("to_front", U), ("to_front_ff", UFF)):
        for q in range(r["Q"]):
            col = [row[q] for row in r[name]]
            left = u * min(map(abs, col)) * big + r["S"] * UBASIS / 16 * max(map(abs, col)) * big
            assert abs(sum(t * s for t, s in zip(col, r["sqw"])) - 1) <= left


@pytest.mark.parametrize("n,p", [(1, p) for p in range(1, 9)])
def test_no_rule_where_the_front_rule_is_as_small(program, n, p):
    assert _rules(program, n, p)["S"] == 0
