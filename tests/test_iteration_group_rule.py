"""The rule for the iterations that are queued between two looks at the solver
state (csrc/iteration_group.h), compiled for the host: bounded after a solve
that crept, unmoved by right-hand sides that broke down, never past the cap."""
import math
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1103_5103_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "iteration_group.h"
using namespace wl;
// input: K, last, n, then per rhs of the last solve: active done breakdown iters rr target2 delta2,
// then delta2 and active of the next one; output: rate, iterations, first group, next group
int main()
{
    int K, n;
    long last;
    while (std::scanf("%d %ld %d", &K, &last, &n) == 3) {
        RhsProgress p[8];
        double d2[8];
        int act[8];
        for (int r = 0; r < n; ++r) {
            int a, d, b;
            std::scanf("%d %d %d %d %lf %lf %lf", &a, &d, &b, &p[r].iters, &p[r].rr, &p[r].target2, &p[r].delta2);
            p[r].active = a, p[r].done = d, p[r].breakdown = b;
        }
        for (int r = 0; r < n; ++r) std::scanf("%lf %d", &d2[r], &act[r]);
        const InnerPace q = learn_pace(p, n);
        std::printf("%.17g %d %d %d\n", q.rate, q.iters, first_group(q, K, last, d2, act, n), next_group(p, n, K, last));
    }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text(PROGRAM)
    exe = str(d / "rule")
    subprocess.check_call([cxx, "-std=c++17", "-I" + CSRC, str(d / "rule.cpp"), "-o", exe])

    def run(K, last, rhs, nxt):
        words = [K, last, len(rhs)] + [w for r in rhs for w in r] + [w for r in nxt for w in r]
        out = subprocess.run([exe], input=" ".join(repr(w) for w in words), text=True, stdout=subprocess.PIPE, check=True)
        rate, iters, first, after = out.stdout.split()
        return float(rate), int(iters), int(first), int(after)
    return run


def _reached(iters, delta2=1e-12, **kw):
    """An rhs of unit residual that reached its target in `iters` iterations."""
    return (1, kw.get("done", 1), kw.get("breakdown", 0), iters, kw.get("rr", delta2), delta2, delta2)


def test_steady_solves_are_queued_whole(rule):
    rate, iters, first, _ = rule(8, 100000, [_reached(40), _reached(30)], [(1e-12, 1), (1e-12, 1)])
    assert iters == 40 and math.isclose(rate, math.log(1e12) / 40)
    assert first == 40
    # less is asked for: fewer; another rhs only counts while it is active
    assert rule(8, 100000, [_reached(40)], [(1e-6, 1)])[2] == 20
    assert rule(8, 100000, [_reached(40), _reached(30)], [(1e-6, 1), (1e-12, 0)])[2] == 20


def test_first_group_is_bounded_by_the_last_solve(rule):
    # ten iterations for one per cent, which was all that was asked for
    rate, iters, first, _ = rule(8, 100000, [_reached(10, 0.99, rr=0.989)], [(1e-12, 1)])
    assert 0 < rate < 2e-3 and iters == 10
    assert first == 20   # ln 1e12 / rate asks for 25 thousand
    assert rule(8, 100000, [_reached(2, 0.99, rr=0.989)], [(1e-12, 1)])[2] == 8   # a block in any case
    assert rule(8, 16, [_reached(40)], [(1e-12, 1)])[2] == 16                     # and the cap


def test_what_failed_teaches_nothing(rule):
    broke = (1, 1, 1, 5, 0.9999, 1e-12, 1e-12)
    stuck = (1, 0, 0, 64, 0.9, 1e-12, 1e-12)
    for bad in (broke, stuck):
        assert rule(8, 100000, [bad, _reached(40)], [(1e-12, 1), (1e-12, 1)])[:3] == \
            rule(8, 100000, [_reached(40)], [(1e-12, 1)])[:3]
        assert rule(8, 100000, [bad], [(1e-12, 1)])[:3] == (0.0, 0, 8)


def test_later_groups(rule):
    half = (1, 0, 0, 20, 1e-6, 1e-12, 1e-12)
    assert rule(50, 100000, [half], [(1e-12, 1)])[3] == 20
    assert rule(8, 100000, [half], [(1e-12, 1)])[3] == 8
    assert rule(8, 3, [half], [(1e-12, 1)])[3] == 3
    assert rule(8, 100000, [(1, 0, 0, 20, 1.5, 1e-12, 1e-12)], [(1e-12, 1)])[3] == 8   # no progress
    assert rule(8, 100000, [(1, 1, 0, 20, 1e-13, 1e-12, 1e-12)], [(1e-12, 1)])[3] == 1
