"""Bounds under which the packed linear kernels run a scoring scheme (the plan
of csrc/diag_plan.h, compiled for the host): over the whole accepted score
range no 16-bit key leaves its half-word in a scheme that the plan takes,
and schemes whose substitutions would are refused."""
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2002_05200_gb300", "csrc")
KS = 32

DRIVER = """
#include <cstdio>
#include "diag_plan.h"
int main() {
    int m, x, g;
    long long X;
    while (std::scanf("%d %d %d %lld", &m, &x, &g, &X) == 4) {
        logan::DiagArgs a{};
        const bool ok = logan::diag_plan(m, x, g, X, &a);
        std::printf("%d %d %d ", ok ? 1 : 0, a.period, a.floor);
        const bool rec = logan::diag_record_plan(m, x, g, X, &a);
        std::printf("%d %d %d\\n", rec ? 1 : 0, a.period, a.floor);
    }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, exe = d / "plan.cpp", d / "plan"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(schemes):
        text = "\n".join(" ".join(map(str, s)) for s in schemes)
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


def key_range(match, mismatch, gap, X, period):
    """Smallest and largest key of a cell that matters, theta starting a period at
    32768: the two anti-diagonals before it may lie 2 |gap| + mp below; in a
    period theta grows by |gap| a step and by mp in any two."""
    g, mp = -gap, max(match, 0)
    live = 32768 - KS * (2 * g + mp)
    top = 32768 + KS * (period * g + mp * (period // 2 + 1))
    lowest = min(live, live + KS * (min(mismatch, match) + 2 * g))
    return lowest, top + KS * (X + mp) + KS - 1, top


def schemes(n):
    rng = random.Random(5)
    for _ in range(n):
        match = rng.choice([1, 2, 5, rng.randint(0, 120), rng.randint(-20, 1000)])
        mismatch = min(match, rng.choice([-1, -1000, -rng.randint(0, 1000), rng.randint(-1000, 1000)]))
        gap = rng.choice([0, -1, -rng.randint(0, 60), -rng.randint(0, 1000)])
        yield match, mismatch, gap, rng.choice([0, 10, 100, 300, rng.randint(0, 1200)])


def test_no_key_leaves_its_half_word(plan):
    cases = list(schemes(20000))
    taken = far = 0
    for s, (ok, period, floor, *_) in zip(cases, plan(cases)):
        if not ok:
            continue
        lowest, highest, top = key_range(*s, period)
        assert 0 <= lowest and highest <= 65535, (s, period)
        assert floor > top - 32768, s                 # theta does not outgrow a dead key
        assert floor < 32768 - KS * (2 * -s[2] + max(s[0], 0)), s   # nor does the floor reach a live one
        taken += 1
        far += max(s[0], 0) - s[1] > 900
    assert taken > 1000 and far > 50


def test_recorded_keys_are_less_than_32768_apart(plan):
    # what the recording sweep subtracts: keys at or above the floor, and a gap
    # move's key and a live diagonal's, KS (max(match, 0) - mismatch) apart at most
    cases = list(schemes(20000))
    taken = 0
    for s, (*_, ok, period, floor) in zip(cases, plan(cases)):
        if not ok:
            continue
        _, highest, top = key_range(*s, period)
        assert highest - floor + KS < 32768, s
        assert floor > top - 32768 and floor < 32768 - KS * (2 * -s[2] + max(s[0], 0)), s
        assert KS * (max(s[0], 0) - s[1]) + KS < 32768, s
        taken += 1
    assert taken > 1000


@pytest.mark.parametrize("scheme,ok", [
    ((25, -1000, -10, 100), 0), ((100, -1000, -50, 100), 0), ((30, -1000, -20, 300), 0),
    ((60, -1000, -30, 300), 0), ((50, -1000, -10, 300), 0),
    # both sides of the bound: max(-mismatch, 0) + 2 match + 2 <= 1021
    ((10, -1000, -5, 100), 0), ((9, -1000, -5, 100), 1), ((9, -1000, -5, 600), 1),
    ((1, -1000, -1, 100), 1), ((1, -1, -1, 1014), 0), ((1, -1, -1, 1013), 1)])
def test_schemes_near_the_bounds(plan, scheme, ok):
    assert plan([scheme])[0][0] == ok
