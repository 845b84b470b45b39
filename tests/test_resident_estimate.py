"""The host's estimate of a session's resident positions (csrc/kvc_estimate.h), which chooses the
attention's split, against the eviction policies on the workloads' token streams: exact where
nothing is evicted, close where the budget binds and where it does not.
"""
import os
import subprocess

import numpy as np
import pytest

from oracle.policy import POLICIES, SessionPolicy
from synth import script as S

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include "kvc_estimate.h"
#include <cstdio>
#include <cstdlib>
// argv: budget window policy sink recent; stdin: tokens of an append, 0 an eviction, -1 a release.
int main(int, char** a) {
  kvc_config c = {};
  c.budget = std::atoll(a[1]);
  c.window = std::atoi(a[2]);
  c.policy = std::atoi(a[3]);
  c.sink = std::atoi(a[4]);
  c.recent = std::atoi(a[5]);
  kvc::ResidentEstimate e;
  for (int n; std::scanf("%d", &n) == 1;) {
    if (n > 0) e.append(n);
    else if (n == 0) e.evict(c);
    else e.release();
    std::printf("%lld\n", (long long)e.positions());
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("estimate")
    src, exe = d / "estimate.cpp", d / "estimate"
    src.write_text(PROGRAM)
    inc = os.path.join(ROOT, "paper_2609_31224_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover",
                    "-I", inc, str(src), "-o", str(exe)], check=True)

    def estimate(ops, budget, window, policy="unit", sink=0, recent=0):
        args = [str(x) for x in (budget, window, POLICIES.index(policy), sink, recent)]
        r = subprocess.run([str(exe), *args], input=" ".join(map(str, ops)), capture_output=True,
                           text=True)
        assert r.returncode == 0, r.stderr
        return [int(x) for x in r.stdout.split()]
    return estimate


def _units(n, seed):
    w = S.SINGLE_BF16.with_(seed=seed)
    sc = S.workload_scripts(w)[0]
    return [sc.unit_types(u) for u in range(n)]


@pytest.mark.parametrize("budget,window,policy", [
    (-1, 10, "unit"), (4096, 10, "unit"), (600, 10, "unit"), (300, 5, "unit"), (256, 20, "unit"),
    (0, 10, "unit"), (0, 1, "unit"), (300, 10, "position"), (0, 10, "position")])
@pytest.mark.parametrize("every", [1, 32])
def test_speech(program, budget, window, policy, every):
    """Every unit evicted on its own, and histories fed back 32 units at a time."""
    pol = SessionPolicy(budget, window, policy)
    ops, want = [], []
    units = _units(400, 3)
    for u in range(0, len(units), every):
        types = np.concatenate(units[u:u + every])
        pol.append(types)
        ops.append(len(types))
        want.append(pol.resident())
        pol.evict()
        ops.append(0)
        want.append(pol.resident())
    got = program(ops, budget, window, policy)
    for g, w in zip(got, want):
        if budget < 0:
            assert g == w
        else:  # (pages: within two of them, or a third)
            assert w - 32 <= g <= max(w + 64, 1.35 * w), (g, w)


def test_sink_recent_and_release(program):
    assert program([100, 0, 7, 0, -1, 5, 0], 0, 0, "sink_recent", 4, 20) == [100, 24, 31, 24, 0, 5, 5]


def test_budgets_of_any_size(program):
    """No sum overflows (the program is built to stop at the first that does)."""
    big = 2**63 - 1
    assert program([1000, 0, 5], big, 2**31 - 1) == [1000, 1000, 1005]
    assert program([1000, 0, 5], 0, 2**31 - 1) == [1000, 1000, 1005]
    assert program([1000, 0], 0, 0, "sink_recent", 2**31 - 1, 2**31 - 1) == [1000, 1000]
