"""Prefix sums of the channel costs by which CTAs share a call, on the host: a
small program built from the same header.  They stay exact while they fit and
are scaled down together where they would not (tens of thousands of channels
at N = 512); every channel keeps a positive share near its part of the cost."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1603_02126_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "epic_batch.h"
int main() {
  std::vector<long long> cost;
  long long c;
  while (std::scanf("%lld", &c) == 1) cost.push_back(c);
  for (int v : epic::cost_prefix(cost)) std::printf("%d\n", v);
  return 0;
}
"""


@pytest.fixture(scope="module")
def prefix(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("cost")
    src, exe = d / "c.cpp", d / "c"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    return lambda cost: np.array(subprocess.run([str(exe)], input="\n".join(map(str, cost)), check=True,
                                                capture_output=True, text=True).stdout.split(), dtype=np.int64)


def test_small_costs_are_exact(prefix):
    cost = [3, 1, 0, 7, 94000]
    assert prefix(cost).tolist() == [0, 3, 4, 5, 12, 94012]


@pytest.mark.parametrize("n,top", [(22000, 100000), (60000, 100000), (1000, 1 << 40)])
def test_large_costs_are_scaled(prefix, n, top):
    cost = np.random.default_rng(n).integers(top // 2, top, n)
    p = prefix(cost.tolist())
    assert p[0] == 0 and p[-1] <= 1 << 30 and np.all(np.diff(p) > 0)
    assert np.max(np.abs(np.diff(p) / p[-1] * cost.sum() / cost - 1)) < 0.01
