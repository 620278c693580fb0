"""Batches of the wide frame-pair form, on the host: a small program built
from the same header prints the batch of many (grid, rows, channels, samples,
budget) combinations.  The kernels address a batch of n samples as
ceil(n / 2) pairs of [channels][N][rows] 16-byte cells, then the calibrator
pixels, so every batch of every call must fit the scratch that is allocated
for it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1603_02126_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "epic_batch.h"
int main() {
  int C, N, rs, tune;
  unsigned long long budget;
  long long T;
  while (std::scanf("%d %d %d %llu %d %lld", &C, &N, &rs, &budget, &tune, &T) == 6) {
    const epic::WideBatch b = epic::wide_batch(C, N, rs, budget, tune, T);
    std::printf("%lld %d %zu %zu %zu\n", b.nt, b.nc, b.spec_n, b.need, epic::wide_scratch(C, N, rs, budget));
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def batch_of(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("batch")
    src, exe = d / "b.cpp", d / "b"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + CSRC, str(src), "-o", str(exe)], check=True)

    def run(cases):
        text = "\n".join(" ".join(map(str, c)) for c in cases)
        out = subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


def _cases():
    for N in (128, 256, 512):
        for rs in (20, 52, 84, 100, 132, 260, 308, 516):
            if rs > N + 4:
                continue
            pair = 2 * N * rs * 8
            for C in (1, 2, 3, 4, 7, 16, 33, 256):
                budgets = [2 << 30, 1 << 30, pair, pair * 3, 64 << 20]
                budgets += [q * C * pair // 2 for q in (257, 301, 302, 1001)]
                for budget in budgets:
                    if budget < pair:
                        continue
                    for T in (1, 2, 3, 255, 256, 257, 258, 515, 2001, 10000):
                        for tune in (0, 1, 7, 128):
                            yield C, N, rs, budget, tune, T


def test_every_batch_fits_its_scratch(batch_of):
    cases = list(_cases())
    for (C, N, rs, budget, tune, T), (nt, nc, spec_n, need, held) in zip(cases, batch_of(cases)):
        case = (C, N, rs, budget, tune, T, nt, nc)
        assert nt >= 2 and nt % 2 == 0, case
        assert 1 <= nc <= C, case
        sizes = {min(nt, T), T % nt or nt}                  # samples of the batches of this call
        pairs = max((n + 1) // 2 for n in sizes)
        assert 2 * pairs * nc * N * rs <= spec_n, case      # spectra end before the pixels
        assert spec_n + max(sizes) * C <= need, case        # pixels end inside the scratch
        assert spec_n * 8 <= budget, case
        assert need <= held, case                           # a scratch held for calls of any length
