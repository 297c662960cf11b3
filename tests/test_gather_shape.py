"""The gather's launch shape (csrc/gather_shape.h), compiled by itself: every
element of every instance is reached by one thread, and no index that a thread
forms, one stride past the last element included, leaves its type."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2602_19699_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "gather_shape.h"
int main(int argc, char** argv) {
  for (int i = 1; i + 4 < argc; i += 5) {
    const long long e = to::gather_elems(atoi(argv[i + 1]), atoi(argv[i + 2]), atoi(argv[i + 3]), atoi(argv[i + 4]));
    const to::GatherShape s = to::gather_shape(atoi(argv[i]), e);
    printf("%lld %u %u %u %u %d %d\n", e, s.bx, s.by, s.gx, s.gy, (int)s.wide, to::kGatherThreads);
  }
}
"""

SYSTEMS = [(4, 2), (6, 3), (14, 7), (36, 12), (5, 2)]
HORIZONS = [1, 2, 7, 50, 255, 400, 5_000_000, 22_000_000, 89_478_485, 268_435_455, 268_435_456, 536_870_912, 2 ** 31 - 2]


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    d = tmp_path_factory.mktemp("gather")
    src, exe = str(d / "shape.cpp"), str(d / "shape")
    with open(src, "w") as f:
        f.write(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, src, "-o", exe], check=True)
    cases = [(B, T, n, m, K) for B in (1, 3, 70_000) for T in HORIZONS for n, m in SYSTEMS for K in (0, 1)]
    out = subprocess.run([exe, *(str(v) for c in cases for v in c)], check=True, capture_output=True, text=True).stdout
    return list(zip(cases, ([int(v) for v in line.split()] for line in out.splitlines())))


def test_indices_fit_their_type_and_reach_every_element(shapes):
    assert len(shapes) == 3 * len(HORIZONS) * len(SYSTEMS) * 2
    kinds = set()
    for (B, T, n, m, K), (elems, bx, by, gx, gy, wide, threads) in shapes:
        assert elems == max((T + 1) * n, T * m * n if K else 0)
        stride = gx * bx
        # a thread's last index, one stride past the output's end, and the sizes that the kernel forms
        assert elems + 2 * stride < 2 ** (63 if wide else 31), (T, n, m, K)
        assert stride >= 1 and 1 <= gy <= min(B, 65535) and gx < 2 ** 31
        assert bx * by == threads and threads % 32 == 0
        # a block less than twice as wide as an instance's output; no set of instances without an instance
        assert bx < max(16, 2 * elems) and (gy - 1) * by < B
        kinds.add(wide)
    assert kinds == {0, 1}
