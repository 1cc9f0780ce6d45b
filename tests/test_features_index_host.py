"""The offsets of the estimator's features walk (csrc/wo_feat.cuh), compiled
for the host: every point of a plane's rows 0 .. Y/2 and its mirror image,
against the same in Python integers, at planes on both sides of what 32 bits
count.  wo_est_features takes any plane that fits the device, and a wrapped
offset would read far outside it."""
import os
import subprocess

import pytest

from paper_2412_09775_gb300.build import CSRC, nvcc

MAIN = r"""
#include <stdio.h>
#include "wo_feat.cuh"
template <class I> void show(int Y, int Xh, long long p) {
  int y, x;
  const wo::FeatPoint<I> f = wo::feat_point((I)p, Y, Xh, &y, &x);
  printf("%d %d %lld %d %d %lld %lld\n", Y, Xh, p, y, x, (long long)f.at, (long long)f.mirror);
}
int main() {
  int Y, Xh;
  long long p;
  while (scanf("%d %d %lld", &Y, &Xh, &p) == 3) {
    if (wo::feat_wide(Y, Xh)) show<long long>(Y, Xh, p);
    else show<int>(Y, Xh, p);
  }
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    d = tmp_path_factory.mktemp("feat")
    src, exe = d / "walk.cu", d / "walk"
    src.write_text(MAIN)
    subprocess.run([nvcc(), "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)

    def run(rows):
        text = "".join("%d %d %d\n" % r for r in rows)
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    return run


@pytest.mark.parametrize("Y,Xh", [(2, 2), (3, 5), (48, 25), (127, 65),     # small planes, odd heights
                                  (65536, 32767), (65536, 32769),           # either side of 2^31 points
                                  (2, 1 << 30), (1 << 30, 3), (200000, 100001)])
def test_points_and_mirrors(walk, Y, Xh):
    points = (Y // 2 + 1) * Xh
    ps = range(points) if points < 5000 else \
        sorted({q for c in (0, Xh, points // 2, points) for q in range(max(c - 70, 0), min(c + 70, points))})
    got = walk([(Y, Xh, p) for p in ps])
    want = []
    for p in ps:
        y, x = divmod(p, Xh)
        want.append((Y, Xh, p, y, x, p, (Y - y) * Xh + x if 0 < y and 2 * y < Y else -1))
    assert got == want
    assert all(w[6] < Y * Xh for w in want)
