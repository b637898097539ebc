"""The brick ranges of a particle's reach (brick_range), compiled for the host from the kernels' own
header: for every origin and reach, huge and non-finite ones among them, each range lies within the
axis and has a <= b, since the ranges index the brick arrays; for ordinary ones they are exactly the
bricks that hold a cell interval the reach meets."""
import math
import os
import subprocess

import numpy as np
import pytest

from paper_2308_05007_gb300 import build

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include "rwmi_internal.cuh"
int main() {
  double o, R;
  int cells, nb, wall;
  while (std::scanf("%lf %lf %d %d %d", &o, &R, &cells, &nb, &wall) == 5) {
    const rwmi::BrickRange r = rwmi::brick_range(o, R, cells, nb, wall);
    std::printf("%d %d %d %d %d\n", r.n, r.a[0], r.b[0], r.a[1], r.b[1]);
  }
}
"""


@pytest.fixture(scope="module")
def ranges(tmp_path_factory):
    d = tmp_path_factory.mktemp("brick_range")
    (d / "range.cu").write_text(PROGRAM)
    exe = str(d / "range")
    subprocess.check_call([build._nvcc(), *build.ARCH, "-std=c++17", "-I" + build.CSRC,
                           "-I" + os.path.join(build.ROOT, "include"), "-o", exe, str(d / "range.cu")])

    def run(rows):
        text = "\n".join(f"{float(o)!r} {float(R)!r} {n} {(n + 7) // 8} {w}" for o, R, n, w in rows) + "\n"
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    return run


def test_ranges_stay_within_the_axis(ranges):
    big = [s * 10.0 ** e * m for e in (16, 17, 31, 32, 33, 40, 100, 250, 300) for m in (1.0, 3.7, 1 / 3) for s in (1, -1)]
    rng = np.random.default_rng(1)
    big += list(rng.uniform(-1, 1, 400) * 10.0 ** rng.uniform(15, 305, 400))
    big += [math.inf, -math.inf, math.nan, 0.0, -0.0]
    rows = [(o, R, n, w) for o in big for R in (0.5, 3.3, 9.0, 1e6, math.inf) for n in (1, 7, 8, 33, 100, 256)
            for w in (0, 1)]
    got = ranges(rows)
    assert len(got) == len(rows)
    for (o, R, n, w), (k, a0, b0, a1, b1) in zip(rows, got):
        assert k in (0, 1, 2)
        for a, b in ((a0, b0), (a1, b1))[:k]:
            assert 0 <= a <= b < (n + 7) // 8, (o, R, n, w)


def test_ranges_are_the_bricks_the_reach_meets(ranges):
    rng = np.random.default_rng(2)
    rows = [(float(o), float(R), int(n), int(w)) for n in (5, 8, 33, 64, 100) for w in (0, 1)
            for o, R in zip(rng.uniform(0, n, 60), rng.uniform(0.3, 0.7 * n, 60))]
    for (o, R, n, w), (k, a0, b0, a1, b1) in zip(rows, ranges(rows)):
        got = set(range(a0, b0 + 1) if k > 0 else ()) | set(range(a1, b1 + 1) if k > 1 else ())
        images = (0,) if w else (-n, 0, n)
        want = {b for b in range((n + 7) // 8)
                if any(o + s + R >= 8 * b and o + s - R < min(8 * b + 8, n) for s in images)}
        assert got >= want and len(got - want) <= 1, (o, R, n, w, got, want)   # a merged gap of no brick
